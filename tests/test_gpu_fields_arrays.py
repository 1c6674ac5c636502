"""Every entry of fields() owns its memory: keeping one does not keep the
others alive."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("three_d", [False, True])
def test_fields_are_arrays_of_their_own(three_d, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10314_gb300 import build as B
    B.build()
    import paper_2311_10314_gb300 as D
    N = 3
    pb = (W.random_problem_3d(12, 9, 7, N, seed=1, width=5.0) if three_d
          else W.random_problem(33, 17, N, seed=1, width=6.0))
    sim = (D.Sim3D if three_d else D.Sim)(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field,
                                          precision=precision)
    sim.step(3)
    f = sim.fields()
    shape = pb.psi.shape
    for k, v in f.items():
        assert v.base is None and v.flags.owndata and v.flags.c_contiguous, k
        assert v.shape == ((N,) + shape if k in ("C", "mu") else shape), k
        assert np.isfinite(v).all(), k
    for i in range(N):
        assert np.array_equal(f["C"][i], sim.read(D.FIELD_C + i))
        assert np.array_equal(f["mu"][i], sim.read(D.FIELD_MU + i))
    for k, field in (("rho", D.FIELD_RHO), ("ux", D.FIELD_UX), ("uy", D.FIELD_UY), ("P", D.FIELD_P)):
        assert np.array_equal(f[k], sim.read(field)), k
    sim.close()
