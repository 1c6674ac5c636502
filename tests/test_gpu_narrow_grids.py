"""FP32 grids of up to 24 columns (narrower than the fused kernel's halo box)
take the order-parameter pass and the plain-load tile kernel, and their
reverse sweep the load / step / save path.  The reverse step reads the
one-node ghost ring of the lagged plane a from the states these write."""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_adjoint import _oracle_gradient, _wall_drop_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ddcc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10314_gb300 import build as B
    B.build()
    import paper_2311_10314_gb300 as D
    from paper_2311_10314_gb300 import adjoint as A
    return D, A


@pytest.mark.parametrize("nx,ny,N,px,py,open_x", [
    (3, 3, 2, 1, 1, False),
    (20, 9, 3, 1, 0, False),
    (24, 17, 3, 0, 1, False),
    (24, 40, 4, 0, 0, False),
    (17, 13, 3, 0, 0, True),
])
def test_saved_state_has_the_ring_of_a(ddcc, nx, ny, N, px, py, open_x):
    """After steps from either copy the saved ring is what loading the state
    anew puts there, bit for bit."""
    from paper_2311_10314_gb300 import _lib
    D, _ = ddcc
    pb = W.random_problem(nx, ny, N, seed=nx * ny + N, periodic_x=px, periodic_y=py, theta_field=True, width=6.0)
    pb.params["rho"] = [1.0, 2.0, 1.5, 0.7][:N]     # a vanishes for equal densities
    ox = (np.full(ny, 0.004), np.full((N - 1, ny), 0.2)) if open_x else None
    sim = D.Sim(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field, precision=D.DDCC_FP32, open_x=ox)
    org, pitch, plane = _lib.state_layout(nx, ny, N, 4)

    def ring():
        s = sim.save_state().view(torch.float32)
        return torch.as_strided(s, (ny + 2, nx + 2), (pitch, 1), org + 9 * N * plane - pitch - 1).cpu().numpy().copy()

    for n in (1, 2, 5):
        sim.step(n)
        got = ring()
        sim.load_state(sim.save_state())      # refills every ghost frame
        want = ring()
        assert np.isfinite(want).all() and (nx == 3 or np.abs(want).max() > 0)
        assert np.array_equal(got, want)
    sim.close()


@pytest.mark.parametrize("nx,ckpt", [(20, 7), (24, 24)])
def test_fp32_gradient_on_narrow_grids(ddcc, nx, ckpt):
    """Against autograd through the FP64 oracle: FP32 states carry C to 2e-5
    after so few steps, so the gradients' relative error is of that size; the
    bar leaves a factor of 50."""
    D, A = ddcc
    params, psi, C0, cf = _wall_drop_problem(nx, 22, 3, seed=nx)
    J_ref, gc_ref, gp_ref = _oracle_gradient(params, psi, C0, cf, 24)
    J, gc, gp = A.centroid_gradient(params, psi, C0, cf, 24, ckpt=ckpt, precision=D.DDCC_FP32)
    assert abs(J - J_ref) <= 1e-5 * abs(J_ref)
    ec = np.abs(gc - gc_ref).max() / np.abs(gc_ref).max()
    ep = np.abs(gp - gp_ref).max() / np.abs(gp_ref).max()
    assert ec <= 1e-3 and ep <= 1e-3, (ec, ep)
