"""A reading that fails leaves nothing behind: under stream capture, where a
read-out may not synchronise, the kernels that would form the fields are only
captured, and the next reading has to form them."""
import ctypes

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


class _Capture:
    """A capture of a torch stream by the driver, ended whatever became of it."""

    def __init__(self, stream):
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.s = ctypes.c_void_p(stream.cuda_stream)

    def __enter__(self):
        assert self.cu.cuStreamBeginCapture_v2(self.s, ctypes.c_int(1)) == 0      # thread-local mode

    def __exit__(self, *_):
        g = ctypes.c_void_p()
        if self.cu.cuStreamEndCapture(self.s, ctypes.byref(g)) == 0 and g:
            self.cu.cuGraphDestroy(g)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("three_d", [False, True])
def test_fields_after_a_read_under_capture(three_d, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10314_gb300 import build as B
    B.build()
    import paper_2311_10314_gb300 as D
    pb = (W.random_problem_3d(12, 9, 7, 3, seed=1, width=5.0) if three_d
          else W.random_problem(33, 17, 3, seed=1, width=6.0))
    stream = torch.cuda.Stream()
    sims = [(D.Sim3D if three_d else D.Sim)(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field,
                                            precision=precision, stream=stream) for _ in range(2)]
    for s in sims:
        s.step(3)
    want = sims[0].fields()
    for field in (D.FIELD_UX, D.FIELD_C):
        sims[1].step(0)                      # nothing is kept from a reading before
        torch.cuda.synchronize()
        with _Capture(stream):
            with pytest.raises(D.DdccError):
                sims[1].read(field)
        got = sims[1].fields()
        for k in want:
            assert np.array_equal(got[k], want[k]), k
    for s in sims:
        s.step(2)
    a, b = (s.fields() for s in sims)
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    for s in sims:
        s.close()
