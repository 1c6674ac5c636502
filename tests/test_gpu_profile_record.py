"""The profiling record is of ddcc_step's launches: steps from buffer to
buffer (ddcc_step_between and the reverse segments' recompute) leave none of
theirs in it."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,N", [(33, 3, 2), (40, 27, 3), (256, 3700, 3)])
def test_steps_between_buffers_are_not_recorded(nx, ny, N):
    """A grid of three rows and one of 64 x 4 tiles fill their rings by a
    launch of their own; the one between writes them with the step."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10314_gb300 import build as B
    B.build()
    import paper_2311_10314_gb300 as D
    from paper_2311_10314_gb300 import _lib
    y = np.arange(ny) + 0.5
    psi = np.full((ny, nx), 1.0)
    C0 = np.stack([np.broadcast_to(W.drop_profile(np.abs(y - 0.5 * ny), 0.2 * ny, 6.0)[:, None], (ny, nx))] * (N - 1))
    sim = D.Sim(W.base_params(nx, ny, N, sigma=0.005), psi, C0 / (N - 1), np.zeros(N - 1), precision=D.DDCC_FP32)
    a, b = (torch.zeros(sim.state_bytes() + 256, dtype=torch.uint8, device="cuda") for _ in range(2))
    pa, pb = ((t.data_ptr() + 255) // 256 * 256 for t in (a, b))
    _lib.ddcc_profile(sim.h, True)
    sim.step(2)
    fills = 2 if ny == 3 or nx * ny > 5e5 else 0
    assert [n for _, n in _lib.ddcc_kernel_times(sim.h).values()] == [0, 2, 0, fills]
    _lib.ddcc_save_state(sim.h, pa, True)
    assert _lib.ddcc_step_between(sim.h, pa, pb) == _lib.DDCC_OK
    assert [n for _, n in _lib.ddcc_kernel_times(sim.h).values()] == [0, 0, 0, 0]
    sim.close()
