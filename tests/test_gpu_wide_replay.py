"""The 64 x 4 form of the FP32 step, with its ring fills, replayed as graphs of
two and of eight steps at ragged sizes: bit for bit the plain launches (which
a handle that profiles keeps to), ghost rings included."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,N,px,py,open_x", [
    (64, 11201, 4, 1, 1, False),     # one tile wide, one row over a tile
    (191, 3751, 4, 1, 0, False),     # a column short of three tiles, walls
    (641, 2101, 2, 0, 0, False),     # one column into the eleventh tile, walls all round
    (641, 2101, 2, 0, 0, True),      # open ends (whose flow this problem bears for some 30 steps)
])
def test_replayed_wide_tiles_match_plain_launches(nx, ny, N, px, py, open_x):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10314_gb300 import build as B
    B.build()
    import paper_2311_10314_gb300 as D
    from paper_2311_10314_gb300 import _lib
    assert nx * ny * (11 * N + 3) * 4 > 128 << 20
    pb = W.random_problem(nx, ny, N, seed=nx + N, periodic_x=px, periodic_y=py, theta_field=True, width=6.0,
                          n_circles=12, n_drops=9)
    ox = (np.full(ny, 0.002), np.full((N - 1, ny), 0.1)) if open_x else None
    org, pitch, plane = _lib.state_layout(nx, ny, N, 4)
    out = []
    for plain in (True, False):
        sim = D.Sim(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field, precision=D.DDCC_FP32, open_x=ox)
        if plain:
            _lib.ddcc_profile(sim.h, True)
        for n in (1, 5, 4, 9) if open_x else (1, 5, 4, 129, 11):    # from either copy; past 128 the longer graph
            sim.step(n)
        s = sim.save_state().view(torch.float32)
        f = torch.as_strided(s, (9 * (N - 1), ny + 4, nx + 4), (plane, pitch, 1), org - 2 * pitch - 2).clone()
        g = torch.as_strided(s, (9 + 2 * N + 3, ny, nx), (plane, pitch, 1), org + 9 * (N - 1) * plane).clone()
        a = torch.as_strided(s, (ny + 2, nx + 2), (pitch, 1), org + 9 * N * plane - pitch - 1).clone()
        out.append((f, g, a))
        sim.close()
    assert torch.isfinite(out[0][0]).all()
    for p, r in zip(*out):
        assert torch.equal(p, r)
