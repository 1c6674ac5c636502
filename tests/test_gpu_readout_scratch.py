"""The read-out of a state uses the scratch of the step and, in FP64, nodes of
the other population copy: reading between steps changes neither the states
that follow, byte for byte with their ghost frames, nor a second reading."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _walls(nx, ny, N):
    """Two solids given by their own psi_k and angles."""
    x, y = np.meshgrid(np.arange(nx) + 0.5, np.arange(ny) + 0.5)
    a = W.psi_from_distance(y - 4.0, xi=1.0)
    b = W.psi_from_distance(np.hypot(x - 0.6 * nx, y - 0.6 * ny) - 4.0, xi=1.0)
    return [(a, np.full(N - 1, 0.3)), (b, np.full(N - 1, -0.2))]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny,N,kind", [
    (3, 3, 2, "plain"), (40, 27, 2, "plain"), (65, 33, 3, "plain"), (130, 45, 4, "plain"),
    (70, 31, 3, "open"), (48, 40, 3, "walls"), (96, 40, 2, "sweep"), (96, 40, 4, "sweep"),
])
def test_reading_leaves_the_run_as_it_is(nx, ny, N, kind, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10314_gb300 import build as B
    B.build()
    import paper_2311_10314_gb300 as D
    px = 0 if kind == "open" else 1
    pb = W.random_problem(nx, ny, N, seed=nx + N, periodic_x=px, periodic_y=0, theta_field=True, width=6.0)
    kw = dict(precision=precision)
    if kind == "open":
        kw["open_x"] = (np.full(ny, 0.002), np.full((N - 1, ny), 0.1))
    if kind == "sweep":
        kw["path"] = "sweep"

    def make():
        if kind == "walls":
            return D.Sim(pb.params, None, pb.C0, walls=_walls(nx, ny, N), **kw)
        return D.Sim(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field, **kw)

    plain, read = make(), make()
    for n in (0, 1, 2, 5, 6):
        plain.step(n)
        read.step(n)
        one = read.fields()
        mu = read.read(D.FIELD_MU + N - 1)
        psi = read.read(20)
        assert np.array_equal(one["mu"][N - 1], mu)
        if kind != "walls":
            assert np.abs(psi - pb.psi).max() <= (0 if precision == 0 else 1e-7)
        two = read.fields()
        for k in one:
            assert np.isfinite(one[k]).all() and np.array_equal(one[k], two[k]), k
        # (a save leaves the padding after the step count as it was)
        a, b = (s.save_state(torch.zeros(s.state_bytes(), dtype=torch.uint8, device="cuda")) for s in (plain, read))
        assert torch.equal(a, b)
    plain.close()
    read.close()
