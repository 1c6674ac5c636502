"""The FP64 phase collision keeps sum_p f at each node to roundings at the
moving populations' scale (they are a thousandth of psi C and less), by the
transforms and by the form for one rate above first order."""
import math

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [2, 4])
@pytest.mark.parametrize("rates", [(1.0, 1.2, 1.2, 1.2, 1.2), (1.0, 0.7, 0.7, 0.7, 0.7), (1.0, 1.2, 1.1, 1.2, 1.2)])
def test_fp64_step_keeps_the_phase_sum(N, rates):
    """One step changes the exact sum of a phase's populations by the sum of
    8 n roundings of moving populations, each a few 2^-53 of its size: the
    bar is ten times their root sum of squares.  The rounding of psi C
    itself, 2^-54 a node, would be above it."""
    from paper_2311_10314_gb300 import build as B
    B.build()
    import paper_2311_10314_gb300 as D
    from paper_2311_10314_gb300 import _lib
    nx, ny = 70, 33
    pb = W.random_problem(nx, ny, N, seed=5 + N, periodic_y=0, theta_field=True, width=6.0)
    pb.params["s_f"] = list(rates)
    sim = D.Sim(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field, precision=D.DDCC_FP64)
    org, pitch, plane = _lib.state_layout(nx, ny, N, 8)

    def populations():
        s = sim.save_state().view(torch.float64)
        return torch.as_strided(s, (N - 1, 9, ny, nx), (9 * plane, plane, pitch, 1), org).cpu().numpy().copy()

    sim.step(10)
    before = populations()
    for _ in range(4):
        sim.step(1)
        after = populations()
        for i in range(N - 1):
            size = max(np.sqrt((v[i, 1:] ** 2).mean()) for v in (before, after))
            bar = 10.0 * math.sqrt(8 * nx * ny) * 2.0 ** -53 * size
            assert bar < math.sqrt(nx * ny) * 2.0 ** -55     # well under psi C's own rounding
            change = math.fsum(np.concatenate([after[i].ravel(), -before[i].ravel()]))
            print(N, rates[1:3], i, change, bar)
            assert abs(change) <= bar
        before = after
    sim.close()


@pytest.mark.parametrize("d0", [0.3, 0.25])
def test_fp32_collision_has_no_mean_exchange(d0):
    """In FP32 the node sums of a phase must not change on average: moving
    populations far from equilibrium (so that every moment relaxes, with a
    mean) over 512 x 512 nodes, one step.  The sums over the weights that
    vanish do so exactly where 1 - d0 in FP32 is one less d0 in FP32 (as for
    these d0), if the weights are products of the 1D weights; the bar is one
    rounding of a moving population (the mean of 2.6e5 node sums scatters by a
    sixtieth of that).  Weights rounded each by itself leave fourteen times
    the bar at d0 = 0.3."""
    from paper_2311_10314_gb300 import build as B
    B.build()
    import paper_2311_10314_gb300 as D
    from paper_2311_10314_gb300 import _lib
    assert np.float32(1) - np.float32(d0) == np.float32(1 - d0)
    n = 512
    params = W.base_params(n, n, 2, d0=d0, sigma=1e-6, width=4.0)
    sim = D.Sim(params, np.ones((n, n)), np.full((1, n, n), 0.5), np.zeros(1), precision=D.DDCC_FP32)
    org, pitch, plane = _lib.state_layout(n, n, 2, 4)
    rng = np.random.default_rng(7)
    f = 1e-3 * (1.0 + 0.5 * rng.standard_normal((9, n, n)))
    f[0] = 0.5 + 0.2 * rng.random((n, n))
    f = f.astype(np.float32)
    state = sim.save_state()
    view = torch.as_strided(state.view(torch.float32), (9, n, n), (plane, pitch, 1), org)
    view.copy_(torch.from_numpy(f))
    sim.load_state(state)
    sim.step(1)
    g = torch.as_strided(sim.save_state().view(torch.float32), (9, n, n), (plane, pitch, 1), org).cpu().numpy()
    sim.close()
    assert np.isfinite(g).all() and np.abs(g[1:] - f[1:]).max() > 1e-4       # it did relax
    mean = (g.astype(np.float64).sum() - f.astype(np.float64).sum()) / (n * n)
    size = math.sqrt((f[1:].astype(np.float64) ** 2).mean())
    print(d0, mean, size * 2.0 ** -24)
    assert abs(mean) <= size * 2.0 ** -24
