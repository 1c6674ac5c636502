"""The reverse step over the forms the forward step takes: two to four
phases, walls or periods along each axis, a body force, grids smaller and
larger than its blocks, both precisions, against autograd through the FP64
oracle.

Bars: FP64 1e-8 of the largest gradient; FP32 1e-3 (the states carry C to
2e-5 after so few steps)."""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_adjoint import _oracle_gradient

pytestmark = pytest.mark.gpu


def forms_problem(nx, ny, N, px, py, body, seed):
    """Drops among solid circles (and on walls where an axis has them), psi
    varying at every node, unequal densities and viscosities, random angles."""
    rng = np.random.default_rng(seed)
    x, y = np.meshgrid(np.arange(nx) + 0.0, np.arange(ny) + 0.0)

    def dist(cx, cy):
        dx, dy = x - cx, y - cy
        if px:
            dx = (dx + nx / 2) % nx - nx / 2
        if py:
            dy = (dy + ny / 2) % ny - ny / 2
        return np.hypot(dx, dy)

    d = np.minimum(dist(0.63 * nx + 0.37, 0.58 * ny + 0.21) - 3.1, dist(0.11 * nx + 0.23, 0.83 * ny + 0.17) - 2.3)
    if not py:
        d = np.minimum(d, y - 2.3)
    if not px:
        d = np.minimum(d, x - 1.4)
    psi = W.psi_from_distance(d, xi=W.SOLID_XI)
    C0 = np.zeros((N - 1, ny, nx))
    left = np.ones((ny, nx))
    for i in range(N - 1):
        C0[i] = left * W.drop_profile(dist((0.3 + 0.25 * i) * nx, (0.35 + 0.2 * i) * ny), 5.5, 4.0)
        left = left - C0[i]
    params = W.base_params(nx, ny, N, periodic_x=px, periodic_y=py, sigma=0.008, width=5.0, xi=W.SOLID_XI,
                           tau=0.8, eta=1.0 if N == 2 else 0.1, body_force=body)
    if N > 2:
        params["m0"] = 0.01
    params["rho"] = [1.0, 2.0, 1.5, 0.7][:N]
    params["nu"] = [0.1, 0.07, 0.13, 0.09][:N]
    return params, psi, C0, rng.uniform(-0.6, 0.6, size=(N - 1, ny, nx))


FORMS = [
    # nx, ny, N, px, py, body, T, ckpt, phase
    (26, 22, 4, 1, 0, (0.0, 0.0), 20, 7, 0),
    (33, 17, 4, 0, 0, (1e-4, -2e-4), 16, 16, 2),      # walls all round, one column over a block
    (31, 19, 3, 0, 1, (0.0, 1e-4), 18, 5, 1),         # walls in x alone
    (40, 16, 2, 1, 1, (2e-4, 0.0), 20, 6, 0),         # periodic box
    (49, 9, 3, 1, 1, (1e-4, 1e-4), 14, 4, 0),
    (25, 25, 2, 0, 0, (0.0, -1e-4), 20, 20, 0),
]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("form", FORMS)
def test_gradients_of_every_form(form, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10314_gb300 import build as B
    B.build()
    from paper_2311_10314_gb300 import adjoint as A
    nx, ny, N, px, py, body, T, ckpt, phase = form
    params, psi, C0, cf = forms_problem(nx, ny, N, px, py, body, seed=nx + ny)
    J_ref, gc_ref, gp_ref = _oracle_gradient(params, psi, C0, cf, T, phase)
    J, gc, gp = A.centroid_gradient(params, psi, C0, cf, T, ckpt=ckpt, precision=precision, phase=phase)
    bar = 1e-8 if precision == 0 else 1e-3
    assert abs(J - J_ref) <= (1e-10 if precision == 0 else 1e-5) * abs(J_ref)
    assert np.isfinite(gc).all() and np.isfinite(gp).all()
    ec = np.abs(gc - gc_ref).max() / np.abs(gc_ref).max()
    ep = np.abs(gp - gp_ref).max() / np.abs(gp_ref).max()
    assert ec <= bar and ep <= bar, (ec, ep)
