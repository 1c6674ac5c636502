"""The workspace of the 2D step holds two copies of the populations and of the
lagged planes, psi and the angles, and as scratch no more than the fractions,
2N+4 planes and N-1 dense ones: a grid's precision and phases alone say
whether it fits.  Host-only entry points; nothing here launches a kernel."""
import pytest

import workloads as W


@pytest.mark.parametrize("nx,ny", [(3, 3), (64, 64), (300, 170), (1021, 1024), (25, 4000), (4096, 4096)])
@pytest.mark.parametrize("N", [2, 3, 4])
@pytest.mark.parametrize("precision", [0, 1])
def test_workspace_bytes(nx, ny, N, precision):
    from paper_2311_10314_gb300 import _lib
    from paper_2311_10314_gb300 import build as B
    B.build()
    size = 8 if precision == 0 else 4
    _, pitch, plane = _lib.state_layout(nx, ny, N, size)
    padded = plane * size
    dense = 8 * nx * ny
    planes = 2 * 9 * N + 2 * (2 * N + 3) + N + (N - 1) + (2 * N + 4)
    small = 304 * 4 * 8 + size * ny * N + 4 * 8 + 16
    got = _lib.ddcc_workspace_bytes(_lib.make_params(W.base_params(nx, ny, N), precision))
    assert 0 < got <= planes * padded + dense * (N - 1) + small + 16 * 256
