"""The FP64 reciprocal, square root and clamp of the node update against the
correctly rounded operators.

The bar: from a seed of relative error below 2^-19 the truncation of both is
below 2^-56 of the value, an eighth of a unit in the last place, so with the
final rounding each result lies within 0.63 units of the exact value and is
one of the two numbers next to it: at most one unit from the rounded one."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def math64():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10314_gb300 import build as B
    B.build()
    from paper_2311_10314_gb300 import _lib

    def run(x):
        d = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        out = torch.empty((5, d.numel()), dtype=torch.float64, device="cuda")
        st = _lib.ddcc_selftest_math64(torch.cuda.current_stream().cuda_stream, d.data_ptr(), out.data_ptr(), d.numel())
        assert st == _lib.DDCC_OK
        return out.cpu().numpy()
    return run


def _ulps(a, b):
    """Distance in units in the last place of values of one sign."""
    return np.abs(a.view(np.int64) - b.view(np.int64))


def _arguments(lo, hi, n, seed):
    """n numbers with exponents spread over [lo, hi) and random mantissas, and
    mantissas next to the powers of two."""
    rng = np.random.default_rng(seed)
    e = rng.integers(lo, hi, n)
    m = rng.random(n)
    m[: n // 8] = rng.integers(0, 64, n // 8) * 2.0 ** -52
    m[n // 8: n // 4] = 1.0 - rng.integers(1, 64, n // 4 - n // 8) * 2.0 ** -52
    return np.ldexp(1.0 + m, e)


@pytest.mark.parametrize("lo,hi", [(-4, 4), (-60, 20), (-1022, 1024)])
def test_one_unit_from_the_operators(math64, lo, hi):
    x = _arguments(lo, hi, 1 << 20, seed=hi)
    x[: 1 << 10] = 1e-6 * (1.0 + np.arange(1 << 10) / (1 << 10))     # the smallest psi in use
    got = math64(x)
    rcp, root = 1.0 / x, np.sqrt(x)
    normal = x < 2.0 ** 1021       # reciprocals above 2^-1021
    print("rcp: max %d, share %.4f; root: max %d, share %.5f" % (
        _ulps(got[0], rcp)[normal].max(), (got[0] != rcp)[normal].mean(), _ulps(got[1], root).max(), (got[1] != root).mean()))
    assert _ulps(got[0], rcp)[normal].max() <= 1
    assert _ulps(got[1], root).max() <= 1
    assert np.array_equal(math64(-x)[0], -got[0])
    # the seeds the bar rests on
    s = np.abs(got[3] * x - 1.0)[normal].max()
    y = np.abs(got[4] * root - 1.0).max()
    print("seed errors 2^%.2f, 2^%.2f" % (np.log2(s), np.log2(y)))
    assert s < 2.0 ** -19 and y < 2.0 ** -19


def test_ends_of_the_range(math64):
    """Zero, infinity and not-a-number as the operators have them; subnormal
    arguments as zero; results beyond the normal numbers within 2^-1021."""
    tiny, top = np.finfo(np.float64).tiny, np.finfo(np.float64).max
    got = math64(np.array([0.0, -0.0, 5e-324, -1e-310, np.nextafter(tiny, 0), np.inf, -np.inf, np.nan, -1.0, -tiny]))
    inf, nan = np.inf, np.nan
    assert np.array_equal(got[0][:8], [inf, -inf, inf, -inf, inf, 0.0, -0.0, nan], equal_nan=True)
    assert np.array_equal(got[1], [0.0, 0.0, 0.0, 0.0, 0.0, inf, nan, nan, nan, nan], equal_nan=True)
    assert np.array_equal(got[2], [0.0, 0.0, 5e-324, 0.0, np.nextafter(tiny, 0), inf, 0.0, 0.0, 0.0, 0.0])
    x = np.array([tiny, np.nextafter(2.0 ** 1021, 0), 2.0 ** 1021, 2.0 ** 1022, 2.0 ** 1023, top])
    got = math64(x)
    assert _ulps(got[0][:2], 1.0 / x[:2]).max() <= 1
    assert np.abs(got[0][2:] - 1.0 / x[2:]).max() <= 2.0 ** -1021
    assert _ulps(got[1], np.sqrt(x)).max() <= 1
