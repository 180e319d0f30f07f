"""Reciprocal and square root on the integer pipe: within 0.501 ulp of the exact
value (the final rounding, and below 0.001 for the last correction's binary32 product),
and without a bias (a packet collects it; the mean of 4e6 rounding errors is 0 to
1.5e-4 ulp, and 2e-3 is asserted), over every binary32 prefix of [1, 4) (both exponent parities), which is
all that the binary32 approximations they start from see; the 29 bits behind
each prefix are drawn.  The exact error comes from the product's own rounding
error (Dekker, 1971)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _two_prod(a, b):
    """a b = p + e exactly."""
    p = a * b
    c = 134217729.0
    ah = a * c - (a * c - a)
    bh = b * c - (b * c - b)
    al, bl = a - ah, b - bh
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


@pytest.mark.parametrize("part", range(4))
def test_every_binary32_prefix(part):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1401_5469_gb300 import mc
    n = 1 << 22
    pre = (np.arange(n, dtype=np.uint64) + np.uint64(part * n)) << np.uint64(29)
    low = np.random.default_rng(part).integers(0, 1 << 29, n, dtype=np.uint64)
    low[::5] = 0
    low[1::5] = (1 << 29) - 1
    x = ((np.uint64(1023) << np.uint64(52)) + (pre | low)).view(np.float64)
    assert x.min() >= 1.0 and x.max() < 4.0
    y = mc.mc_selftest_math(mc.MC_MATH_RCP, x)[0]
    p, e = _two_prod(x, y)
    ulps = ((1.0 - p) - e) / x / np.spacing(y)
    assert np.abs(ulps).max() <= 0.501, np.abs(ulps).max()
    assert abs(ulps.mean()) < 2e-3, ulps.mean()
    s = mc.mc_selftest_math(mc.MC_MATH_SQRT, x)[0]
    p, e = _two_prod(s, s)
    ulps = ((x - p) - e) / (2.0 * s) / np.spacing(s)
    assert np.abs(ulps).max() <= 0.501, np.abs(ulps).max()
    assert abs(ulps.mean()) < 2e-3, ulps.mean()
