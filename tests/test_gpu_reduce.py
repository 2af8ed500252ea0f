"""The fixed-point block sums of the reductions, through the dot product:
FP64's range, infinities, NaN and cancellation.  Tolerance as
tests/test_gpu_blas1.py: 1e-13 of sum |x_i y_i| (reordered FP64 sums)."""
import math

import numpy as np
import pytest

from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 257, 1025, 300_001])
def test_dot_range_and_special_values(gko, n):
    G = gko
    rng = np.random.default_rng(n)
    x, y = rng.uniform(-1, 1, n), rng.uniform(-1, 1, n)
    d = G.gko_dot(dev(x), dev(y))
    for k in (-900, -300, 300, 900):  # powers of two: the same digits
        assert G.gko_dot(dev(np.ldexp(x, k)), dev(y)) == math.ldexp(d, k)
    wide = np.ldexp(x, rng.integers(-500, 500, n))  # addends of any size: those far below the largest vanish
    assert abs(G.gko_dot(dev(wide), dev(y)) - math.fsum(wide * y)) <= 1e-13 * math.fsum(np.abs(wide * y))
    tiny = np.full(n, 5e-324)  # subnormal sums are exact
    assert G.gko_dot(dev(tiny), dev(np.ones(n))) == n * 5e-324
    assert G.gko_dot(dev(np.zeros(n)), dev(y)) == 0.0
    one = np.ones(n)
    for v in (np.inf, -np.inf):
        z = x.copy()
        z[n // 2] = v
        assert G.gko_dot(dev(z), dev(one)) == v
    z[0] = np.nan
    assert math.isnan(G.gko_dot(dev(z), dev(one)))
    if n > 1:
        z = x.copy()
        z[0], z[-1] = np.inf, -np.inf
        assert math.isnan(G.gko_dot(dev(z), dev(one)))
