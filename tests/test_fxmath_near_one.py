"""Logarithms of arguments near 1 (a Troe blend's F_cent comes as close as the mechanism's data do) and the
largest exponentials of csrc/fxmath.cuh, against exact decimal arithmetic.

Near 1 the logarithm is held to an absolute bound, the one its sums need.  With s = 2^7 z, |s| < 1.06, as
fx_log2_mant's argument, the upper 32 bits of s in the fourth term leave 2^-30 E_4 s^3 / 2^7 = 0.84 2^-59,
the 32-bit fourth coefficient 1.5 2^-53 s^4 / 2^7 = 0.95 2^-59, the Q62 sums, the table and the series 0.32 2^-59;
with the rounding to a double, 2.2 2^-59 + 1/2 unit in the last place.
"""
from decimal import Decimal, getcontext

import numpy as np
import pytest

from tests.test_fxmath import fx  # noqa: F401


@pytest.mark.parametrize("f", ["l", "2"])
def test_logarithms_near_one(fx, f):  # noqa: F811
    getcontext().prec = 50
    ln2 = Decimal(2).ln()
    rng = np.random.default_rng(6)
    edge = np.array([1 + i / 64.0 for i in range(8)] + [0.5 + i / 128.0 for i in range(56, 64)])  # the tables' intervals
    xs = np.concatenate([rng.uniform(0.9, 1.1, 400), 1.0 + rng.normal(size=100) * 1e-6, edge, np.nextafter(edge, 0.0),
                         np.nextafter(edge, 9.0), 1.0 + 2.0 ** -np.arange(4, 53), 1.0 - 2.0 ** -np.arange(4, 54)])
    for x, y in zip(xs, fx(f, xs)):
        ref = Decimal(float(x)).ln()
        ref = ref if f == "l" else ref / ln2
        half = Decimal(float(np.spacing(abs(float(ref))))) / 2
        assert abs(Decimal(y) - ref) <= Decimal(2.2 * 2.0 ** -59) + half, (f, x, y, float(ref))


def test_largest_exponentials(fx):  # noqa: F811
    getcontext().prec = 50
    xs = [1023.0, 1023.5, 1024.0 - 2.0 ** -30]
    for x, y in zip(xs, fx("p", xs)):
        ref = (Decimal(x) * Decimal(2).ln()).exp()
        assert abs(Decimal(y) - ref) <= Decimal(0.54) * Decimal(float(np.spacing(float(ref)))), (x, y)
