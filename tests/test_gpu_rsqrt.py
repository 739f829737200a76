"""The FP64 pairs' reciprocal square root against integer square roots, on both
sides of the exponents where it hands over to the library's function."""
import math
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _ulps(v, y):
    """|y - 1/sqrt(v)| in units in the last place of y."""
    q = 1 / Fraction(v)
    s = max(0, 200 - (q.numerator.bit_length() - q.denominator.bit_length()) // 2)  # at least 200 bits of the root
    exact = Fraction(math.isqrt((q.numerator << (2 * s)) // q.denominator), 1 << s)
    return float(abs(Fraction(y) - exact) / Fraction(float(np.spacing(y))))


def test_within_1_02_units_in_the_last_place():
    """The seed (FP32, within 2 units of 2^-23 of a truncated argument) leaves e below
    2^-20.7, its cube 2^-63; the residual is rounded at 2^-53, half of which
    reaches the result, and the last operation rounds by half a unit."""
    from paper_1105_4840_gb300 import pmf

    g = np.random.default_rng(3)
    v = [g.uniform(1.0, 4.0, 4000), 2.0 ** g.uniform(-30, 30, 4000), 2.0 ** g.uniform(-119.9, 120.9, 4000)]
    edge = 2.0 ** np.array([-120.0, -119.0, 120.0, 121.0])
    v += [edge, np.nextafter(edge, 0), np.nextafter(edge, np.inf), np.nextafter(2.0 ** np.arange(-40.0, 40.0), 0)]
    v += [1.0 + np.arange(64) * 2.0**-52, 4.0 - np.arange(1, 64) * 2.0**-51]
    v += [2.0 ** g.uniform(-1000, -121, 500), 2.0 ** g.uniform(121, 1000, 500), np.array([1e-300, 1e300, 5e-324])]
    v = np.concatenate(v)
    y = pmf.pmf_rsqrt(v)
    assert max(_ulps(float(a), float(b)) for a, b in zip(v, y)) <= 1.02
    special = pmf.pmf_rsqrt(np.array([0.0, np.inf, np.nan]))
    assert special[0] == np.inf and special[1] == 0.0 and np.isnan(special[2])
