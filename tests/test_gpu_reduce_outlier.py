"""The jackknife of the exponential average where one replica outweighs all
others, up to 110 kT above them: the leave-one-out sums against sums in
extended precision.

Tolerance: the sum that is left has the relative rounding of a sum of up to 600
positive terms, at most 16 x 2^-53, its logarithm of at least 20 then 1e-16, and the
spread's two sums lose a factor of 2 at most: 1e-12 is far outside that and
far inside an error of the sum left (1e-11 at 47 kT if the largest term's
rounding reaches it)."""
import math
from fractions import Fraction

import numpy as np
import pytest

from paper_1105_4840_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pmf():
    from paper_1105_4840_gb300 import pmf as m
    return m


def _expected_se(P, k, kT):
    """Standard errors of the profile's increments, first window alone."""
    R = P.shape[0]
    m = P[:, 0].min()
    e = [Fraction(float(s)) * Fraction(math.exp(-(float(w) - m) / kT)) for w, s in zip(P[:, 0], P[:, 1])]
    total, n = sum(e), P[:, 2].sum()

    def log(q):  # of a Fraction, to double precision whatever its size
        shift = q.numerator.bit_length() - q.denominator.bit_length()
        return math.log(float(q / Fraction(2) ** shift)) + shift * math.log(2.0)

    loo = [-kT * log((total - v) / Fraction(float(n - c))) for v, c in zip(e, P[:, 2])]
    mean = math.fsum(loo) / R
    return math.sqrt((R - 1) / R * math.fsum((v - mean) ** 2 for v in loo))


@pytest.mark.parametrize("above", [20.0, 47.0, 61.0, 75.0, 110.0])
@pytest.mark.parametrize("R", [2, 7, 32, 130, 600])
def test_one_replica_above_all_others(pmf, R, above):
    lam, k, kT = np.array([1.3, 1.4]), 500.0, inputs.kT_of(300.0)
    g = np.random.default_rng(R)
    P = np.zeros((2, R, 5))
    P[:, :, 0] = 1.0 + 0.5 * g.standard_normal((2, R))
    P[:, :, 1] = 1.0 + 10.0 * g.random((2, R))
    P[:, :, 2] = 50.0
    P[:, :, 3] = g.standard_normal((2, R))
    P[:, :, 4] = 0.15 + P[:, :, 3] ** 2 / 50.0
    P[0, R // 2, 0] = P[0, :, 0].min() - above * kT
    got = pmf.pmf_free_energy_from_partials(P, lam, k, kT)
    want = _expected_se(P[0], k, kT)
    assert abs(got["se_JE"][1] - want) <= 1e-12 * want
