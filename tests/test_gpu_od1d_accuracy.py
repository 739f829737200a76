"""End positions of the 1D integrator against its map in exact arithmetic, and
their bits in launches of different company."""
from fractions import Fraction

import numpy as np
import pytest

from paper_1105_4840_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pmf():
    from paper_1105_4840_gb300 import pmf as m
    return m


@pytest.mark.parametrize("lam,b", [(8.0, 4), (-6.3, 3), (0.7, 0)])
def test_trap_without_wells(pmf, lam, b):
    """A pure trap (a = 0, k dt = 1e-3) without noise remembers 1000 steps, so a
    rounding that always goes one way adds up to 1000 of its means (the
    products' 2 1/4 units of 2^(b-62) would give 7.8e-15 at b = 4).  Rounding to either side
    leaves 1.2 units x sqrt(1000 / 2), five times that is 134 units, and 4 units for
    the offset's own 1/256; the end position is then rounded to a double."""
    run = inputs.RunSettings(k=1.0, kT=1e-40, dt=1e-3, gamma=1.0, n_steps=20000, n_equil=0, stride=100, replicas=2, seed=3)
    sysh = pmf.pmf_create_system_1d(0.0, 0.25)
    rr = pmf.pmf_run_windows(sysh, np.array([lam]), pmf.make_params(run))
    c, one = Fraction(-1e-3), 2**180  # the coefficient as the kernel has it; positions in units of 2^-180
    q = int(Fraction(1e-3 * lam) * one)
    x = one // 4
    for _ in range(run.n_steps):
        x += (x * c.numerator) // c.denominator + q
    for got in rr.final_state()[0]:
        assert abs(Fraction(float(got)) - Fraction(x, one)) <= 138 * Fraction(2) ** (b - 62) + Fraction(np.spacing(abs(got)) / 2)


def _run(pmf, a, x0, lam, replicas, steps, uid_base=0, **kw):
    run = inputs.RunSettings(**dict(dict(k=20.0, kT=1.0, dt=1e-3, gamma=1.0, n_steps=steps, n_equil=0, stride=50,
                                         replicas=replicas, seed=21), **kw))
    rr = pmf.pmf_run_windows(pmf.pmf_create_system_1d(a, x0), np.asarray(lam, dtype=np.float64),
                             pmf.make_params(run, uid_base=uid_base))
    return np.asarray(rr.final_state()[0]).reshape(len(lam), replicas)


@pytest.mark.parametrize("a,lam", [(0.0, [-5.0, 0.0, 0.3, 2.0**20]), (2.0, [-1.5, 0.0, 1.2, 3.1, 30.0])])
def test_bits_do_not_depend_on_the_other_windows(pmf, a, lam):
    """Each window alone (same uids) and beside the others: the traps far away
    neither widen its fixed-point range nor send it to FP64."""
    together = _run(pmf, a, -0.4, lam, 3, 700)
    for w, l in enumerate(lam):
        assert np.array_equal(_run(pmf, a, -0.4, [l], 3, 700, uid_base=3 * w)[0], together[w]), l


@pytest.mark.parametrize("start", [None, 5.5])
def test_bits_do_not_depend_on_the_number_of_simulations(pmf, start):
    """The same uids in launches of 2 and of 2100 simulations, whose steps come
    in blocks of 8160 and 3960: from inside the range, and from outside (FP64
    until it is back)."""
    got = []
    for replicas in (2, 2100):
        run = inputs.RunSettings(k=20.0, kT=1.0, dt=1e-3, gamma=1.0, n_steps=8500, n_equil=3, stride=7, replicas=replicas, seed=9)
        sysh, prm = pmf.pmf_create_system_1d(0.5, -1.0), pmf.make_params(run)
        rr = (pmf.pmf_run_prepare(sysh, np.array([0.3]), prm) if start is None else
              pmf.pmf_run_prepare_seeded(sysh, np.array([0.3]), prm, np.full(replicas, start)))
        rr.launch()
        rr.wait()
        got.append((np.asarray(rr.final_state()[0])[:2], np.asarray(rr.x_samples()[0])[:2]))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])


@pytest.mark.parametrize("dt", [1e-3, 0.02])
def test_pulled_bits_do_not_depend_on_the_number_of_simulations(pmf, dt):
    got = []
    for replicas in (2, 2100):
        run = inputs.RunSettings(k=20.0, kT=1.0, dt=dt, gamma=1.0, n_steps=8500, n_equil=30, stride=10, replicas=replicas, seed=9)
        rr = pmf.pmf_run_prepare_smd(pmf.pmf_create_system_1d(2.0, -1.0), -1.2, 0.25e-3 / dt, pmf.make_params(run))
        rr.launch()
        rr.wait()
        got.append((np.asarray(rr.final_state()[0])[:2], np.asarray(rr.x_samples()[0])[:2], np.asarray(rr.smd_work())[:2]))
    for small, large in zip(*got):
        assert np.array_equal(small, large)
