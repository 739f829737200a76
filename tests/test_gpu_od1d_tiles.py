"""The 1D integrator's tiles (40 steps x 32 simulations per CTA) and its two
arithmetics, against the FP64 oracle: fixed point where the launch's
parameters bound the motion, FP64 where they do not, and a switch in mid-run
for a simulation that leaves the range.

Tolerances: samples are the position rounded to FP32, at most half a unit in
the last place (2^-23 relative spacing, |x| < 4: 2.4e-7) apart unless the two
roundings fall on different sides, then one: 5e-7 absolute, relative for
larger positions.  End positions are doubles of a contracting map whose FP64
rounding is 1e-16 a step: 1e-13; the unstable case multiplies errors by the
growth of the map."""
import numpy as np
import pytest

from oracle import _clib, spp
from paper_1105_4840_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pmf():
    from paper_1105_4840_gb300 import pmf as m
    return m


def _settings(**kw):
    d = dict(k=20.0, kT=1.0, dt=1e-3, gamma=1.0, n_steps=100, n_equil=0, stride=1, replicas=3, seed=8)
    d.update(kw)
    return inputs.RunSettings(**d)


def _check(pmf, a, x0, lam, run, spw=None, uid_base=0, rtol=0.0, ptol=1e-13):
    sysh = pmf.pmf_create_system_1d(a, x0)
    rr = pmf.pmf_run_windows(sysh, lam, pmf.make_params(run, n_steps_per_window=spw, uid_base=uid_base))
    xs, pos = rr.x_samples(), rr.final_state()[0].reshape(lam.size, run.replicas)
    for w in range(lam.size):
        n = run.n_steps if spw is None else spw[w]
        for r in range(run.replicas):
            x, end = _clib.od1d_run(a, lam[w], run.k, run.kT, run.gamma, run.dt, n, run.n_equil, run.stride, run.seed,
                                    uid_base + w * run.replicas + r, x0)
            np.testing.assert_allclose(xs[w][r], x, atol=5e-7, rtol=max(rtol, 2.4e-7))
            np.testing.assert_allclose(pos[w, r], end, atol=ptol, rtol=max(rtol, ptol))


@pytest.mark.parametrize("steps,equil,stride", [(1, 0, 1), (31, 30, 1), (32, 0, 32), (33, 1, 31), (40, 0, 40), (41, 39, 1), (64, 7, 3), (97, 0, 96), (513, 0, 16),
                                                (8224, 4600, 1)])
@pytest.mark.parametrize("windows,replicas", [(1, 1), (3, 11), (2, 16)])
def test_tile_edges(pmf, steps, equil, stride, windows, replicas):
    lam = np.linspace(-1.2, 1.0, windows) if windows > 1 else np.array([0.4])
    _check(pmf, 2.0, -1.0, lam, _settings(n_steps=steps, n_equil=equil, stride=stride, replicas=replicas))


def test_ragged_windows(pmf):
    lam = np.array([-1.0, -0.2, 0.5, 1.4])
    _check(pmf, 2.0, -1.0, lam, _settings(n_equil=5, stride=4, replicas=9), spw=[9, 33, 64, 200], uid_base=5)


# dt 0.02: a step from inside the range could wrap; k tiny: the range needed
# is wide against the wells; a = 0: a pure trap of small extent
@pytest.mark.parametrize("a,k,dt", [(2.0, 20.0, 0.02), (2.0, 0.01, 1e-3), (0.0, 1e8, 1e-9), (0.0, 2.0, 0.05)])
def test_other_ranges(pmf, a, k, dt):
    lam = np.array([-0.5, 0.25])
    _check(pmf, a, -0.4, lam, _settings(k=k, dt=dt, n_steps=150, stride=7, replicas=5), ptol=1e-12)


def test_leaving_the_range_in_mid_run(pmf):
    """An inverted well: the trajectories start inside the fixed-point range,
    |x| < 4, leave it within the second tile and go on in FP64 (the map
    multiplies an error by about 30 over the run)."""
    lam = np.array([0.9, 1.3])
    run = _settings(k=1.0, kT=0.01, dt=5e-3, n_steps=45, replicas=20)
    ends = [_clib.od1d_run(-0.1, lam[0], 1.0, 0.01, 1.0, 5e-3, 45, 0, 1, run.seed, u, 2.5)[1] for u in range(20)]
    assert min(ends) > 4.0 and max(ends) < 100.0
    _check(pmf, -0.1, 2.5, lam, run, ptol=1e-12)


def test_start_outside_the_range(pmf):
    lam = np.array([-0.5, 0.25])
    run = _settings(n_steps=45, stride=2, replicas=4)
    start = np.array([0.1, 5.5, -6.0, 1.0, 0.0, 4.5, 3.9, -4.1])
    sysh = pmf.pmf_create_system_1d(0.5, 0.0)
    rr = pmf.pmf_run_prepare_seeded(sysh, lam, pmf.make_params(run), start)
    rr.launch()
    rr.wait()
    xs = rr.x_samples()
    for w in range(2):
        for r in range(4):
            x, _ = _clib.od1d_run(0.5, lam[w], run.k, run.kT, run.gamma, run.dt, run.n_steps, 0, 2, run.seed, 4 * w + r,
                                  start[4 * w + r])
            np.testing.assert_allclose(xs[w][r], x, atol=5e-7, rtol=2.4e-7)


@pytest.mark.parametrize("replicas,steps,equil,stride,dt", [(1, 40, 0, 1, 1e-3), (33, 130, 31, 7, 1e-3),
                                                            (40, 8300, 32, 100, 1e-3), (5, 90, 10, 8, 0.02)])
def test_pulling_work(pmf, replicas, steps, equil, stride, dt):
    """Work records: fixed-point sums across launches (8192 steps each) and
    the FP64 form (dt 0.02)."""
    run = _settings(n_steps=steps, n_equil=equil, stride=stride, replicas=replicas, dt=dt)
    v = 0.5e-3 / dt
    rr = pmf.pmf_run_prepare_smd(pmf.pmf_create_system_1d(2.0, -1.0), -1.2, v, pmf.make_params(run, uid_base=2))
    rr.launch()
    rr.wait()
    xs, W = rr.x_samples()[0], rr.smd_work()
    for r in range(replicas):
        xo, wo = _clib.od1d_smd(2.0, -1.2, v * dt, run.k, run.kT, run.gamma, dt, steps, equil, stride, run.seed, 2 + r, -1.0)
        np.testing.assert_allclose(xs[r], xo, atol=5e-7, rtol=2.4e-7)
        np.testing.assert_allclose(W[r], wo, atol=1e-11, rtol=1e-11)


def test_sequential_window_boundaries_inside_tiles(pmf):
    run = _settings(n_steps=45, n_equil=4, stride=5, replicas=35)
    lam = np.linspace(-1.0, 1.0, 5)
    rr = pmf.pmf_run_prepare_sequential(pmf.pmf_create_system_1d(2.0, -1.0), lam, pmf.make_params(run))
    rr.launch()
    rr.wait()
    xo, xf = spp.od1d_spp(2.0, -1.0, lam, run)
    for x, want in zip(rr.x_samples(), xo):
        np.testing.assert_allclose(x, want, atol=5e-7, rtol=2.4e-7)
    np.testing.assert_allclose(rr.final_state()[0], xf, atol=1e-13, rtol=1e-13)
