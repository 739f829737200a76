"""The reductions' splits: 1, 2, 4 or 8 warps per replica, one or several
turns of a CTA over a window's replicas, halves of 128 threads over the
replicas of a window, profile warps whose lanes own one or more windows.
Sizes at the edges of each, against the FP64 oracle, with the tolerances of
the reduction's parity tests (1e-12 of the profile, 1e-8 of the errors)."""
import numpy as np
import pytest

from oracle import estimators as est
from paper_1105_4840_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pmf():
    from paper_1105_4840_gb300 import pmf as m
    return m


def _compare(g, o, kT):
    for key in ("dF_JE", "dF_fluct", "dF_G", "dF_com", "uncertainty", "W_mean", "acc_force"):
        assert np.all(np.abs(g[key] - o[key]) <= 1e-12 * np.maximum(np.abs(o[key]), kT)), key
    for key in ("mean_x", "var_x", "gamma2"):
        np.testing.assert_allclose(g[key], o[key], rtol=1e-10, err_msg=key)
    for key in ("se_JE", "se_fluct", "var_ZW"):
        np.testing.assert_allclose(g[key], o[key], rtol=1e-8, equal_nan=True, err_msg=key)


# (windows, replicas, samples): team sizes change at 256, 512 and 1024 samples
# (few replicas); 3648 replicas fill the GPU with one warp each and 19456 give
# a CTA two turns; halves fill at 128 replicas; profile lanes own one window up to
# 32, two up to 64
@pytest.mark.parametrize("s,R,T", [(2, 2, 255), (2, 3, 256), (3, 2, 511), (3, 5, 512), (2, 3, 1023), (2, 2, 1025),
                                   (3, 31, 7), (3, 33, 5), (2, 127, 9), (2, 129, 16), (3, 257, 17), (32, 2, 3), (33, 3, 2),
                                   (65, 2, 4), (16, 228, 33), (4, 4865, 18)])
def test_teams_and_turns(pmf, s, R, T):
    lam = inputs.lambda_grid(1.3, 1.3 + 0.1 * (s - 1), s)
    k, kT = 500.0, inputs.kT_of(300.0)
    x = inputs.gaussian_x_samples(lam, k, kT, R, T, seed=s * 1000 + R)
    g = pmf.pmf_free_energy_from_samples(x.ravel(), lam, R, [T] * s, k, kT)
    xd = [x[i].astype(np.float64) for i in range(s)]
    _compare(g, est.free_energy_from_partials(est.window_partials(xd, lam, k, kT), lam, k, kT), kT)


def test_ragged_windows_share_one_team_size(pmf):
    """Windows of 1 to 3000 samples a replica: the team size follows the
    longest, short windows leave most of their team without a sample."""
    lam = np.array([-0.5, -0.1, 0.2, 0.9])
    k, kT, R, T = 20.0, 1.0, 3, [3000, 1, 40, 700]
    g = np.random.default_rng(6)
    xs = [(l + 0.2 * g.standard_normal((R, t))).astype(np.float32) for l, t in zip(lam, T)]
    got = pmf.pmf_free_energy_from_samples(np.concatenate([b.ravel() for b in xs]), lam, R, T, k, kT)
    xd = [b.astype(np.float64) for b in xs]
    _compare(got, est.free_energy_from_partials(est.window_partials(xd, lam, k, kT), lam, k, kT), kT)


def test_partials_without_samples_and_a_lone_weight(pmf):
    """Replicas without samples, and one replica with 1e10 times the others'
    weight: the leave-one-out sum of the others must survive the cut of the
    exponential sums."""
    s, R, k, kT = 3, 140, 500.0, inputs.kT_of(300.0)
    lam = np.array([1.3, 1.4, 1.55])
    g = np.random.default_rng(2)
    P = np.zeros((s, R, 5))
    P[:, :, 0] = 1.0 + 0.5 * g.standard_normal((s, R))
    P[:, :, 1] = 1.0 + 10.0 * g.random((s, R))
    P[:, :, 2] = 50.0
    P[:, :, 3] = 1.0 * g.standard_normal((s, R))
    P[:, :, 4] = 0.15 + P[:, :, 3] ** 2 / 50.0
    P[0, 100, 0] -= 23.0 * kT  # e^23 = 1e10 of the others' weight
    P[:, 7] = [np.inf, 0.0, 0.0, 0.0, 0.0]
    got = pmf.pmf_free_energy_from_partials(P, lam, k, kT)
    want = est.free_energy_from_partials(P, lam, k, kT)
    _compare(got, want, kT)
