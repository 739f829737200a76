"""Clustered training (2 to 8 tiles a step) against launches per step, and a
call of n steps against n calls of one: the same bits.  The cluster keeps
Adam's moments in registers, the next step's samples and bias corrections ahead, and
is launched again after 10 000 steps."""
import numpy as np
import pytest

from paper_1105_4840_gb300 import inputs
from tests.test_gpu_mlp import _params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pmf():
    from paper_1105_4840_gb300 import pmf as m
    return m


@pytest.fixture(scope="module")
def run(pmf):
    w = inputs.od1d_workload()
    sysh = pmf.pmf_create_system_1d(w["a"], w["x0"])
    return pmf.pmf_run_windows(sysh, w["run"].lambdas, pmf.make_params(w["run"]))


def _train(pmf, run, tiles, calls, cluster=True):
    m = pmf.Mlp(pmf.pack_mlp_params(_params(11, jitter=0.0)), 0.0, 1.5)
    m.set_cluster(cluster)
    for steps in calls:
        loss = m.train(run, steps, 128 * tiles, 3e-3, 7)
    out = m.params()
    m.close()
    assert np.isfinite(out).all()
    return out.view(np.uint32), loss


@pytest.mark.parametrize("tiles", [2, 3, 5, 8, 9])
def test_same_bits_as_launches_per_step(pmf, run, tiles):
    want, want_loss = _train(pmf, run, tiles, [37], cluster=False)
    for calls in ([37], [1] * 37, [5, 30, 2]):
        got, loss = _train(pmf, run, tiles, calls)
        assert np.array_equal(got, want) and loss == want_loss


def test_same_bits_across_the_relaunch(pmf, run):
    want, want_loss = _train(pmf, run, 2, [10_003], cluster=False)
    got, loss = _train(pmf, run, 2, [10_003])
    assert np.array_equal(got, want) and loss == want_loss
