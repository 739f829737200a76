"""Launch rules of the chain kernel: short default launches cut their steps
into segments when the replicas do not all fit at once, and short chains with
many replicas run the five-CTA build; launches of few replicas have helper
warps for the bonded terms and the noise.  None of it changes a bit of the
result: replica (w, r) with uid u equals the same uid in a launch of few
replicas (every one resident, one segment, helpers), for 4 and 8 warps a
replica and in FP64."""
import numpy as np
import pytest

from paper_1105_4840_gb300 import inputs
from tests.helpers import f32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pmf():
    from paper_1105_4840_gb300 import pmf as m
    return m


def _run(pmf, sysh, lam, replicas, n_steps, uid_base=0):
    run = inputs.RunSettings(k=500.0, kT=inputs.kT_of(300.0), dt=0.001, gamma=5.0, n_steps=n_steps, n_equil=5,
                             stride=3, replicas=replicas, seed=23)
    rr = pmf.pmf_run_windows(sysh, lam, pmf.make_params(run, uid_base=uid_base))
    return rr.x_samples(), rr.final_state()[0].reshape(lam.size, replicas, -1)


# lengths around the five-CTA line (72 padded beads), one tile to five;
# steps below, at and off multiples of the shortest segment (16)
@pytest.mark.parametrize("prec,warps", [(0, 4), (0, 8), (1, 4)])
@pytest.mark.parametrize("n,steps", [(13, 40), (40, 16), (72, 33), (73, 17), (104, 50), (130, 35)])
def test_many_replicas_equal_few(pmf, n, steps, prec, warps):
    p = inputs.chain_params(n, 40 + n)
    start = f32(inputs.chain_start(p, 50 + n))
    lam = np.array([1.0, 1.2])
    sysh = pmf.pmf_create_system_chain([p], [start], precision=prec)
    pmf.pmf_chain_set_warps(sysh, 0, warps)
    if prec:
        steps = min(steps, 20)
    R = 450  # 900 replicas: more than five CTAs on each of 152 SMs
    xm, pm = _run(pmf, sysh, lam, R, steps)
    for w, r0 in ((0, 0), (1, R - 6)):
        xf, pf = _run(pmf, sysh, lam[w:w + 1], 6, steps, uid_base=w * R + r0)
        np.testing.assert_array_equal(xm[w][r0:r0 + 6], xf[0])
        np.testing.assert_array_equal(pm[w, r0:r0 + 6], pf[0])
