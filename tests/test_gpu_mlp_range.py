"""Surrogate MLP on the GPU at the edges of its kernels' rules: activations far
outside the range of the straight-line SiLU, and every shape of the clustered
training (2 to 8 tiles a step; 9 tiles take the per-step launches)."""
import numpy as np
import pytest

from oracle import surrogate as sg
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


@pytest.mark.parametrize("scale", [1.0, 60.0, 400.0])
def test_forward_far_from_zero(pmf, scale):
    """First-layer inputs up to a few hundred either side of zero, where
    e^-z overflows FP32: the bound is the BF16 one of the 64x64 layer (products
    of relative error 2^-8, SiLU 1.1-Lipschitz)."""
    p = _params(3)
    p["W1"] = np.asarray(p["W1"] * scale, dtype=np.float32).astype(np.float64)
    lam = np.linspace(-1.0, 1.0, 129)
    m = pmf.Mlp(pmf.pack_mlp_params(p), 0.0, 1.0)
    mu, lv = m.predict(lam)
    o = sg.forward(p, lam)
    bound = 1.1 * (2.0 ** -8 * (np.abs(o["h1"]) @ np.abs(p["W2"]).T)) @ np.abs(p["W3"]).T + 1e-5 * (1 + np.abs(o["out"]))
    assert np.all(np.abs(mu - o["out"][:, 0]) <= bound[:, 0])
    assert np.all(np.abs(lv - o["out"][:, 1]) <= bound[:, 1])
    m.close()


@pytest.mark.parametrize("tiles", [2, 3, 5, 8, 9])
def test_tiles_of_a_step(pmf, run, tiles):
    """One Adam step moves every weight by lr sign(g): split and one-CTA
    training differ only where the order of the tiles' sum turns a gradient
    of nearly zero, so in fewer than 1 % of the weights."""
    p0 = pmf.pack_mlp_params(_params(11, jitter=0.0))
    out = []
    for split in (1, 0):
        m = pmf.Mlp(p0, 0.0, 1.5)
        m.set_split(split)
        m.train(run, 1, 128 * tiles, 3e-3, 7)
        out.append(m.params())
        m.close()
    d = np.abs(out[1] - out[0])
    assert np.mean(d > 1e-6) < 0.01 and d.max() <= 2 * 3e-3
