"""Nothing that a call of the reductions leaves in its scratch reaches the next
one: the allocation-free call after its counter of finished windows was left
anywhere."""
import numpy as np
import pytest

from paper_1105_4840_gb300 import inputs
from tests.test_zz_no_alloc import FIELDS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pmf():
    from paper_1105_4840_gb300 import pmf as m
    return m


@pytest.mark.parametrize("s,left", [(5, 1), (5, 4), (5, 1000), (1000, 1), (1000, 500), (1000, 999), (1000, 2**32 - 1)])
def test_noalloc_after_a_counter_left_behind(pmf, s, left):
    """The call before is on other samples, so that a window read before its
    combination shows; with many windows the first to finish is far ahead of the last."""
    torch = pytest.importorskip("torch")
    R, T = 16, 32
    lam = inputs.lambda_grid(1.3, 1.3 + 0.1 * (s - 1), s)
    k, kT = 500.0, inputs.kT_of(300.0)
    ld = torch.from_numpy(lam.copy()).cuda()
    xs = [torch.from_numpy(inputs.gaussian_x_samples(lam, k, kT, R, T, seed=q).ravel()).cuda() for q in (5, 6)]

    def call(x):
        o = torch.full((len(FIELDS), s), float("nan"), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        pmf.pmf_free_energy_noalloc(x.data_ptr(), ld.data_ptr(), s, R, T, k, kT, o.data_ptr())
        torch.cuda.synchronize()
        return o.cpu().numpy()

    pmf.pmf_noalloc_set_counter(0)
    want = call(xs[0])
    for _ in range(3):
        call(xs[1])
        pmf.pmf_noalloc_set_counter(left)
        assert np.array_equal(call(xs[0]), want, equal_nan=True)
    assert np.isfinite(want[1]).all()
