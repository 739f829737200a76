"""The surrogate's straight-line SiLU against CUDA's own divisions, bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


def test_every_float():
    """All 2^32 arguments, both edges of the straight lines (-69 and 2^100),
    denormals, infinities and NaNs among them."""
    from paper_1105_4840_gb300 import pmf

    assert pmf.pmf_mlp_silu_check(0, 2**32) == 0
