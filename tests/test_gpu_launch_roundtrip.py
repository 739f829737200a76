"""What pmf_chain_get_launch reports can be handed back to pmf_chain_set_grid:
a launch shape left to the library stays with the library."""
import pytest

from paper_1105_4840_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ctas,seg", [(0, 0), (0, 16), (0, 1000), (-1, 0), (300, 250)])
def test_launch_shape_round_trip(ctas, seg):
    from paper_1105_4840_gb300 import pmf

    p = inputs.chain_params(24, 1)
    sysh = pmf.pmf_create_system_chain([p], [inputs.chain_start(p, 2)])
    assert pmf.pmf_chain_get_launch(sysh, 0)[1:] == (0, 0)
    pmf.pmf_chain_set_grid(sysh, 0, ctas, seg)
    w, c, g = pmf.pmf_chain_get_launch(sysh, 0)
    assert (c, g) == (ctas, seg)
    pmf.pmf_chain_set_grid(sysh, 0, c, g)
    assert pmf.pmf_chain_get_launch(sysh, 0) == (w, ctas, seg)
