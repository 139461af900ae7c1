"""Which form of the chunked refresh kernel a call gets, by its sizes alone (host arithmetic)."""
import pytest

import paper_2608_30386_b200 as dasc

OWN, WALK, ALONE = 0, 1, 2


@pytest.mark.parametrize("bound", [1 << 20, (1 << 31) - 32, (1 << 31) - 31, (1 << 31) - 1])
@pytest.mark.parametrize("n_req,units", [(80, 8), (300, 8), (128, 24)])
def test_a_bound_that_says_nothing_gives_every_unit_a_block(bound, n_req, units):
    assert dasc.dasc_debug_refresh_form(n_req, units, n_req * 200, bound) == (OWN, n_req * units)
