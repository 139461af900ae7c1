"""Which form of the chunked refresh kernel a call gets, by its sizes alone (host arithmetic)."""
import pytest

import paper_2608_30386_b200 as dasc

OWN, WALK, ALONE = 0, 1, 2


@pytest.mark.parametrize("bound", [1 << 20, (1 << 31) - 32, (1 << 31) - 31, (1 << 31) - 1])
@pytest.mark.parametrize("n_req,units", [(80, 8), (300, 8), (128, 24)])
def test_a_bound_that_says_nothing_gives_every_unit_a_block(bound, n_req, units):
    assert dasc.dasc_debug_refresh_form(n_req, units, n_req * 200, bound) == (OWN, n_req * units)


@pytest.mark.parametrize("kind_of_call", ["bound x 1", "bound x 4", "bound x 1000", "window"])
@pytest.mark.parametrize("tokens", [9, 40, 95, 100, 300, 1000])
def test_above_an_sm_each_the_bound_does_not_decide_for_one_block_per_sm(kind_of_call, tokens):
    # even lengths, which the host cannot tell from one long request among short ones by any upper bound
    for n_req in range(38, 75):  # x 4 heads: 152 .. 296 units
        window = 512 if kind_of_call == "window" else 0
        bound = window or tokens * int(kind_of_call.split()[-1])
        assert dasc.dasc_debug_refresh_form(n_req, 4, n_req * tokens, bound, window) == (OWN, n_req * 4)


def test_long_requests_leave_half_of_the_sms_to_other_streams():
    for units in (1, 32, 74):
        assert dasc.dasc_debug_refresh_form(1, units, 1 << 20, 1 << 20) == (ALONE, units)
    for units in (75, 128, 148):
        assert dasc.dasc_debug_refresh_form(1, units, 2048, 2048) == (ALONE, units)
        assert dasc.dasc_debug_refresh_form(1, units, 2049, 2049) == (OWN, units)
        assert dasc.dasc_debug_refresh_form(1, units, 300, 1 << 30) == (ALONE, units)  # no request is longer than all tokens
    assert dasc.dasc_debug_refresh_form(1, 149, 300, 300) == (OWN, 149)


@pytest.mark.parametrize("tokens", [300, 700, 1000])
def test_a_bound_of_twice_the_length_does_not_make_blocks_walk_where_that_could_lose(tokens):
    for n_req, form in ((104, OWN), (106, OWN), (110, OWN), (111, WALK), (120, WALK), (148, WALK)):  # x 4 heads: 416 .. 592 units
        assert dasc.dasc_debug_refresh_form(n_req, 4, n_req * tokens, 2 * tokens)[0] == form
