"""The merge mode without outputs has a variant of the chunked kernel that leaves out what a zero start state makes superfluous in a
unit's first chunk.  Its states against the oracle and against the general variant, which the same call with outputs takes."""
import numpy as np
import pytest
import torch

import oracle
import paper_2608_30386_b200 as dasc
from helpers import assert_refresh_close, make_refresh_case, run_refresh_gpu, run_refresh_oracle
from paper_2608_30386_b200 import binding

pytestmark = pytest.mark.gpu

OWN, WALK, ALONE = 0, 1, 2
LENS = [9, 31, 32, 33, 64, 65, 0, 97, 1, 128]


# alone on an SM; a block per unit, two to an SM; several units to a block, first chunks in the middle of its work
@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("heads,lens,form", [(4, LENS, ALONE), (8, LENS * 2 + [129], OWN), (8, LENS * 7, WALK)])
def test_units_that_start_from_zero(kind, heads, lens, form):
    assert dasc.dasc_debug_refresh_form(len(lens), heads, sum(lens), max(lens))[0] == form
    case = make_refresh_case(81, kind, 1, heads, heads if kind == dasc.KDA else heads // 2, 128, 128, lens, scope=dasc.SCOPE_LAYER,
                             keep_ratio=0.4)
    merge = dict(mode=dasc.REFRESH_SCRATCH_MERGE_LOCAL)
    got, _ = run_refresh_gpu(case, want_o=False, **merge)
    ref, _ = run_refresh_oracle(case, mode=oracle.MODE_SCRATCH_MERGE_LOCAL, want_o=False)
    assert_refresh_close(case, got, None, ref, None, 1e-3)
    assert np.array_equal(got, run_refresh_gpu(case, **merge)[0])  # (zeros of either sign)


FORMS = [(4, [160, 9, 64, 33], ALONE), (8, [160, 9, 64, 33, 96, 31] * 5, OWN), (8, [160, 9, 64, 33, 96, 31] * 12, WALK)]


def merge_call(case, bound, algo):
    """The merge mode without outputs: states, status, counters."""
    dev, n, dense = case.state0.device, case.cu.numel() - 1, case.H_v * 128 * 128
    s, state = case.streams, case.state0.clone()
    ws = torch.zeros(dasc.dasc_refresh_workspace_bytes(case.plan, n, 1, algo), dtype=torch.uint8, device=dev)
    dasc.dasc_refresh(case.plan, state, dense, dense, torch.arange(n, dtype=torch.int32, device=dev), s.q, s.k, s.v, s.g, s.beta,
                      case.cu.to(dev), int(case.cu[-1]), bound, mode=dasc.REFRESH_SCRATCH_MERGE_LOCAL, algo=algo, workspace=ws)
    torch.cuda.synchronize()
    return state, dasc.dasc_refresh_status(ws), dasc.dasc_refresh_counters(ws)


# the chunked kernel alone: first chunks of 1 to 8 tokens, which AUTO leaves to the exact kernel, and units without tokens
@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("heads,lens,form", [(4, [1, 2, 0, 7, 8, 32, 65], ALONE), (8, [1, 2, 0, 7, 8, 32, 65] * 4, OWN),
                                             (8, [1, 2, 0, 7, 8, 32, 65] * 10, WALK)])
def test_short_first_chunks(kind, heads, lens, form):
    assert dasc.dasc_debug_refresh_form(len(lens), heads, sum(lens), max(lens))[0] == form
    case = make_refresh_case(82, kind, 1, heads, heads if kind == dasc.KDA else heads // 2, 128, 128, lens, scope=dasc.SCOPE_LAYER,
                             keep_ratio=0.4)
    state, status, _ = merge_call(case, max(lens), dasc.ALGO_CHUNKED)
    assert status == binding.OK
    ref, _ = run_refresh_oracle(case, mode=oracle.MODE_SCRATCH_MERGE_LOCAL, want_o=False)
    assert_refresh_close(case, state.cpu().numpy(), None, ref, None, 1e-3)


@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("heads,lens,form", FORMS)
def test_a_unit_that_leaves_the_range_ahead_of_others(kind, heads, lens, form):
    """It is left out with whatever it has made of the accumulator, which the first chunk of the unit behind it must replace: the longest
    requests come first in a walk, so that these have others behind them."""
    assert dasc.dasc_debug_refresh_form(len(lens), heads, sum(lens), max(lens))[0] == form
    case = make_refresh_case(83, kind, 1, heads, heads if kind == dasc.KDA else heads // 2, 128, 128, lens, scope=dasc.SCOPE_LAYER,
                             keep_ratio=0.4)
    out = [(r, h) for r in range(0, len(lens), 6) for h in (0, heads - 1)]  # requests of 160 tokens; -7 x 16 is beyond the kernel's 80
    for r, h in out:
        case.streams.g[0, int(case.cu[r]) + 40:int(case.cu[r + 1]), h] = -7.0
    left, status, _ = merge_call(case, max(lens), dasc.ALGO_CHUNKED)
    assert status == binding.ERR_DOMAIN
    state, status, counters = merge_call(case, max(lens), dasc.ALGO_AUTO)
    assert status == binding.OK and counters == (len(out), len(out))
    ref, _ = run_refresh_oracle(case, mode=oracle.MODE_SCRATCH_MERGE_LOCAL, want_o=False)
    assert_refresh_close(case, state.cpu().numpy(), None, ref, None, 1e-3)
    for r, h in out:
        state[r, 0, h] = case.state0[r, 0, h]  # the kernel alone leaves these as they were, and nothing else differs
    assert torch.equal(left.view(torch.int32), state.view(torch.int32))


@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("heads,lens,form", FORMS)
def test_a_wait_that_runs_out(kind, heads, lens, form):
    case = make_refresh_case(84, kind, 1, heads, heads if kind == dasc.KDA else heads // 2, 128, 128, lens, scope=dasc.SCOPE_LAYER,
                             keep_ratio=0.4)
    first, status, _ = merge_call(case, max(lens), dasc.ALGO_CHUNKED)
    assert status == binding.OK
    try:
        dasc.dasc_debug_set_refresh_poll_limit(1)
        state, status, _ = merge_call(case, max(lens), dasc.ALGO_CHUNKED)
    finally:
        dasc.dasc_debug_set_refresh_poll_limit(0)
    assert status == binding.ERR_TIMEOUT and torch.equal(state, case.state0)  # no unit was written back
    state, status, _ = merge_call(case, max(lens), dasc.ALGO_CHUNKED)
    assert status == binding.OK and torch.equal(state, first)                 # the next call finds nothing left over
