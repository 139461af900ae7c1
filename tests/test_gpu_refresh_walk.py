"""The chunked kernel's CTAs replay several units one behind the other where a launch has enough of them and no request is much
longer than a CTA's share; the caller's bound on the longest request is part of that rule, so a loose bound gives every unit a
CTA of its own.  Both have to give the same bits, and the oracle's results."""
import numpy as np
import pytest
import torch

import oracle
import paper_2608_30386_b200 as dasc
from helpers import RefreshCase, assert_refresh_close, make_plans, make_refresh_case, run_refresh_oracle
from paper_2608_30386_b200 import synth

pytestmark = pytest.mark.gpu

LOOSE = 1 << 30  # tokens: no request can be that long


def replay(case, bound, mode, o_dtype, algo=dasc.ALGO_AUTO):
    dev, n = case.state0.device, case.cu.numel() - 1
    dense = case.H_v * 128 * 128
    s, state, T = case.streams, case.state0.clone(), int(case.cu[-1])
    o = None if o_dtype is None else torch.full((case.L, T, case.H_v, 128), float("nan"), device=dev, dtype=o_dtype)
    ws = torch.zeros(dasc.dasc_refresh_workspace_bytes(case.plan, n, case.L, algo), dtype=torch.uint8, device=dev)
    dasc.dasc_refresh(case.plan, state, dense, case.L * dense, torch.arange(n, dtype=torch.int32, device=dev), s.q, s.k, s.v, s.g,
                      s.beta, case.cu.to(dev), T, bound, o=o, mode=mode, algo=algo, workspace=ws)
    torch.cuda.synchronize()
    assert dasc.dasc_refresh_status(ws) == 0
    return state, o, dasc.dasc_refresh_counters(ws)


# units and lengths around what changes a walk: 2 and 3 units of 2 chunks each; single chunks, 16 units to a CTA and the step to a
# larger grid behind it (296 x 16 = 4736 units); ragged with empty requests, requests of at most 8 tokens (handed over
# from the middle of a walk) and full chunks; more requests than are put in order; 1.3 and 1.4 units to a CTA of very
# different lengths; outputs in both types and none
@pytest.mark.parametrize("kind,L,H,lens,mode,o_dtype", [
    (dasc.KDA, 1, 8, [64] * 60, dasc.REFRESH_CONTINUE, torch.bfloat16),
    (dasc.GDN, 1, 8, [50] * 111, dasc.REFRESH_CONTINUE, torch.float32),
    (dasc.KDA, 1, 32, [32] * 148, dasc.REFRESH_SCRATCH_MERGE_LOCAL, None),
    (dasc.GDN, 1, 32, [9] * 149, dasc.REFRESH_SCRATCH_MERGE_LOCAL, None),
    (dasc.KDA, 2, 8, [1, 96, 0, 33, 8, 64, 9, 31] * 12, dasc.REFRESH_CONTINUE, torch.float32),
    (dasc.KDA, 2, 8, [1, 96, 0, 33, 8, 64, 9, 31] * 12, dasc.REFRESH_SCRATCH_MERGE_LOCAL, None),
    (dasc.GDN, 2, 8, [96, 32, 0, 95, 65, 97, 2] * 14, dasc.REFRESH_CONTINUE, torch.bfloat16),
    (dasc.KDA, 1, 4, [64] * 250, dasc.REFRESH_CONTINUE, torch.bfloat16),
    (dasc.KDA, 1, 8, [129, 9, 33, 0, 64, 160, 17] * 7, dasc.REFRESH_CONTINUE, torch.float32),
    (dasc.GDN, 1, 8, [300, 9, 33, 0, 64, 600, 17, 65, 8] * 6, dasc.REFRESH_SCRATCH_MERGE_LOCAL, None),
])
def test_walked_units_match_units_of_their_own(kind, L, H, lens, mode, o_dtype):
    case = make_refresh_case(61, kind, L, H, H if kind == dasc.KDA else H // 2, 128, 128, lens, scope=dasc.SCOPE_LAYER, keep_ratio=0.4)
    if kind == dasc.KDA and L > 1:  # a unit in the middle leaves the kernel's log-decay range and is replayed exactly
        case.streams.g[1, int(case.cu[9]):int(case.cu[10]), 3, 7] = -7.0
    walked, alone = replay(case, max(lens), mode, o_dtype), replay(case, LOOSE, mode, o_dtype)
    assert walked[2] == alone[2]
    assert torch.equal(walked[0].view(torch.int32), alone[0].view(torch.int32))
    if o_dtype is not None:
        assert torch.equal(walked[1], alone[1])
    if len(lens) * L * H <= 1600 and o_dtype != torch.bfloat16:
        merge = mode != dasc.REFRESH_CONTINUE
        ref_s, ref_o = run_refresh_oracle(case, mode=oracle.MODE_SCRATCH_MERGE_LOCAL if merge else oracle.MODE_CONTINUE, want_o=not merge)
        assert_refresh_close(case, walked[0].cpu().numpy(), None if merge else walked[1].cpu().numpy(), ref_s, ref_o, 1e-3)


def _half_kept_case(kind, kept_half):
    """Requests with and without tokens; KDA: nearly all rows of one half of the channels are retained, nearly none of the other."""
    L, H, lens = 1, 8, [64, 0, 0, 40, 0, 33] * 24
    gen = synth.generator(62)
    if kind == dasc.KDA:
        rates = torch.full((L, H, 128), 0.08)
        rates[:, :, kept_half * 64:kept_half * 64 + 64] = 0.002
        rates *= 1 + 0.01 * torch.rand(rates.shape, generator=gen)
    else:
        rates = synth.decay_rates(gen, L, H, 1, 0.01, 0.1)
    plan, oplan = make_plans(kind, L, H, H if kind == dasc.KDA else H // 2, 128, 128, rates, sel=dasc.SEL_TOP_RATIO,
                             scope=dasc.SCOPE_LAYER, keep_ratio=0.48)
    cu = torch.zeros(len(lens) + 1, dtype=torch.int32)
    cu[1:] = torch.cumsum(torch.tensor(lens), 0).to(torch.int32)
    s = synth.token_streams(gen, kind, L, int(cu[-1]), H, H if kind == dasc.KDA else H // 2, 128, 128, rates)
    for f in ("q", "k", "v", "g", "beta"):
        setattr(s, f, getattr(s, f).to("cuda"))
    state0 = synth.states(gen, (len(lens), L, H, 128, 128)).to("cuda")
    return RefreshCase(kind, L, H, H if kind == dasc.KDA else H // 2, 128, 128, cu, s, state0, plan, oplan)


def replay_static(case, bound, mode):
    dev, n = case.state0.device, case.cu.numel() - 1
    dense = case.H_v * 128 * 128
    s, state = case.streams, case.state0.clone()
    scratch = dasc.dasc_refresh_static(case.plan, state, dense, case.L * dense, torch.arange(n, dtype=torch.int32, device=dev), s.q, s.k,
                                       s.v, s.g, s.beta, case.cu.to(dev), int(case.cu[-1]), bound, mode=mode)
    torch.cuda.synchronize()
    assert dasc.dasc_refresh_status(scratch) == 0
    return state


# Where the caller asks for the chunked kernel alone, requests without tokens stay in a CTA's list, behind those with tokens; in the
# merge mode they have rows to write, and nothing to wait for before they do.  Chain warps of channels 0-63 and 64-127 then end the unit
# before at different times.
@pytest.mark.parametrize("kind,kept_half", [(dasc.KDA, 0), (dasc.KDA, 1), (dasc.GDN, 0)])
def test_units_without_tokens_behind_others_in_a_walk(kind, kept_half):
    case, mode = _half_kept_case(kind, kept_half), dasc.REFRESH_SCRATCH_MERGE_LOCAL
    own = replay(case, LOOSE, mode, None, dasc.ALGO_CHUNKED)[0]
    ref_s, _ = run_refresh_oracle(case, mode=oracle.MODE_SCRATCH_MERGE_LOCAL, want_o=False)
    assert_refresh_close(case, own.cpu().numpy(), None, ref_s, None, 1e-3)
    for _ in range(6):
        assert torch.equal(replay(case, 64, mode, None, dasc.ALGO_CHUNKED)[0].view(torch.int32), own.view(torch.int32))
    assert torch.equal(replay_static(case, 64, mode).view(torch.int32), replay_static(case, LOOSE, mode).view(torch.int32))
