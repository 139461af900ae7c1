"""Calls of more than 148 units, where two blocks of the chunked kernel share an SM and may replay several units each: padded strides, a
permuted request map, layer ranges, windows, units outside the log-decay range, repeated launches.  Up to 148 units a block has an SM to
itself; that form is held to the oracle by the other tests, and gives the same bits, so each large call is compared with the same
requests in small calls (and a few of its units with the oracle)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2608_30386_b200 as dasc
from helpers import make_plans, rel_err
from helpers_fullsize import oracle_one_unit
from paper_2608_30386_b200 import binding, synth

pytestmark = pytest.mark.gpu

OWN, WALK, ALONE = 0, 1, 2
GUARD = -123.0
LOOSE = 1 << 30


class Large:
    """`lens` requests on layers [1, L) of a plan with three layers, states in a padded layout, request i in slot slots[i]."""

    def __init__(self, seed, kind, H, lens, strong=()):
        gen, rng = synth.generator(seed), np.random.default_rng(seed)
        self.kind, self.H, self.H_k, self.lens, self.L, self.lb = kind, H, H if kind == dasc.KDA else H // 2, lens, 3, 1
        rates = synth.decay_rates(gen, self.L, H, 128 if kind == dasc.KDA else 1, 1e-3, 1.0)
        self.plan, self.oplan = make_plans(kind, self.L, H, self.H_k, 128, 128, rates, sel=dasc.SEL_TOP_RATIO, scope=dasc.SCOPE_LAYER,
                                           keep_ratio=0.4)
        self.cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
        s = synth.token_streams(gen, kind, self.L - self.lb, int(self.cu[-1]), H, self.H_k, 128, 128, rates[self.lb:])
        for r, l, h in strong:  # a log-decay that the chunked kernel's factors cannot carry
            s.g[(l, slice(self.cu[r], self.cu[r + 1]), h) + ((5,) if kind == dasc.KDA else ())] = -7.0
        self.s = [getattr(s, f).to("cuda") for f in ("q", "k", "v", "g", "beta")]
        dense = H * 128 * 128
        self.layer_stride, n = dense + 256, len(lens) + 2
        self.req_stride = self.L * self.layer_stride + 128
        self.slots = rng.permutation(n)[:len(lens)].astype(np.int32)
        self.state0 = torch.full((n, self.req_stride), GUARD, device="cuda")
        for l in range(self.L):
            self.state0[:, l * self.layer_stride:l * self.layer_stride + dense] = synth.states(gen, (n, dense)).to("cuda")

    def units(self, n=None):
        return (len(self.lens) if n is None else n) * (self.L - self.lb) * self.H

    def call(self, state, lo, hi, *, bound=None, o=None, window=0, **kw):
        """Requests lo .. hi - 1; returns (outputs, workspace, first replayed tokens)."""
        t0, t1 = int(self.cu[lo]), int(self.cu[hi])
        q, k, v, g, beta = (x[:, t0:t1].contiguous() for x in self.s)
        ids = torch.from_numpy(self.slots[lo:hi]).to("cuda")
        cu = torch.from_numpy((self.cu[lo:hi + 1] - t0).astype(np.int32)).to("cuda")
        out = None if o is None else torch.full((self.L - self.lb, t1 - t0, self.H, 128), float("nan"), device="cuda", dtype=o)
        ws = torch.zeros(dasc.dasc_refresh_workspace_bytes(self.plan, hi - lo, self.L - self.lb), dtype=torch.uint8, device="cuda")
        wb = torch.full((hi - lo,), -1, dtype=torch.int32, device="cuda")
        if window:
            dasc.dasc_refresh_window(self.plan, state, self.layer_stride, self.req_stride, ids, q, k, v, g, beta, cu, t1 - t0, wb,
                                     window=window, layer_begin=self.lb, o=out, workspace=ws, **kw)
        else:
            dasc.dasc_refresh(self.plan, state, self.layer_stride, self.req_stride, ids, q, k, v, g, beta, cu, t1 - t0,
                              max(self.lens) if bound is None else bound, layer_begin=self.lb, o=out, workspace=ws, **kw)
        torch.cuda.synchronize()
        return out, ws, wb

    def small(self, **kw):
        """The same in calls of at most 148 units."""
        step = 148 // self.units(1)
        assert step and dasc.dasc_debug_refresh_form(step, self.units(1), step * max(self.lens), max(self.lens))[0] == ALONE
        state, outs = self.state0.clone(), []
        for lo in range(0, len(self.lens), step):
            out, ws, _ = self.call(state, lo, min(lo + step, len(self.lens)), **kw)
            assert dasc.dasc_refresh_status(ws) == binding.OK
            outs.append(out)
        return state, None if outs[0] is None else torch.cat(outs, 1)

    def form(self, bound, window=0):
        return dasc.dasc_debug_refresh_form(len(self.lens), self.units(1), int(self.cu[-1]), bound, window)[0]

    def check_oracle(self, state, mode, picks):
        q, k, v, g, beta = self.s
        merge = mode == dasc.REFRESH_SCRATCH_MERGE_LOCAL
        for r, l, h in picks:
            off = (self.lb + l) * self.layer_stride + h * 128 * 128
            s0, s1 = (x[int(self.slots[r]), off:off + 128 * 128].cpu().numpy().reshape(128, 128) for x in (self.state0, state))
            keep = self.oplan.mask[self.lb + l].reshape(self.H, -1)[h]
            keep = keep if self.kind == dasc.KDA else np.full(128, keep[0], np.uint8)
            ref, _ = oracle_one_unit(self.kind, self.H, self.H_k, s0, q, k, v, g, beta, torch.from_numpy(self.cu.astype(np.int32)), r, l, h,
                                     mode=oracle.MODE_SCRATCH_MERGE_LOCAL if merge else oracle.MODE_CONTINUE, keep_rows=keep, q_scale=1.0)
            assert rel_err(s1, ref) <= 1e-3, (r, l, h)


def same(a, b):
    return torch.equal(a.contiguous().view(torch.int32), b.contiguous().view(torch.int32))


SHORT = [20, 33, 0, 1, 64, 50, 8, 9, 31, 32] * 7
UNEVEN = [600, 9, 33, 0, 64, 400, 17, 65, 8, 31, 250, 96, 5] * 2


@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("lens,heads,bound,form", [(SHORT, 8, 64, WALK), (SHORT, 8, LOOSE, OWN), (UNEVEN, 8, 600, OWN),
                                                   ([40] * 10, 8, 40, OWN), ([30] * 239 + [61], 2, 61, WALK), ([30] * 240 + [61], 2, 61, OWN)])
@pytest.mark.parametrize("mode,o_dtype", [(dasc.REFRESH_CONTINUE, torch.bfloat16), (dasc.REFRESH_CONTINUE, torch.float32),
                                          (dasc.REFRESH_SCRATCH_MERGE_LOCAL, None)])
def test_large_calls_match_small_ones(kind, lens, heads, bound, form, mode, o_dtype):
    c = Large(91, kind, heads, lens)
    assert c.form(bound) == form
    state = c.state0.clone()
    out, ws, _ = c.call(state, 0, len(lens), bound=bound, mode=mode, o=o_dtype)
    assert dasc.dasc_refresh_status(ws) == binding.OK
    want_state, want_out = c.small(mode=mode, o=o_dtype)
    assert same(state, want_state)                        # padding and unused slots included
    assert out is None or torch.equal(out, want_out)
    c.check_oracle(state, mode, [(0, 0, 0), (1, 1, heads - 1), (len(lens) - 1, 0, 1)])


@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("lens,window,form", [(SHORT, 33, WALK), (SHORT, 4096, OWN), ([100] * 12, 512, OWN)])
@pytest.mark.parametrize("o_dtype", [None, torch.float32])
def test_large_windows_match_small_ones(kind, lens, window, form, o_dtype):
    c = Large(92, kind, 8, lens)
    assert c.form(window, window) == form
    state = c.state0.clone()
    out, ws, begin = c.call(state, 0, len(lens), window=window, o=o_dtype)
    assert dasc.dasc_refresh_status(ws) == binding.OK
    assert np.array_equal(begin.cpu().numpy(), np.maximum(c.cu[:-1], c.cu[1:] - window))
    want_state, want_out = c.small(window=window, o=o_dtype)
    assert same(state, want_state)
    assert out is None or same(out, want_out)             # (tokens before a window are not written in either)


@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("bound,form", [(64, WALK), (LOOSE, OWN)])
def test_units_outside_the_range_are_left_as_they_are(kind, bound, form):
    strong = [(1, 0, 3), (4, 1, 7), (5, 1, 0), (40, 0, 2), (64, 1, 1)]  # in the middle of walks and at their ends
    c = Large(93, kind, 8, SHORT, strong)
    plain = Large(93, kind, 8, SHORT)
    assert c.form(bound) == form
    state = c.state0.clone()
    _, ws, _ = c.call(state, 0, len(SHORT), bound=bound, algo=dasc.ALGO_CHUNKED)
    assert dasc.dasc_refresh_status(ws) == binding.ERR_DOMAIN and dasc.dasc_refresh_counters(ws) == (len(strong), 0)
    listed = set(ws[256:256 + 4 * len(strong)].view(torch.int32).tolist())
    assert listed == {(r * 2 + l) * 8 + h for r, l, h in strong}
    want = plain.state0.clone()                           # every other unit is what it is without those
    plain.call(want, 0, len(SHORT), bound=bound, algo=dasc.ALGO_CHUNKED)
    for r, l, h in strong:
        off = (c.lb + l) * c.layer_stride + h * 128 * 128
        want[int(c.slots[r]), off:off + 128 * 128] = c.state0[int(c.slots[r]), off:off + 128 * 128]
    assert same(state, want)


@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("o_dtype", [torch.bfloat16, None])
@pytest.mark.parametrize("lens,bound,form", [(SHORT, 64, WALK), (SHORT, LOOSE, OWN), (UNEVEN, 600, OWN), (UNEVEN[:9], 600, ALONE)])
def test_repeated_large_launches_give_identical_bits(kind, o_dtype, lens, bound, form):
    c = Large(94, kind, 8, lens)
    assert c.form(bound) == form
    first = None
    for _ in range(8):
        state = c.state0.clone()
        out, _, _ = c.call(state, 0, len(lens), bound=bound, algo=dasc.ALGO_CHUNKED, o=o_dtype)
        if first is None:
            first = state, out
        assert same(state, first[0]) and (out is None or torch.equal(out, first[1]))
