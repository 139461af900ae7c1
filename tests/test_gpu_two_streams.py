"""A Store on one stream runs beside a refresh on another that leaves most of the GPU unused, also when the refresh's own
stream has more work queued: blocks of that later work that wait for the refresh must not hold the idle SMs meanwhile."""
import pytest
import torch

import paper_2608_30386_b200 as dasc
from helpers import make_refresh_case
from paper_2608_30386_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("io_dtype,tokens", [(torch.bfloat16, 16384), (torch.float32, 8192)])
def test_store_does_not_wait_for_a_small_refresh_on_another_stream(io_dtype, tokens):
    # a long serial chain on a few SMs: more than a millisecond
    case = make_refresh_case(61, dasc.KDA, 1, 2, 2, 128, 128, [tokens], io_dtype=io_dtype, scope=dasc.SCOPE_LAYER, keep_ratio=0.38)
    dev, s = case.state0.device, case.streams
    one = torch.zeros(1, dtype=torch.int32, device=dev)
    ws = torch.zeros(max(256, dasc.dasc_refresh_workspace_bytes(case.plan, 1, 1)), dtype=torch.uint8, device=dev)
    o = torch.empty_like(s.v)
    # a copy of about 0.1 ms on the whole GPU, much more than that on the few SMs the refresh runs on
    layers, heads, batch = 24, 32, 16
    dense = heads * 128 * 128
    rates = synth.decay_rates(synth.generator(62), layers, heads, 128, 1e-3, 1.0)
    plan = dasc.dasc_plan(dasc.KDA, layers, heads, heads, 128, 128, *synth.decay_params(rates), sel=dasc.SEL_TOP_RATIO,
                          scope=dasc.SCOPE_LAYER, keep_ratio=0.38)
    ids = torch.arange(batch, dtype=torch.int32, device=dev)
    states = torch.randn((layers, batch, dense), device=dev)
    pools = [torch.zeros((batch, int(plan.slot_floats)), device=dev) for _ in range(2)]
    loaded = torch.empty_like(states)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()

    def both():
        state = case.state0.clone()
        start, stored, done = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        torch.cuda.synchronize()
        start.record(a)
        dasc.dasc_refresh(case.plan, state, 2 * 128 * 128, 2 * 128 * 128, one, s.q, s.k, s.v, s.g, s.beta, case.cu.to(dev), tokens,
                          tokens, o=o, workspace=ws, stream=a)
        dasc.dasc_restore(plan, pools[0], ids, loaded, batch * dense, dense, ids, stream=a)
        dasc.dasc_pack(plan, states, batch * dense, dense, ids, pools[1], ids, stream=b)
        stored.record(b)
        done.record(a)
        torch.cuda.synchronize()
        return start.elapsed_time(stored), start.elapsed_time(done)

    both()
    share = min(x / y for x, y in (both() for _ in range(5)))
    assert share < 0.5, f"the store ended at {share:.2f} of the time of the refresh and what follows it"


@pytest.mark.parametrize("requests,heads", [(2, 32), (4, 32), (4, 37)])
def test_store_does_not_wait_for_a_long_refresh_of_up_to_all_sms(requests, heads):
    # a unit per SM of 64, 128 or 148: a Store has to get in beside it, not behind it
    dev, tokens, dense = "cuda", 4096, heads * 128 * 128
    gen, dgen = synth.generator(63), synth.generator(63, "cuda")
    rates = synth.decay_rates(gen, 1, heads, 128, 1e-3, 1.0)
    plan = dasc.dasc_plan(dasc.KDA, 1, heads, heads, 128, 128, *synth.decay_params(rates), sel=dasc.SEL_TOP_RATIO, scope=dasc.SCOPE_LAYER,
                          keep_ratio=0.38)
    total = requests * tokens
    s = synth.token_streams(dgen, synth.KDA, 1, total, heads, heads, 128, 128, rates, torch.bfloat16, dev)
    cu = torch.arange(requests + 1, dtype=torch.int32, device=dev) * tokens
    state, ids = synth.states(dgen, (1, requests, dense), dev), torch.arange(requests, dtype=torch.int32, device=dev)
    ws = torch.zeros(dasc.dasc_refresh_workspace_bytes(plan, requests, 1), dtype=torch.uint8, device=dev)
    o = torch.empty((1, total, heads, 128), dtype=torch.bfloat16, device=dev)
    layers, batch, s_dense = 24, 8, 32 * 128 * 128
    s_rates = synth.decay_rates(gen, layers, 32, 128, 1e-3, 1.0)
    s_plan = dasc.dasc_plan(dasc.KDA, layers, 32, 32, 128, 128, *synth.decay_params(s_rates), sel=dasc.SEL_TOP_RATIO,
                            scope=dasc.SCOPE_LAYER, keep_ratio=0.38)
    s_ids = torch.arange(batch, dtype=torch.int32, device=dev)
    states = torch.randn((layers, batch, s_dense), device=dev)
    pool = torch.zeros((batch, int(s_plan.slot_floats)), device=dev)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()

    def both():
        start, stored, done = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        torch.cuda.synchronize()
        start.record(a)
        dasc.dasc_refresh(plan, state, requests * dense, dense, ids, s.q, s.k, s.v, s.g, s.beta, cu, total, tokens, o=o, workspace=ws,
                          stream=a)
        dasc.dasc_pack(s_plan, states, batch * s_dense, s_dense, s_ids, pool, s_ids, stream=b)
        stored.record(b)
        done.record(a)
        torch.cuda.synchronize()
        return start.elapsed_time(stored) / start.elapsed_time(done)

    both()
    share = min(both() for _ in range(7))
    assert share < 0.7, f"the store ended at {share:.2f} of the time of the refresh"
