"""Small dependent calls on one stream with nothing between them: each kernel is on the GPU before the one in front of it has
finished, and reads what that one wrote (slots, states, scales)."""
import pytest
import torch

import paper_2608_30386_b200 as dasc
from helpers import make_refresh_case
from paper_2608_30386_b200 import synth

pytestmark = pytest.mark.gpu

LAYERS, HEADS, REQUESTS, SLOTS = 3, 2, 4, 2
DENSE = HEADS * 128 * 128


def _chain(plan, int8, states, wait):
    """Three states go round through two slots, so a slot and a state hold another one's values each time they are reused; the
    last two calls of a turn read what the call right before them wrote."""
    if int8:
        pool = torch.zeros((SLOTS, dasc.dasc_int8_slot_bytes(plan)), dtype=torch.uint8, device="cuda")
        pack, restore = dasc.dasc_pack_int8, dasc.dasc_restore_int8
    else:
        pool = torch.zeros((SLOTS, int(plan.slot_floats)), device="cuda")
        pack, restore = dasc.dasc_pack, dasc.dasc_restore
    ids = [torch.tensor([i], dtype=torch.int32, device="cuda") for i in range(REQUESTS)]

    def store(req, slot):
        pack(plan, states, REQUESTS * DENSE, DENSE, ids[req], pool, ids[slot])
        if wait:
            torch.cuda.synchronize()

    def load(slot, req):
        restore(plan, pool, ids[slot], states, REQUESTS * DENSE, DENSE, ids[req])
        if wait:
            torch.cuda.synchronize()

    torch.cuda.synchronize()
    store(0, 0)
    for i in range(48):
        req, held, free = (i + 1) % 3, i % 2, (i + 1) % 2
        store(req, free)
        load(held, req)
        store(req, held)
        load(held, 3)
    torch.cuda.synchronize()
    return states, pool


@pytest.mark.parametrize("int8", [False, True])
def test_a_chain_of_small_calls_is_the_calls_one_by_one(int8):
    rates = synth.decay_rates(synth.generator(71), LAYERS, HEADS, 128, 1e-3, 1.0)
    plan = dasc.dasc_plan(dasc.KDA, LAYERS, HEADS, HEADS, 128, 128, *synth.decay_params(rates), sel=dasc.SEL_TOP_RATIO,
                          scope=dasc.SCOPE_LAYER, keep_ratio=0.38)
    for seed in range(20):
        states = synth.states(synth.generator(seed, "cuda"), (LAYERS, REQUESTS, DENSE), "cuda")
        want, want_pool = _chain(plan, int8, states.clone(), True)
        got, got_pool = _chain(plan, int8, states.clone(), False)
        assert torch.equal(got.view(torch.int32), want.view(torch.int32))
        assert torch.equal(got_pool.view(torch.uint8), want_pool.view(torch.uint8))


def test_the_chain_and_a_refresh_in_a_graph():
    """The same calls captured once and replayed: the order on the stream is kept by the graph too."""
    case = make_refresh_case(72, dasc.KDA, 1, 2, 2, 128, 128, [70, 5, 33], scope=dasc.SCOPE_LAYER, keep_ratio=0.38)
    dev, s, plan, dense, total = case.state0.device, case.streams, case.plan, 2 * 128 * 128, 108
    cu, ids = case.cu.to(dev), torch.arange(3, dtype=torch.int32, device=dev)
    ws = torch.zeros(dasc.dasc_refresh_workspace_bytes(plan, 3, 1), dtype=torch.uint8, device=dev)
    state, o = torch.empty_like(case.state0), torch.empty((1, total, 2, 128), device=dev)
    pool, begin = torch.zeros((3, int(plan.slot_floats)), device=dev), torch.empty(3, dtype=torch.int32, device=dev)

    def calls():
        state.copy_(case.state0)
        for _ in range(2):
            dasc.dasc_pack(plan, state, dense, dense, ids, pool, ids)
            dasc.dasc_restore(plan, pool, ids, state, dense, dense, ids)
            dasc.dasc_refresh(plan, state, dense, dense, ids, s.q, s.k, s.v, s.g, s.beta, cu, total, 70, o=o, workspace=ws)
            dasc.dasc_refresh_window(plan, state, dense, dense, ids, None, s.k, s.v, s.g, s.beta, cu, total, begin, window=40,
                                     workspace=ws)

    calls()
    torch.cuda.synchronize()
    want = [t.clone() for t in (state, o, pool, begin)]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    for _ in range(3):
        for t in (state, o, pool, begin):
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert dasc.dasc_refresh_status(ws) == 0
        for got, ref in zip((state, o, pool, begin), want):
            assert torch.equal(got.view(torch.int32), ref.view(torch.int32))
