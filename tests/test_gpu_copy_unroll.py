"""Store and Load pick the loads in flight per thread from the size of the grid: each choice, at sizes where the last block of
a layer is partial, against plain indexing of the same bits."""
import pytest
import torch

import paper_2608_30386_b200 as dasc
from paper_2608_30386_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,requests", [(1, 1), (8, 1), (8, 2), (9, 1), (13, 2), (32, 2)])
@pytest.mark.parametrize("layers,d_v", [(24, 128), (5, 36)])
def test_every_unroll_moves_the_same_bits(heads, requests, layers, d_v):
    gen = synth.generator(heads * 7 + requests)
    rates = synth.decay_rates(gen, layers, heads, 128, 1e-3, 1.0)
    plan = dasc.dasc_plan(dasc.KDA, layers, heads, heads, 128, d_v, *synth.decay_params(rates), sel=dasc.SEL_TOP_RATIO,
                          scope=dasc.SCOPE_MODEL, keep_ratio=0.37)
    dense = heads * 128 * d_v
    state = torch.randn((layers, requests, dense), device="cuda")
    ids = torch.arange(requests, dtype=torch.int32, device="cuda")
    slots = ids.flip(0).contiguous()
    pool = torch.zeros((requests, int(plan.slot_floats)), device="cuda")
    dasc.dasc_pack(plan, state, requests * dense, dense, ids, pool, slots)
    keep = torch.from_numpy(plan.mask()).cuda().bool()                       # [layers][rows]
    rows = state.view(layers, requests, heads * 128, d_v)
    for r in range(requests):
        want = torch.cat([rows[l, r][keep[l]] for l in range(layers)]).reshape(-1)
        assert torch.equal(pool[requests - 1 - r].view(torch.int32), want.view(torch.int32))
    out = torch.full_like(state, float("nan"))
    dasc.dasc_restore(plan, pool, slots, out, requests * dense, dense, ids)
    want = torch.where(keep[:, None, :, None], rows, torch.zeros((), device="cuda"))
    assert torch.equal(out.view(-1).view(torch.int32), want.reshape(-1).view(torch.int32))
