"""The chunked kernel takes the requests longest first (up to 240 of them): results, windows and the indices of the units
it hands over are those of the caller's numbering, on both sides of that limit."""
import numpy as np
import pytest
import torch

import oracle
import paper_2608_30386_b200 as dasc
from helpers import assert_refresh_close, make_refresh_case, run_refresh_gpu, run_refresh_oracle, stream_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_req", [2, 3, 239, 240, 241])
def test_any_number_of_ragged_requests(n_req):
    lens = np.random.default_rng(n_req).integers(9, 70, n_req).tolist()
    case = make_refresh_case(51, dasc.KDA, 1, 1, 1, 128, 128, lens, scope=dasc.SCOPE_LAYER, keep_ratio=0.38)
    ref_s, ref_o = run_refresh_oracle(case)
    got_s, got_o = run_refresh_gpu(case)
    assert_refresh_close(case, got_s, got_o, ref_s, ref_o, 1e-3)


def test_unit_indices_are_the_callers():
    case = make_refresh_case(52, dasc.KDA, 2, 2, 2, 128, 128, [40, 10, 96], scope=dasc.SCOPE_LAYER, keep_ratio=0.38)
    case.streams.g[1, 50:146, 1, 5] = -7.0     # request 2, layer 1, head 1 leaves the kernel's log-decay range
    dev, T = case.state0.device, 146
    s, state = case.streams, case.state0.clone()
    ws = torch.zeros(dasc.dasc_refresh_workspace_bytes(case.plan, 3, 2, dasc.ALGO_CHUNKED), dtype=torch.uint8, device=dev)
    dasc.dasc_refresh(case.plan, state, 2 * 128 * 128, 4 * 128 * 128, torch.arange(3, dtype=torch.int32, device=dev), s.q, s.k, s.v,
                      s.g, s.beta, case.cu.to(dev), T, 96, algo=dasc.ALGO_CHUNKED, workspace=ws)
    torch.cuda.synchronize()
    assert dasc.dasc_refresh_counters(ws) == (1, 0)
    assert int(ws[256:260].view(torch.int32).item()) == (2 * 2 + 1) * 2 + 1
    got_s, got_o = run_refresh_gpu(case)       # AUTO replays it exactly
    ref_s, ref_o = run_refresh_oracle(case)
    assert_refresh_close(case, got_s, got_o, ref_s, ref_o, 1e-3)


@pytest.mark.parametrize("n_req", [5, 300])
def test_windows(n_req):
    lens = np.random.default_rng(n_req).integers(1, 60, n_req).tolist()
    case = make_refresh_case(53, dasc.GDN, 1, 2, 1, 128, 128, lens, scope=dasc.SCOPE_LAYER, keep_ratio=0.5)
    dev, cu = case.state0.device, case.cu.to("cuda")
    s, state = case.streams, case.state0.clone()
    wb = torch.full((n_req,), -1, dtype=torch.int32, device=dev)
    ws = torch.zeros(dasc.dasc_refresh_workspace_bytes(case.plan, n_req, 1), dtype=torch.uint8, device=dev)
    dasc.dasc_refresh_window(case.plan, state, 2 * 128 * 128, 2 * 128 * 128, torch.arange(n_req, dtype=torch.int32, device=dev), None,
                             s.k, s.v, s.g, s.beta, cu, int(case.cu[-1]), wb, window=33, workspace=ws)
    torch.cuda.synchronize()
    want = torch.maximum(case.cu[:-1], case.cu[1:] - 33)
    assert torch.equal(wb.cpu(), want)
    got = state.cpu().numpy()
    for r in range(n_req):                      # the oracle on the token slices the windows name
        a, b = int(want[r]), int(case.cu[r + 1])
        st = case.state0[r:r + 1].cpu().numpy().copy()
        sl = [x[:, a:b].contiguous() for x in (s.k, s.v, s.g, s.beta)]
        _, s64 = oracle.refresh(dasc.GDN, 1, 2, 1, 128, 128, st, 2 * 128 * 128, 2 * 128 * 128, np.zeros(1, np.int32),
                                stream_np(sl[0]), stream_np(sl[0]), stream_np(sl[1]), stream_np(sl[2]), stream_np(sl[3]), np.array([0, b - a], np.int32),
                                want_o=False, mode=oracle.MODE_SCRATCH_MERGE_LOCAL, mask=case.oplan.mask, want_state64=True)
        for h in range(2):
            ref = s64[0, 0, h]
            assert np.abs(got[r, 0, h] - ref).max() <= 1e-3 * np.abs(ref).max()
