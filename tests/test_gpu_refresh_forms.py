"""The chunked kernel has two forms: up to 148 units a CTA has an SM to itself, with second buffers and more warps; above, two CTAs
share one.  Both sides of the line against the oracle, at lengths around the boundaries of chunks."""
import pytest
import torch

import oracle
import paper_2608_30386_b200 as dasc
from helpers import assert_refresh_close, make_refresh_case, run_refresh_gpu, run_refresh_oracle

pytestmark = pytest.mark.gpu

# one chunk to nine (the longest rings have eight places), tails of one token and of one less than a chunk, an empty request
LENS = [9, 31, 32, 33, 63, 64, 65, 97, 128, 129, 0, 161, 193, 225, 257, 288, 47]


@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("n_req", [17, 37, 38, 75])  # x 4 heads: 68, 148, 152 and 300 units, the last two in the form for two CTAs
def test_both_sides_of_the_lines(kind, n_req):
    lens = (LENS * 5)[:n_req]
    case = make_refresh_case(71, kind, 1, 4, 4 if kind == dasc.KDA else 2, 128, 128, lens, scope=dasc.SCOPE_LAYER, keep_ratio=0.4)
    ref_s, ref_o = run_refresh_oracle(case, q_scale=0.5)
    got_s, got_o = run_refresh_gpu(case, q_scale=0.5)
    assert_refresh_close(case, got_s, got_o, ref_s, ref_o, 1e-3)
    # the same outputs rounded to bf16, and the merge mode without outputs
    _, got_b = run_refresh_gpu(case, q_scale=0.5, o_dtype=torch.bfloat16)
    assert torch.equal(torch.from_numpy(got_o).to(torch.bfloat16).float(), torch.from_numpy(got_b))
    ref_s, _ = run_refresh_oracle(case, mode=oracle.MODE_SCRATCH_MERGE_LOCAL, want_o=False)
    got_s, _ = run_refresh_gpu(case, mode=dasc.REFRESH_SCRATCH_MERGE_LOCAL, want_o=False)
    assert_refresh_close(case, got_s, None, ref_s, None, 1e-3)


@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
def test_even_requests_just_above_an_sm_each(kind):
    # 152 units of the same length: the form for two CTAs
    case = make_refresh_case(72, kind, 1, 4, 4 if kind == dasc.KDA else 2, 128, 128, [95] * 38, scope=dasc.SCOPE_LAYER, keep_ratio=0.4)
    ref_s, ref_o = run_refresh_oracle(case)
    got_s, got_o = run_refresh_gpu(case)
    assert_refresh_close(case, got_s, got_o, ref_s, ref_o, 1e-3)
