"""Where units are few the fp32 refresh replays four tokens at a time: every tail of a block and of a group of 16,
all dimensions and widths of the column parts, strong decay included, against the fp64 oracle at the fp32 tolerance."""
import pytest
import torch

import oracle
import paper_2608_30386_b200 as dasc
from helpers import assert_refresh_close, make_refresh_case, run_refresh_gpu, run_refresh_oracle

pytestmark = pytest.mark.gpu


# (dimension, value heads), four requests: every width, from the narrowest parts (8 columns, 16 at d = 32) up to whole units
@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("dim,heads", [(32, 2), (32, 20), (64, 2), (64, 8), (64, 18), (64, 20), (128, 2), (128, 4), (128, 8), (128, 18)])
@pytest.mark.parametrize("lens", [[1, 2, 3, 4], [5, 15, 16, 17], [18, 33, 64, 0], [47, 65, 80, 31]])
def test_tails_of_blocks_and_groups(kind, dim, heads, lens):
    case = make_refresh_case(81, kind, 1, heads, heads // 2, dim, dim, lens, io_dtype=torch.float32, scope=dasc.SCOPE_LAYER, keep_ratio=0.5)
    case.streams.g[:, 1::7] *= 40.0    # decays down to nothing between ordinary ones
    case.streams.g[:, 3::11] = -200.0
    ref_s, ref_o = run_refresh_oracle(case, q_scale=0.5)
    got_s, got_o = run_refresh_gpu(case, algo=dasc.ALGO_SEQUENTIAL, q_scale=0.5)
    assert_refresh_close(case, got_s, got_o, ref_s, ref_o, 1e-5)
    ref_s, _ = run_refresh_oracle(case, mode=oracle.MODE_SCRATCH_MERGE_LOCAL, want_o=False)
    got_s, _ = run_refresh_gpu(case, mode=dasc.REFRESH_SCRATCH_MERGE_LOCAL, algo=dasc.ALGO_SEQUENTIAL, want_o=False)
    assert_refresh_close(case, got_s, None, ref_s, None, 1e-5)


@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("dim", [32, 64, 128])
def test_bf16_streams_and_outputs(kind, dim):
    # bf16 streams are exact in fp32, so the fp32 tolerance holds for the state; bf16 outputs are the fp32 ones rounded
    case = make_refresh_case(82, kind, 1, 2, 1, dim, dim, [37, 6], scope=dasc.SCOPE_LAYER, keep_ratio=0.5)
    ref_s, ref_o = run_refresh_oracle(case)
    got_s, got_o = run_refresh_gpu(case, algo=dasc.ALGO_SEQUENTIAL)
    assert_refresh_close(case, got_s, got_o, ref_s, ref_o, 1e-5)
    _, got_b = run_refresh_gpu(case, algo=dasc.ALGO_SEQUENTIAL, o_dtype=torch.bfloat16)
    assert torch.equal(torch.from_numpy(got_o).to(torch.bfloat16).float(), torch.from_numpy(got_b))


# Calls of a few tokens: blocks of a group that have none are left out in the wider parts, so nothing that lies in their place may be
# read.  Every length up to a group and one over, behind a long request (whose blocks were in the same buffers) and alone
@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("dim,heads", [(32, 2), (32, 37), (32, 74), (64, 2), (64, 8), (64, 18), (64, 36), (128, 2), (128, 4), (128, 8), (128, 18)])
@pytest.mark.parametrize("lens", [[1, 4], [5, 8], [9, 12], [13, 16], [16 + 1, 16 + 4], [32 + 5, 32 + 9], [2, 26], [1, 1]])
def test_calls_of_a_few_tokens(kind, dim, heads, lens):
    case = make_refresh_case(83, kind, 1, heads, heads // 2 if heads % 2 == 0 else heads, dim, dim, lens, io_dtype=torch.float32,
                             scope=dasc.SCOPE_LAYER, keep_ratio=0.5)
    ref_s, ref_o = run_refresh_oracle(case)
    for _ in range(2):
        got_s, got_o = run_refresh_gpu(case, algo=dasc.ALGO_SEQUENTIAL)
        assert_refresh_close(case, got_s, got_o, ref_s, ref_o, 1e-5)
