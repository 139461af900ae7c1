"""The token-by-token kernel has one variant per range of unit counts (columns split over CTAs, whole units in blocks of four, token by token): each
at the edges of its token groups and on both sides of the counts where the choice changes, against the fp64 oracle."""
import pytest
import torch

import oracle
import paper_2608_30386_b200 as dasc
from helpers import assert_refresh_close, make_refresh_case, run_refresh_gpu, run_refresh_oracle

pytestmark = pytest.mark.gpu

LENS = [1, 15, 16, 17, 32, 33, 0, 49]  # tokens come in groups of 16


@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("dim,heads", [(32, 4), (32, 20), (64, 4), (64, 6), (128, 2), (128, 4), (128, 10)])
def test_every_variant_of_the_sequential_kernel(kind, dim, heads):
    case = make_refresh_case(31, kind, 1, heads, heads // 2, dim, dim, LENS, io_dtype=torch.float32,
                             scope=dasc.SCOPE_LAYER, keep_ratio=0.5)
    ref_s, ref_o = run_refresh_oracle(case)
    got_s, got_o = run_refresh_gpu(case, algo=dasc.ALGO_SEQUENTIAL)
    assert_refresh_close(case, got_s, got_o, ref_s, ref_o, 1e-5)
    ref_s, _ = run_refresh_oracle(case, mode=oracle.MODE_SCRATCH_MERGE_LOCAL, want_o=False)
    got_s, _ = run_refresh_gpu(case, mode=dasc.REFRESH_SCRATCH_MERGE_LOCAL, algo=dasc.ALGO_SEQUENTIAL, want_o=False)
    assert_refresh_close(case, got_s, None, ref_s, None, 1e-5)
