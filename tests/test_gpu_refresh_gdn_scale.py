"""GDN: the chunked kernel keeps the scale of the state in tensor memory over several chunks while the accumulated log-decay
allows it and moves it otherwise.  Decay rates on both sides of that choice, lengths from one chunk to many."""
import pytest

import oracle
import paper_2608_30386_b200 as dasc
from helpers import assert_refresh_close, make_refresh_case, run_refresh_gpu, run_refresh_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rate_lo,rate_hi", [(1e-4, 1e-3), (0.05, 0.2), (0.5, 1.2), (1.5, 2.5)])
def test_kept_and_moved_scales(rate_lo, rate_hi):
    case = make_refresh_case(61, dasc.GDN, 1, 4, 2, 128, 128, [31, 32, 33, 65, 700], scope=dasc.SCOPE_LAYER, keep_ratio=0.5,
                             rate_lo=rate_lo, rate_hi=rate_hi)
    ref_s, ref_o = run_refresh_oracle(case)
    got_s, got_o = run_refresh_gpu(case, algo=dasc.ALGO_CHUNKED)
    assert_refresh_close(case, got_s, got_o, ref_s, ref_o, 1e-3)
    ref_s, _ = run_refresh_oracle(case, mode=oracle.MODE_SCRATCH_MERGE_LOCAL, want_o=False)
    got_s, _ = run_refresh_gpu(case, mode=dasc.REFRESH_SCRATCH_MERGE_LOCAL, algo=dasc.ALGO_CHUNKED, want_o=False)
    assert_refresh_close(case, got_s, None, ref_s, None, 1e-3)
