"""The merge mode without outputs has a variant of the chunked kernel that leaves out what a zero start state makes superfluous in a
unit's first chunk.  Its states against the oracle and against the general variant, which the same call with outputs takes."""
import numpy as np
import pytest

import oracle
import paper_2608_30386_b200 as dasc
from helpers import assert_refresh_close, make_refresh_case, run_refresh_gpu, run_refresh_oracle

pytestmark = pytest.mark.gpu

OWN, WALK, ALONE = 0, 1, 2
LENS = [9, 31, 32, 33, 64, 65, 0, 97, 1, 128]


# alone on an SM; a block per unit, two to an SM; several units to a block, first chunks in the middle of its work
@pytest.mark.parametrize("kind", [dasc.KDA, dasc.GDN])
@pytest.mark.parametrize("heads,lens,form", [(4, LENS, ALONE), (8, LENS * 2 + [129], OWN), (8, LENS * 7, WALK)])
def test_units_that_start_from_zero(kind, heads, lens, form):
    assert dasc.dasc_debug_refresh_form(len(lens), heads, sum(lens), max(lens))[0] == form
    case = make_refresh_case(81, kind, 1, heads, heads if kind == dasc.KDA else heads // 2, 128, 128, lens, scope=dasc.SCOPE_LAYER,
                             keep_ratio=0.4)
    merge = dict(mode=dasc.REFRESH_SCRATCH_MERGE_LOCAL)
    got, _ = run_refresh_gpu(case, want_o=False, **merge)
    ref, _ = run_refresh_oracle(case, mode=oracle.MODE_SCRATCH_MERGE_LOCAL, want_o=False)
    assert_refresh_close(case, got, None, ref, None, 1e-3)
    assert np.array_equal(got, run_refresh_gpu(case, **merge)[0])  # (zeros of either sign)
