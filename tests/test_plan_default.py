"""Task plans of one code with the default min_steps (0): passes that a few
prefixes a lane spread over the grid."""
import numpy as np
import pytest

from paper_2603_29942_gb300 import _binding as B
from paper_2603_29942_gb300 import inputs


@pytest.mark.parametrize("p,n,k", [(3, 43, 23), (3, 61, 20), (5, 40, 14), (7, 40, 20), (31, 32, 7), (13, 40, 9)])
@pytest.mark.parametrize("ctas", [1, 7, 152, 608])
def test_default_plan_tiles_each_pass(p, n, k, ctas):
    """Every prefix of a pass in one lane of one task, as under the explicit
    plans; passes of up to four prefixes a lane take one task per CTA at
    most and no more than four prefixes, the others the plan of eight."""
    code = inputs.single_code(60 + n, p, n, k)
    pr = B.fpcode_prepare(p, n, k, code.G, B.fpcode_opts_default(pair_leaves=0))
    for i, (g, _j, _Lb, _La, _re, _size, nprefix) in enumerate(B.fpcode_prepared_passes(pr)[:14]):
        if g < 2 or nprefix > 1 << 21:
            continue
        tasks = B.fpcode_test_task_ranges(pr, i, ctas, 0, 0)
        if 256 * ctas < nprefix <= 4 * 256 * ctas:
            steps = -(-nprefix // (256 * ctas))
            assert len(tasks) <= ctas and all(hi - lo == 256 * steps for lo, hi in tasks[:-1])
        else:
            assert tasks == B.fpcode_test_task_ranges(pr, i, ctas, 0, 8)
        lo, hi = (x.astype(np.int64) for x in B.fpcode_test_lane_ranges(pr, i, ctas, 0, 0))
        lo, hi = lo[hi > lo], hi[hi > lo]
        order = np.argsort(lo, kind="stable")
        assert lo[order][0] == 0 and hi[order][-1] == nprefix and (lo[order][1:] == hi[order][:-1]).all()
