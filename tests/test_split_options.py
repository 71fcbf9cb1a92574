"""Options that only the leaf kernels' plans know keep a search on them."""
import pytest

from paper_2603_29942_gb300 import _binding as B
from paper_2603_29942_gb300 import inputs


@pytest.mark.parametrize("p,n,k", [(3, 80, 40), (5, 51, 24), (7, 50, 25)])
@pytest.mark.parametrize("option", [{}, {"prefixes_per_lane": 4}, {"min_steps": 16}, {"task_work": 96},
                                    {"task_share": 2}, {"ctas_per_sm": 2}, {"budget": 10 ** 10}])
def test_task_sizes_keep_the_leaf_kernels(p, n, k, option):
    """A task size that a caller sets is the plan's, not dropped without a word."""
    code = inputs.single_code(60 + n, p, n, k)
    pr = B.fpcode_prepare(p, n, k, code.G, B.fpcode_opts_default(**option))
    last = max(i for i, ps in enumerate(B.fpcode_prepared_schedule(pr)) if ps["g"] <= 3)
    split = B.fpcode_test_split_pass(pr, last, cap=1 << 16) is not None
    assert split is not (set(option) <= {"prefixes_per_lane", "min_steps", "task_work", "task_share"} and bool(option))
