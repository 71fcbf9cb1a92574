"""Several uploaded codes of one kernel at a time, with different amounts of
shared memory: each handle stays searchable whatever is prepared after it."""
import pytest

from paper_2603_29942_gb300 import _binding as B
from paper_2603_29942_gb300 import inputs

# two codes of one kernel, the first with more shared memory: one-row leaves
# with class labels past 48 KiB, and the tensor-core kernel
PAIRS = [((17, 114, 64), (17, 110, 60)), ((13, 114, 64), (13, 120, 64 - 1)),
         ((3, 80, 40), (3, 85, 25)), ((7, 50, 25), (7, 54, 24))]


@pytest.mark.gpu
@pytest.mark.parametrize("big,small", PAIRS)
@pytest.mark.parametrize("first", [0, 1])
def test_handles_of_one_kernel(big, small, first):
    o = B.fpcode_opts_default(budget=10 ** 9 if big[0] < 11 else 10 ** 7, mid_pass_exit=0)
    shapes = (big, small) if first == 0 else (small, big)
    codes = [inputs.single_code(700 + n, p, n, k) for p, n, k in shapes]
    preps = [B.fpcode_prepare(c.p, c.n, c.k, c.G, o) for c in codes]
    want = []
    for pr in preps:
        B.fpcode_prepared_upload(pr, None)
        want.append(B.fpcode_min_distance_ex(pr, None, o))
    # a whole call on a third code of the same kernel in between: one row more (certified at once: d = 1)
    p, n, k = shapes[1]
    third = inputs.single_code(900, p, n, k - 1).G.copy()
    third[0, k - 1:] = 0
    for _ in range(2):
        for pr, w in zip(preps, want):
            r = B.fpcode_min_distance_ex(pr, None, o)
            assert (r.status, r.L, r.U, r.counts, r.best_key, r.enumerated) == \
                (w.status, w.L, w.U, w.counts, w.best_key, w.enumerated)
        assert B.fpcode_min_distance(p, n, k - 1, third)[0] == 1
