"""What `enumerated` of a batch's codes promises, with and without the early
exit inside a pass."""
import numpy as np
import pytest

from paper_2603_29942_gb300 import _binding as B
from paper_2603_29942_gb300 import inputs


@pytest.mark.gpu
def test_enumerated_of_a_batch():
    """mid_pass_exit 0: the counts of the passes entered, in every run.  1:
    everything but `enumerated` and the choice among equal weights repeats
    and equals that; `enumerated` holds at least the passes before the last
    and at most all of them (how much of a pass had begun when the record
    that ends it fell is a matter of timing)."""
    codes = inputs.batch_codes()
    full = B.fpcode_min_distance_batch(codes, None, B.fpcode_opts_default(budget=10 ** 7, mid_pass_exit=0))
    counts = full.field("counts").sum(axis=1)
    assert (full.field("enumerated") == counts).all()
    cut = B.fpcode_opts_default(budget=10 ** 7)
    for _ in range(4):
        r = B.fpcode_min_distance_batch(codes, None, cut)
        for f in ("status", "d", "L", "U", "npasses", "counts"):
            assert np.array_equal(r.field(f), full.field(f)), f
        assert (r.field("enumerated") <= counts).all()
        for i, c in enumerate(codes[:64]):
            pr = B.fpcode_prepare(c.p, c.n, c.k, c.G, B.fpcode_opts_default(budget=10 ** 7, pair_leaves=0))
            before = sum(ps[5] for ps in B.fpcode_prepared_passes(pr)[:int(r.field("npasses")[i]) - 1])
            assert r.field("enumerated")[i] >= before


@pytest.mark.gpu
def test_kernel_time_of_a_launch_is_its_own():
    """Launches of one batch run side by side: a short one that waits for SMs
    that a long one holds does not count the wait as its kernel time."""
    long = inputs.single_code(21, 11, 60, 20)
    short = [inputs.single_code(22 + i, 3, 24, 10) for i in range(4)]
    o = B.fpcode_opts_default(budget=10 ** 10, mid_pass_exit=0)
    for _ in range(3):
        r = B.fpcode_min_distance_batch([long] + short, None, o)
        launches = {x.launch for x in r[1:]}
        assert len(launches) == 1 and r[0].launch not in launches
        assert 0 < r[1].t_kernel_ms < 0.25 * r[0].t_kernel_ms
        assert all(x.t_kernel_ms <= x.t_total_ms for x in r)
