"""Split passes (the tensor-core kernel of one code): the walk on the CPU,
and results on the GPU against the leaf kernels and the oracle."""
import math

import numpy as np
import pytest

import oracle
from paper_2603_29942_gb300 import _binding as B
from paper_2603_29942_gb300 import inputs


@pytest.fixture(scope="module")
def lib():
    return B.lib()


def _prep(code, **over):
    return B.fpcode_test_prepare_split(code.p, code.n, code.k, code.G, B.fpcode_opts_default(**over))


# (p, n, k): one-row and pair keys (pair: the search is expected to be large)
WALKS = [(3, 16, 8, 0), (3, 70, 24, 1), (5, 24, 9, 0), (7, 20, 7, 0), (7, 38, 14, 1)]


@pytest.mark.parametrize("p,n,k,pair", WALKS)
def test_split_pass_visits_each_class_once(p, n, k, pair, lib):
    """The keys of a split pass are pairwise different, decode to codewords of
    the pass, and number C(k, g) (p-1)^(g-1): under the plan's own tasks for
    several grids, and with tails of two and three rows in blocks and runs
    that leave remainders."""
    pr = _prep(inputs.single_code(11, p, n, k), defer=0)
    assert (B.fpcode_test_pair_mode(pr) > 0) == bool(pair)
    checked = 0
    for i, (g, j, _lb, _la, _re, size, _np) in enumerate(B.fpcode_prepared_passes(pr)):
        if g < 2 or size > 80000 or j > 0:
            continue
        walks = [dict(ctas=152), dict(ctas=3)]
        walks += [dict(tail_rows=t, block=bl, unit=u, esplit=s) for t in (2, 3) if t <= g
                  for bl, u, s in ((96, 1, 0), (192, 4, 1), (7 * 96, 6, 0))]
        for w in walks:
            keys = B.fpcode_test_split_pass(pr, i, **w)
            assert keys is not None and len(keys) == size == math.comb(k, g) * (p - 1) ** (g - 1), (g, w)
            assert len(np.unique(keys)) == size, (g, w)
        for key in keys[:: max(1, size // 500)]:
            got = B.fpcode_test_key_coefficients(pr, int(key))
            assert got is not None and got[0] == g and got[1] == j and sum(1 for c in got[2] if c) == g
        checked += 1
    assert checked >= 2


@pytest.mark.parametrize("p,n,k", [(3, 80, 40), (3, 74, 50), (7, 40, 20), (5, 51, 24), (3, 30, 15)])
@pytest.mark.parametrize("ctas", [152, 1])
def test_split_plan_covers_early_passes(p, n, k, ctas, lib):
    """At the sizes of the workloads the plan's tasks visit every codeword of
    the early passes once (both the exact and the tensor-core form)."""
    pr = _prep(inputs.single_code(2, p, n, k))
    for i, (g, j, _lb, _la, _re, size, _np) in enumerate(B.fpcode_prepared_passes(pr)):
        if g < 2 or j > 0 or size > 2500000:
            continue
        keys = B.fpcode_test_split_pass(pr, i, ctas=ctas)
        assert len(keys) == size and len(np.unique(keys)) == size


@pytest.mark.parametrize("p", [3, 5, 7])
def test_split_plan_runs_fit_the_kernels_copy(p, lib):
    """No pass of any shape has more than 192 runs of tasks (the kernel copies
    those of one pass when a code has too many in all)."""
    most, seen = 0, 0
    for k in (5, 12, 20, 28, 36, 40, 43, 50, 57, 64):
        for red in (6, 20, 33, 41, 70, 120):
            pr = _prep(inputs.single_code(1, p, k + red, k))
            if pr is None:
                continue
            for ctas in (152, 7):
                for i, x in enumerate(B.fpcode_prepared_passes(pr)):
                    if x[0] >= 2 and x[1] == 0:
                        most = max(most, B.fpcode_test_split_runs(pr, i, ctas))
                        seen += 1
    assert seen > 100 and 1 <= most <= 192


def test_which_codes_are_split(lib):
    """p = 3, 5, 7 with the leaf form left to the library; not with a leaf
    form asked for, other primes, or rows that hold too many class values."""
    def split(p, n, k, **kw):
        return _prep(inputs.single_code(9, p, n, k), **kw) is not None
    assert split(3, 80, 40) and split(7, 40, 20) and split(5, 51, 24)
    assert not split(3, 80, 40, pair_leaves=1) and not split(7, 40, 20, pair_leaves=0)
    assert not split(11, 30, 10) and not split(31, 40, 8)
    assert not split(7, 70, 20)   # 150 class values
    assert not split(3, 10, 2) and not split(3, 12, 10)


def _same(a, b, what=("status", "d", "L", "U", "m", "npasses", "counts", "kj", "best_key")):
    for f in what:
        assert getattr(a, f) == getattr(b, f), f


# K = 32 .. 128, word edges, padded and full last tiles, rank-deficient sets, k = 64
GPU_CODES = [(3, 22, 8, 0), (3, 41, 13, 0), (3, 47, 15, 0), (3, 64, 32, 2 * 10 ** 8), (3, 80, 40, 0), (3, 95, 60, 10 ** 8),
             (3, 76, 12, 0), (3, 110, 14, 0), (3, 136, 12, 10 ** 7), (3, 100, 64, 10 ** 8), (5, 20, 11, 0), (5, 40, 20, 0),
             (5, 66, 24, 10 ** 8), (7, 14, 9, 0), (7, 40, 20, 0), (7, 52, 19, 3 * 10 ** 8), (7, 62, 20, 10 ** 8),
             (7, 53, 12, 10 ** 8), (3, 12, 8, 0), (7, 8, 4, 0)]


@pytest.mark.gpu
@pytest.mark.parametrize("p,n,k,budget", GPU_CODES)
def test_split_search_equals_leaf_kernels(p, n, k, budget):
    """Same interval, counts, best key and witness as the popcount kernel of
    the same leaf form, with every pass enumerated in full."""
    code = inputs.single_code(1000 + n, p, n, k)
    o = B.fpcode_opts_default(budget=budget, mid_pass_exit=0)
    pr = B.fpcode_test_prepare_split(p, n, k, code.G, o)
    pair = 1 if B.fpcode_test_pair_mode(pr) > 0 else 0
    a = B.fpcode_min_distance_ex(pr, None, o)
    o1 = B.fpcode_opts_default(budget=budget, mid_pass_exit=0, pair_leaves=pair)
    b = B.fpcode_min_distance_ex(B.fpcode_prepare(p, n, k, code.G, o1), None, o1)
    _same(a, b)
    assert a.enumerated == b.enumerated == sum(a.counts)
    assert np.array_equal(a.witness, b.witness)
    c = B.fpcode_min_distance_ex(pr, None, B.fpcode_opts_default(budget=budget))  # the same handle again, with early exits
    _same(c, b, ("status", "d", "L", "U", "m", "npasses", "counts", "kj"))


@pytest.mark.parametrize("p,n,k,split", [(3, 80, 40, True), (3, 85, 25, True), (5, 51, 24, True), (7, 50, 25, True),
                                         (3, 80, 22, False), (3, 65, 24, False), (5, 33, 19, False), (7, 40, 20, False)])
def test_split_only_where_passes_are_large(p, n, k, split, lib):
    """Many passes with little work each stay on the leaf kernels."""
    code = inputs.single_code(60 + n, p, n, k)
    pr = B.fpcode_prepare(p, n, k, code.G, B.fpcode_opts_default())
    last = max(i for i, ps in enumerate(B.fpcode_prepared_schedule(pr)) if ps["g"] <= 3)
    assert (B.fpcode_test_split_pass(pr, last, cap=1 << 16) is not None) is split


# the widest rows of p = 3 (n - k = 128: 124 positions compared), and of p = 5 and 7 (n - k = 42)
ORACLE_CODES = [(3, 140, 12), (3, 139, 11), (3, 138, 12), (3, 137, 13), (3, 60, 20), (5, 53, 11), (5, 30, 12), (7, 53, 11),
                (7, 33, 9)]


@pytest.mark.gpu
@pytest.mark.parametrize("p,n,k", ORACLE_CODES)
def test_split_search_equals_oracle(p, n, k):
    """Interval, schedule and counts as the oracle's, every pass in full, and
    a witness of the best weight."""
    code = inputs.single_code(1700 + n, p, n, k)
    o = B.fpcode_opts_default(budget=3 * 10 ** 6, mid_pass_exit=0)
    pr = B.fpcode_test_prepare_split(p, n, k, code.G, o)
    a = B.fpcode_min_distance_ex(pr, None, o)
    b = oracle.bz(code, threads=4, budget=3 * 10 ** 6)
    assert {oracle.OK: B.OK, oracle.EBUDGET: B.EBUDGET}[b.status] == a.status
    assert (a.L, a.U) == (b.L, b.U) and list(a.counts) == list(b.counts)
    assert a.enumerated == sum(a.counts)
    assert np.count_nonzero(np.array(a.witness)) == a.U


@pytest.mark.parametrize("p,most", [(3, 128), (5, 42), (7, 42)])
def test_widest_split_rows(p, most, lib):
    """Redundant symbols up to which the class values fit a row."""
    assert _prep(inputs.single_code(5, p, 20 + most, 20)) is not None
    if most < 128:
        assert _prep(inputs.single_code(5, p, 21 + most, 20)) is None
