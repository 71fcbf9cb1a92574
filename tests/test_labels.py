"""Class labels of the one-row leaf filter (p = 5 and the primes above 7)."""
import numpy as np
import pytest

import oracle
from paper_2603_29942_gb300 import _binding as B
from paper_2603_29942_gb300 import inputs

PRIMES = [p for p in range(5, 252) if p != 7 and all(p % q for q in range(2, p))]


def test_label_tells_classes_apart():
    """v and p - v share a label of r - 1 bits, other symbols do not, and only
    0 has label 0: every prime, every symbol."""
    for p in PRIMES:
        lab = [x for v in range(0, p, 32) for x in B.fpcode_test_class_label(p, range(v, min(v + 32, p)))]
        assert len(lab) == p and max(lab) < 1 << (p.bit_length() - 1)
        cls = {}
        for v, x in enumerate(lab):
            cls.setdefault(x, set()).add(v)
        assert sorted(map(sorted, cls.values())) == sorted(sorted({v, (p - v) % p}) for v in range(p // 2 + 1))
        assert cls[0] == {0}


@pytest.mark.parametrize("p", [31, 127])
def test_log_of_classes(p):
    """3^(log s) is s or -s, and log s - log t is the class e with
    s = +-3^e t (0 also as all ones): every pair of nonzero symbols."""
    h = (p - 1) // 2
    pairs = [(s, t) for s in range(1, p) for t in range(1, p)]
    for i in range(0, len(pairs), 32):
        ss, ts = zip(*pairs[i:i + 32])
        logs, diffs = B.fpcode_test_class_log(p, ss, ts)
        for s, t, a, d in zip(ss, ts, logs, diffs):
            assert a < h and pow(3, a, p) in (s, p - s)
            assert pow(3, d % h, p) * t % p in (s, p - s) and d <= h


# n - k at one to four words and off their edges; (251, 20, 9): labels do not fit behind the
# multiples; (61, 130, 4 and 6): a shape without labels
CODES = [(5, 20, 5), (5, 45, 12), (5, 74, 10), (5, 104, 8), (5, 140, 12), (11, 30, 6), (13, 60, 6), (11, 100, 5),
         (13, 133, 5), (17, 40, 5), (31, 24, 5), (31, 70, 6), (31, 42, 10), (31, 36, 4), (31, 100, 4), (31, 132, 4), (61, 40, 4), (61, 130, 4),
         (127, 30, 3), (127, 70, 3), (127, 35, 3), (127, 66, 2), (127, 30, 18), (251, 20, 3), (251, 20, 9), (251, 60, 3), (61, 130, 6)]


@pytest.mark.gpu
@pytest.mark.parametrize("p,n,k", CODES)
def test_label_search_equals_oracle(p, n, k):
    """Interval, schedule, counts and distance as the oracle's, the pass
    counts enumerated in full, for budgets both sides can enumerate."""
    code = inputs.single_code(300 + n, p, n, k)
    o = B.fpcode_opts_default(budget=2 * 10**6, mid_pass_exit=0)
    a = B.fpcode_min_distance_ex(B.fpcode_prepare(p, n, k, code.G, o), None, o)
    b = oracle.bz(code, threads=4, budget=2 * 10**6)
    assert {oracle.OK: B.OK, oracle.EBUDGET: B.EBUDGET}[b.status] == a.status
    assert (a.L, a.U) == (b.L, b.U) and list(a.counts) == list(b.counts)
    assert a.enumerated == sum(a.counts)
    w = np.array(a.witness)
    assert np.count_nonzero(w) == a.U
