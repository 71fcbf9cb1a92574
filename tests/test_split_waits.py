"""What the tensor-core kernel does when a product never counts as complete:
its waits end, and the launch leaves a usable handle behind."""
import time

import pytest

from paper_2603_29942_gb300 import _binding as B
from paper_2603_29942_gb300 import inputs


def _same(a, b):
    for f in ("status", "d", "L", "U", "m", "npasses", "counts", "kj", "best_key", "enumerated"):
        assert getattr(a, f) == getattr(b, f), f


@pytest.mark.gpu
@pytest.mark.parametrize("p,n,k,budget", [(3, 80, 40, 0), (7, 52, 19, 3 * 10 ** 8), (5, 40, 20, 0)])
def test_lost_product_ends_the_launch(p, n, k, budget):
    """One warpgroup of each CTA waits for an arrival that nobody makes: it
    gives up after about a second, the other warps of its CTA are not left in
    a barrier, and the same handle then gives the same result as before."""
    code = inputs.single_code(400 + n, p, n, k)
    o = B.fpcode_opts_default(budget=budget, mid_pass_exit=0)
    pr = B.fpcode_test_prepare_split(p, n, k, code.G, o)
    before = B.fpcode_min_distance_ex(pr, None, o)
    B.fpcode_test_lose_products(pr, True)
    t0 = time.time()
    for _ in range(2):
        B.fpcode_min_distance_ex(pr, None, o)
    assert time.time() - t0 < 20
    B.fpcode_test_lose_products(pr, False)
    _same(B.fpcode_min_distance_ex(pr, None, o), before)


@pytest.mark.gpu
@pytest.mark.parametrize("p,n,k,budget", [(3, 80, 40, 0), (7, 52, 19, 3 * 10 ** 8), (5, 40, 20, 0)])
def test_lost_product_is_a_timeout(p, n, k, budget):
    """A task that was not compared in full is not counted off: the search
    reports a timeout, certifies nothing and claims no distance."""
    code = inputs.single_code(400 + n, p, n, k)
    o = B.fpcode_opts_default(budget=budget, mid_pass_exit=0)
    pr = B.fpcode_test_prepare_split(p, n, k, code.G, o)
    whole = B.fpcode_min_distance_ex(pr, None, o)
    B.fpcode_test_lose_products(pr, True)
    r = B.fpcode_min_distance_ex(pr, None, o)
    assert r.status == B.ETIMEOUT and r.d == -1
    assert r.L <= whole.L and r.U >= whole.U


@pytest.mark.gpu
@pytest.mark.parametrize("p,n,k", [(3, 80, 40), (7, 40, 20), (5, 51, 24)])
def test_search_that_ends_inside_direct_passes(p, n, k):
    """A code with a codeword of weight 1 certifies with its first pass, while
    other CTAs walk stems of the passes after it with every weight exact: the
    finished flag reaches them in the middle, 200 times over."""
    code = inputs.single_code(500 + n, p, n, k)
    G = code.G.copy()
    G[0, k:] = 0
    o = B.fpcode_opts_default()
    pr = B.fpcode_test_prepare_split(p, n, k, G, o)
    for _ in range(200):
        r = B.fpcode_min_distance_ex(pr, None, o)
        assert r.status == B.OK and r.d == 1 and r.enumerated == sum(r.counts)
