"""The work that users of this framework have it do, as cases to be timed.

A case is one call, or one prepared search, a batch or a burst of requests,
through the public entry points (paper_2603_29942_gb300/_binding.py, which
keeps the names of the C interface).  Kinds:

  call    fpcode_min_distance: from a host matrix to a certified distance and
          a witness (preparation, upload, search, read-back);
  search  fpcode_min_distance_ex on a prepared, uploaded code, as programs do
          that search the same code under a budget, resume it or repeat it;
  batch   fpcode_min_distance_batch over many codes of uneven shape;
  serve   a server that is kept, a burst of requests submitted and polled.

The codes are seeded random systematic codes, as in the paper's experiments.
A case names a base code ("code", a seed); `seed` picks another member of its
class: rows and redundant columns permuted and scaled by nonzero constants.
Every member has the same parameters and minimum distance, so every seed asks
for about the same work on other matrices (random codes of one shape differ
in d, and with it in work by a factor of ten).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2603_29942_gb300 import _binding as B
from paper_2603_29942_gb300 import inputs

SERVE_SLOTS = 64


def listed():
    return [
        # Table 5's 15 x 30 matrix over F_3: the smallest call, all latency.
        {"name": "call_f3_n30_k15", "kind": "call", "p": 3, "n": 30, "k": 15, "code": 0, "work": 450},
        # The heptary code of the configurations, from a host matrix: an ordinary small search.
        {"name": "call_f7_n40_k20", "kind": "call", "p": 7, "n": 40, "k": 20, "code": 1, "work": 42363808},
        # The headline code end to end: what a program pays for one distance.
        {"name": "call_f3_n80_k40", "kind": "call", "p": 3, "n": 80, "k": 40, "code": 2, "work": 268257056},
        # The headline code prepared once and searched again (the device search itself).
        {"name": "search_f3_n80_k40", "kind": "search", "p": 3, "n": 80, "k": 40, "code": 2, "work": 268257056},
        # Table 3's parameters over F_7: a search of some 10^9 codewords.
        {"name": "search_f7_n50_k25", "kind": "search", "p": 7, "n": 50, "k": 25, "code": 5, "work": 2.898e9},
        # Table 4's parameters over F_7, three information sets, the last one rank-deficient: the longest search.
        {"name": "search_f7_n52_k19", "kind": "search", "p": 7, "n": 52, "k": 19, "code": 6, "work": 2.889e10},
        # The far end of the paper's ternary data set (k <= 50, n <= 74): high rate, a second set of rank 24.
        {"name": "search_f3_n74_k50", "kind": "search", "p": 3, "n": 74, "k": 50, "code": 7, "budget": 10**10,
         "work": 6.937e9},
        # p = 5, odd sizes, every pass enumerated in full so that the counts can be checked (no mid-pass exit).
        {"name": "search_f5_n51_k24", "kind": "search", "p": 5, "n": 51, "k": 24, "code": 8, "mid_pass_exit": 0,
         "work": 2.988e8},
        # A prime with five bits a symbol and two words a slice, stopped at a budget and returned as an interval.
        {"name": "search_f31_n70_k10", "kind": "search", "p": 31, "n": 70, "k": 10, "code": 9, "budget": 10**9,
         "work": 8.569e8},
        # The batched workload of the configurations: 512 uneven codes with a budget each.
        {"name": "batch512_f37", "kind": "batch", "count": 512, "primes": "3,7", "nlo": 24, "nhi": 64, "code": 3,
         "budget": 10**8, "work": 9.53e9},
        # A small batch with the primes that share a launch and one that has its own.
        {"name": "batch24_f35711", "kind": "batch", "count": 24, "primes": "3,5,7,11", "nlo": 20, "nhi": 48,
         "code": 10, "budget": 10**7, "work": 6.23e7},
        # A burst of requests at a server that has as many slots (p in {3, 5, 7}, n up to 72).
        {"name": "serve64_f357", "kind": "serve", "count": 64, "primes": "3,5,7", "nlo": 20, "nhi": 72, "code": 4,
         "budget": 10**8, "work": 1.518e9},
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _expected(p, n, k, extra):
    """Codewords a search is expected to take if d lies `extra` above the Gilbert-Varshamov estimate."""
    total, d = 0, n
    for i in range(n + 1):
        total += math.comb(n, i) * (p - 1) ** i
        if total >= p ** (n - k):
            d = i + 1
            break
    m, work = max(1, n // k), 0
    for g in range(1, k + 1):
        work += m * math.comb(k, g) * (p - 1) ** (g - 1)
        if m * (g + 1) >= d + extra:
            break
    return work


def draw(rng):
    kind = rng.choice(["call", "call", "search", "search", "search", "search", "batch", "serve"])
    code = rng.randrange(1000, 10**6)
    if kind in ("batch", "serve"):
        primes = rng.choice(["3", "7", "3,7", "3,5,7", "3,5,7,11"] if kind == "batch" else ["3", "3,5,7", "3,7"])
        nlo = rng.randrange(16, 32)
        case = {"kind": kind, "count": _loguniform(rng, 2, 512 if kind == "batch" else SERVE_SLOTS), "primes": primes,
                "nlo": nlo, "nhi": rng.randrange(nlo + 8, 65 if kind == "batch" else 73), "code": code,
                "budget": _loguniform(rng, 10**6, 10**8)}
        case["work"] = float(case["count"] * case["budget"]) / 4
        return case
    while True:
        p = rng.choice([3, 3, 3, 7, 7, 5, 5, 11, 13, 31, 127])
        k = _loguniform(rng, 5, 12 if p > 30 else 64)
        n = k + _loguniform(rng, 5, 96)
        r = p.bit_length()
        words = (r * -(-(n - k) // 32) + 3) // 4 * 4
        if k * (p - 1) * words * 4 > 80 * 1024 or n < 10:
            continue
        case = {"kind": kind, "p": p, "n": n, "k": k, "code": code}
        if kind == "call":
            work = _expected(p, n, k, 3)
            if p > 13 or work > 4 * 10**9:
                continue
        else:
            case["budget"] = _loguniform(rng, 10**5, 5 * 10**9 if p <= 7 else 5 * 10**8)
            case["mid_pass_exit"] = rng.randrange(2)
            case["per_round_check"] = rng.choice([0, 0, 0, 1])
            work = min(case["budget"], _expected(p, n, k, 0))
        case["work"] = float(work)
        return case


def _member(rng, p, n, k, A):
    """[I | A'] with A' = A, its rows and columns permuted and scaled by nonzero constants."""
    rows = rng.permutation(k)
    cols = rng.permutation(n - k)
    rs = rng.integers(1, p, size=(k, 1))
    cs = rng.integers(1, p, size=(1, n - k))
    return inputs.systematic(p, n, k, (A[rows][:, cols].astype(np.int64) * rs * cs % p).astype(np.uint8))


def _code(case, seed):
    p, n, k = case["p"], case["n"], case["k"]
    base = inputs.single_code(case["code"], p, n, k)
    return _member(np.random.default_rng([seed, 17]), p, n, k, base.G[:, k:])


def _codes(case, seed):
    """`count` codes: p from the case's primes, n from its range, rate between 1/3 and 2/3."""
    base = np.random.default_rng(case["code"])
    rng = np.random.default_rng([seed, 18])
    primes = [int(x) for x in case["primes"].split(",")]
    out = []
    for _ in range(case["count"]):
        p = primes[int(base.integers(len(primes)))]
        n = int(base.integers(case["nlo"], case["nhi"] + 1))
        k = int(round(float(base.uniform(1 / 3, 2 / 3)) * n))
        out.append(_member(rng, p, n, k, base.integers(0, p, size=(k, n - k), dtype=np.uint8)))
    return out


def _opts(case):
    over = {f: case[f] for f in ("budget", "mid_pass_exit", "per_round_check") if f in case}
    return B.fpcode_opts_default(**over)


_server = None  # a program keeps one server; a short idle time gives the GPU back soon after a burst


def prepare(case, seed):
    global _server
    stream = torch.cuda.current_stream()
    state = {"kind": case["kind"], "stream": stream}
    if case["kind"] == "call":
        state["code"] = _code(case, seed)
    elif case["kind"] == "search":
        code = _code(case, seed)
        state["opts"] = _opts(case)
        state["prep"] = B.fpcode_prepare(code.p, code.n, code.k, code.G, state["opts"])
        B.fpcode_prepared_upload(state["prep"], stream)
    else:
        state["codes"] = _codes(case, seed)
        state["budget"] = case["budget"]
        if case["kind"] == "batch":
            state["opts"] = _opts(case)
        else:
            if _server is None:
                _server = B.fpcode_serve_create(
                    B.fpcode_serve_opts_default(slots=SERVE_SLOTS, max_words=4, idle_exit_s=0.001), stream)
            state["server"] = _server
    return state


def _padded(rows, width):
    out = np.zeros((len(rows), width), dtype=np.int64)
    for i, r in enumerate(rows):
        if r is not None:
            out[i, :len(r)] = r
    return out


def _outputs(results):
    """Every field of the results but the times and the launch's number, as arrays."""
    out = {f: np.array([getattr(r, f) for r in results], dtype=np.int64)
           for f in ("status", "d", "L", "U", "m", "npasses", "enumerated")}
    out["best_key"] = np.array([r.best_key for r in results], dtype=np.uint64).view(np.int64)
    out["counts"] = _padded([np.array(r.counts, dtype=np.uint64).view(np.int64) for r in results], B.MAX_K + 1)
    out["kj"] = _padded([r.kj for r in results], B.MAX_M)
    out["witness"] = _padded([r.witness for r in results], B.MAX_N)
    return out


def run(state):
    kind = state["kind"]
    if kind == "call":
        c = state["code"]
        d, witness = B.fpcode_min_distance(c.p, c.n, c.k, c.G, state["stream"])
        return {"d": d, "witness": witness}
    if kind == "search":
        return _outputs([B.fpcode_min_distance_ex(state["prep"], state["stream"], state["opts"])])
    if kind == "batch":
        res = B.fpcode_min_distance_batch(state["codes"], state["stream"], state["opts"])
        f = res.field
        out = {x: f(x) for x in ("status", "d", "L", "U", "m", "npasses", "enumerated", "kj")}
        out["best_key"] = f("best_key").view(np.int64)
        out["counts"] = f("counts").view(np.int64)
        out["witness"] = res._wit
        return out
    server, codes = state["server"], state["codes"]
    order, got, at = {}, [None] * len(codes), 0
    left = len(codes)
    while left:
        if at < len(codes):
            ticket = B.fpcode_serve_submit(server, codes[at], state["budget"])
            if ticket is not None:
                order[ticket] = at
                at += 1
                continue
        for ticket, r in B.fpcode_serve_poll(server):
            got[order[ticket]] = r
            left -= 1
    return _outputs(got)


def work(case):
    """Input matrices and witnesses once; per codeword evaluated and 32-bit
    word of its redundant part, one operation per slice and one count."""
    if case["kind"] in ("call", "search"):
        n, k, p = case["n"], case["k"], case["p"]
        words, num = -(-(n - k) // 32), 1
    else:
        n = (case["nlo"] + case["nhi"]) // 2
        k, p = n // 2, max(int(x) for x in case["primes"].split(","))
        words, num = -(-(n - k) // 32), case["count"]
    return {"bytes": float(num * (n * k + n)), "flops": float(case["work"]) * words * (p.bit_length() + 1)}


def exact(case, seed):
    """The least weight over all messages, in plain numpy, where there are few of them."""
    if case["kind"] != "call" or case["p"] ** case["k"] > 2 * 10**7:
        return None
    c = _code(case, seed)
    p, k, h = c.p, c.k, c.k // 2

    def span(rows):
        words = np.zeros((1, c.n), dtype=np.int64)
        for row in rows.astype(np.int64):
            words = np.concatenate([(words + v * row) % p for v in range(p)])
        return words.astype(np.uint8)

    low, high = span(c.G[:h]), span(c.G[h:k])
    neg = (p - high) % p
    d = c.n
    for i in range(len(low)):
        w = (neg != low[i]).sum(axis=1)
        d = min(d, int(w[w > 0].min()))
    return {"d": d, "witness": None}
