"""What is measured: the calls a program that counts primes makes, through the package's public
entry points (Context and Server), from queries where launches and latency count to ones that
fill the GPU for a tenth of a second or more.

A case fixes the call and the size of x; the x itself comes from the seed, within 3 percent above
the case's size (a batch or a served stream draws all of its queries from the seed).  A program
that counts primes keeps its Context: it holds the device tables and the scratch.  So prepare()
makes one and calls it once at the largest x of the case, and run() is one call on other numbers.
Every output is a whole number.
"""
from __future__ import annotations

import math

import numpy as np

import paper_1503_01839_gb300 as pc
from paper_1503_01839_gb300 import inputs

SPREAD = 0.03   # a case's x lies in [x, x * (1 + SPREAD))


def listed():
    return [
        # the smallest query that runs the whole method (below 2^20 pi(x) is one table lookup)
        {"name": "pi_3e7", "kind": "pi", "x": 30_000_000, "alpha": 0},
        # the paper's plainest setting, y = iroot3(x): every special leaf is a hard one
        {"name": "pi_1e10_alpha1", "kind": "pi", "x": 10 ** 10, "alpha": 1},
        # single queries, the library choosing alpha: short ones, an ordinary one, the
        # paper's two headline sizes
        {"name": "pi_1e12", "kind": "pi", "x": 10 ** 12, "alpha": 0},
        {"name": "pi_1e14", "kind": "pi", "x": 10 ** 14, "alpha": 0},
        {"name": "pi_1e16", "kind": "pi", "x": 10 ** 16, "alpha": 0},
        {"name": "pi_1e18", "kind": "pi", "x": 10 ** 18, "alpha": 0},
        # the partial sieve function, its tree cut at p_a
        {"name": "phi_1e14_a1000", "kind": "phi", "x": 10 ** 14, "a": 1000},
        # the hard special leaves on their own: the benchmark's step
        {"name": "s2_hard_1e18", "kind": "s2_hard", "x": 10 ** 18, "alpha": 20, "c": 5},
        # the second partial sum on its own
        {"name": "p2_1e17", "kind": "p2", "x": 10 ** 17, "alpha": 20},
        # all five parts, at an odd alpha and a shallow wheel, the tree cut at p_a
        {"name": "leaf_sums_1e15", "kind": "leaf_sums", "x": 10 ** 15, "alpha": 9, "c": 3, "a": 20_000},
        # many mixed queries at once: the benchmark's batch
        {"name": "batch_4096", "kind": "batch", "n": 4096, "lo": 8.0, "hi": 15.0},
        # a burst of served requests, a fifth of them phi(x, a), eight of them running at a time
        {"name": "serve_48", "kind": "serve", "n": 48, "lo": 9.0, "hi": 17.0},
    ]


def draw(rng):
    kind = rng.choice(["pi", "pi", "pi", "phi", "s2_hard", "p2", "leaf_sums", "batch", "serve"])

    def x_of(lo, hi):
        return int(10.0 ** rng.uniform(lo, hi))

    if kind == "pi":
        x = x_of(7.0, 18.9)
        # a fixed alpha is mostly used for small x, where it costs little
        alpha = rng.randint(1, 20) if x < 10 ** 12 and rng.random() < 0.3 else 0
        return {"kind": kind, "x": x, "alpha": alpha}
    if kind == "phi":
        return {"kind": kind, "x": x_of(9.0, 17.0), "a": rng.randint(5, 5000)}
    if kind == "s2_hard":
        return {"kind": kind, "x": x_of(11.0, 18.3), "alpha": rng.randint(10, 40), "c": rng.choice([4, 5, 5, 6])}
    if kind == "p2":
        return {"kind": kind, "x": x_of(11.0, 18.3), "alpha": rng.randint(10, 40)}
    if kind == "leaf_sums":
        return {"kind": kind, "x": x_of(9.0, 16.5), "alpha": rng.randint(2, 30), "c": rng.randint(1, 7),
                "a": rng.choice([0, 0, rng.randint(20, 60)])}
    if kind == "batch":
        lo = rng.uniform(7.0, 10.0)
        return {"kind": kind, "n": int(2 ** rng.uniform(4.0, 12.0)), "lo": lo, "hi": rng.uniform(lo + 1.0, 15.0)}
    lo = rng.uniform(8.0, 11.0)
    return {"kind": kind, "n": rng.randint(8, 48), "lo": lo, "hi": rng.uniform(lo + 2.0, 17.0)}


def _iroot3(n):
    r = round(n ** (1.0 / 3.0))
    while r ** 3 > n:
        r -= 1
    while (r + 1) ** 3 <= n:
        r += 1
    return r


def _y(case, x):
    return min(case["alpha"] * _iroot3(x), math.isqrt(x))


def _x(case, seed):
    return case["x"] + int(np.random.default_rng(seed).uniform(0.0, SPREAD) * case["x"])


def _call(cx, case, x):
    kind = case["kind"]
    if kind == "pi":
        return cx.pi_count(x, case["alpha"])
    if kind == "phi":
        return cx.phi(x, case["a"])
    if kind == "s2_hard":
        return cx.s2_hard(x, _y(case, x), case["c"])
    if kind == "p2":
        return cx.p2(x, _y(case, x))
    return cx.leaf_sums(x, _y(case, x), case["c"], case["a"])


def prepare(case, seed):
    cx = pc.Context(0)
    if case["kind"] == "batch":
        xs = inputs.log_uniform_x(case["n"], case["lo"], case["hi"], seed)
        cx.pi_count_batch([int(10.0 ** case["hi"])])
        return {"case": case, "cx": cx, "xs": xs}
    if case["kind"] == "serve":
        trace = inputs.served_trace(case["n"], seed=seed, lo_exp=case["lo"], hi_exp=case["hi"])
        return {"case": case, "cx": cx, "trace": trace, "srv": pc.Server(cx, int(10.0 ** case["hi"]), 5000)}
    _call(cx, case, case["x"] + int(SPREAD * case["x"]))
    return {"case": case, "cx": cx, "x": _x(case, seed)}


def run(state):
    case, cx = state["case"], state["cx"]
    if case["kind"] == "batch":
        return np.array(cx.pi_count_batch(state["xs"]), dtype=np.int64)
    if case["kind"] == "serve":
        srv = state["srv"]
        for i, q in enumerate(state["trace"]):
            srv.submit(pc.PC_QUERY_PI if q["kind"] == "pi" else pc.PC_QUERY_PHI, q["x"], q["a"], tag=i)
        value = np.zeros(case["n"], dtype=np.int64)
        got = 0
        while got < case["n"]:
            for r in srv.poll(timeout_ms=-1):
                if r["status"] != pc.PC_OK:
                    raise RuntimeError("request %d failed with %d" % (r["tag"], r["status"]))
                value[r["tag"]] = r["value"]
                got += 1
        return value
    return _call(cx, case, state["x"])


def _ops(x):
    """Integer operations of one evaluation at x: the method's x^(2/3) / ln^2 x."""
    return x ** (2.0 / 3.0) / math.log(x) ** 2


def work(case):
    """One number or pair of numbers in and one out per query; the operations are the method's
    x^(2/3) / ln^2 x (a mean over the range for a batch or a stream)."""
    if case["kind"] in ("batch", "serve"):
        n, lo, hi = case["n"], case["lo"], case["hi"]
        mean = sum(_ops(10.0 ** (lo + (hi - lo) * (k + 0.5) / 64)) for k in range(64)) / 64
        return {"bytes": 16 * n, "flops": n * mean}
    return {"bytes": 24, "flops": _ops(float(case["x"]))}


def _sieved(x, a):
    """S(x) = #{2 <= n <= x: n prime, or every prime factor of n above p_a}, by the recurrence over
    the values floor(x / i) (every prime up to isqrt(x) when a is None)."""
    r = math.isqrt(x)
    small = np.arange(r + 1, dtype=np.int64) - 1              # S(v), v <= r
    idx = np.arange(1, r + 1, dtype=np.int64)
    large = np.concatenate([np.zeros(1, dtype=np.int64), x // idx - 1])   # S(x // i)
    k = 0
    for p in range(2, r + 1):
        if small[p] == small[p - 1]:
            continue
        if a is not None and k == a:
            break
        k += 1
        before = int(small[p - 1])
        top = min(r, x // (p * p))
        i = np.arange(1, top + 1, dtype=np.int64)
        near = int(np.searchsorted(i * p, r, side="right"))   # i * p <= r
        take = np.empty(top, dtype=np.int64)
        take[:near] = large[i[:near] * p]
        take[near:] = small[x // (i[near:] * p)]
        large[1:top + 1] -= take - before
        if p * p <= r:
            v = np.arange(p * p, r + 1, dtype=np.int64)
            small[p * p:] -= small[v // p] - before
    return int(large[1]), k


def exact(case, seed):
    """pi(x) and phi(x, a) for x up to 10^12, by a recurrence that shares nothing with the package."""
    if case["kind"] not in ("pi", "phi") or case["x"] > 10 ** 12:
        return None
    x = _x(case, seed)
    if case["kind"] == "pi":
        return _sieved(x, None)[0]
    s, k = _sieved(x, case["a"])
    # S(x) counts the primes up to p_k too, phi(x, a) the integer 1 instead; past isqrt(x) only
    # primes are left, and each further p_a takes one of them
    return s - k + 1 if k == case["a"] else max(1, s - case["a"] + 1)
