"""The arithmetic of the one-product quotient of the easy leaves, on CPU.

This restates in Python the formula of QuotOf (pc_common.cuh), not the kernel: the kernels'
results are checked on the GPU by the pi(x) and leaf-sum parity tests.  For a dividend n with
k = max(0, bits - 32), T = floor(n / 2^k), and a divisor d with s = floor(log2 d),
v = floor((2^(32+s) - 1) / d), the estimate floor(floor(T v / 2^32) / 2^(s-k)) is the quotient
or one less below 2^30, s >= k there, and the remainder's low 32 bits settle it.  From 2^30 up
to 2^31 (a clustered run's bound, clamped to q < 2^29) it may fall short by two."""
import random

import pytest


def estimate(n, d):
    k = max(0, n.bit_length() - 32)
    s = d.bit_length() - 1
    v = ((1 << (32 + s)) - 1) // d
    assert s >= k, (n, d)
    return (((n >> k) * v) >> 32) >> (s - k)


def quot(n, d):
    q = estimate(n, d)
    r = ((n & 0xFFFFFFFF) - q * d) & 0xFFFFFFFF
    return q + (r >= d)


def check(n, d):
    want = n // d
    if want < 1 << 30:
        assert estimate(n, d) in (want - 1, want), (n, d)
        assert quot(n, d) == want, (n, d)
    else:
        assert want - 2 <= estimate(n, d) <= want, (n, d)
        assert quot(n, d) >= 1 << 29


@pytest.mark.parametrize("dbits", [2, 3, 13, 22, 29, 30])
def test_quotients(dbits):
    rng = random.Random(dbits)
    ds = [(1 << dbits) - 1, 1 << (dbits - 1), (1 << (dbits - 1)) + 1]
    ds += [rng.randrange(1 << (dbits - 1), 1 << dbits) for _ in range(400)]
    for d in ds:
        qs = [0, 1, 2, (1 << 30) - 1, 1 << 30, (1 << 30) + 1, (1 << 31) - 3]
        qs += [rng.randrange(1, 1 << rng.randrange(1, 31)) for _ in range(60)]
        qs += [((1 << e) // d) + o for e in range(31, 61) for o in (-1, 0, 1)]   # n around a power of two
        for q in qs:
            for r in (0, 1, d // 2, d - 1):
                if 0 <= q < (1 << 31) - 2 and 0 < q * d + r < 1 << 63:
                    check(q * d + r, d)


def near(n, d):
    s = d.bit_length() - 1
    k = max(0, s - 13)
    v = ((1 << (32 + s)) - 1) // d
    t = n >> k
    assert t < 1 << 32
    q = ((t * v) >> 32) >> (s - k)
    return q + (n - q * d >= d)


@pytest.mark.parametrize("dbits", [1, 2, 13, 14, 15, 27, 31, 32])
def test_near(dbits):
    # div_near: quotients below 2^18, any 32-bit divisor (the offset of a leaf in a sub-range)
    rng = random.Random(dbits)
    lo, hi = 1 << (dbits - 1), (1 << dbits) - 1
    for d in {lo, hi, min(lo + 1, hi)} | {rng.randrange(lo, hi + 1) for _ in range(500)}:
        for q in [0, 1, (1 << 18) - 1, 245759] + [rng.randrange(1 << 18) for _ in range(50)]:
            for r in {0, d // 2, d - 1}:
                assert near(q * d + r, d) == q, (q, d, r)


def two_steps(n, d):
    s = d.bit_length() - 1
    top = d >> (s - 15) if s >= 15 else d << (15 - s)
    v = 0xFFFFFFFF // (top + 1)
    assert v < 1 << 17
    k = max(0, s - 9)
    assert n >> k < 1 << 32
    q = ((n >> k) * v) >> (17 + s - k)
    r = n - q * d
    assert 0 <= r < d << 9, (n, d)
    k2 = max(0, s - 21)
    assert r >> k2 < 1 << 32
    q2 = ((r >> k2) * v) >> (17 + s - k2)
    r -= q2 * d
    assert 0 <= r < 4 * d, (n, d)
    return q + q2 + r // d


@pytest.mark.parametrize("dbits", [1, 2, 8, 15, 16, 17, 23, 24, 31, 32])
def test_two_steps(dbits):
    # p2_div (pc_p2.cu): quotients below 2^22, any 32-bit divisor
    rng = random.Random(dbits)
    lo, hi = 1 << (dbits - 1), (1 << dbits) - 1
    for d in {lo, hi, min(lo + 1, hi)} | {rng.randrange(lo, hi + 1) for _ in range(500)}:
        for q in [0, 1, 2, (1 << 22) - 1] + [rng.randrange(1 << rng.randrange(1, 23)) for _ in range(50)]:
            for r in {0, d // 2, d - 1}:
                assert two_steps(q * d + r, d) == q, (q, d, r)
