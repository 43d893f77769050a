"""GPU test of the hard-leaf sieve's crossing counter: every multiple k p_b (k >= p_b, coprime to
30) that a step of a prime above 64 crosses off is counted once, whatever the runs' lengths."""
import numpy as np
import pytest

import oracle as o
import paper_1503_01839_gb300 as pc

pytestmark = pytest.mark.gpu


def primes_upto(n):
    s = np.ones(n + 1, dtype=bool)
    s[:2] = False
    for i in range(2, int(n ** 0.5) + 1):
        if s[i]:
            s[i * i::i] = False
    return np.flatnonzero(s)


def crossings(x, y, seg):
    """Over segments [L, L + span) of [0, z]: the step of p_b, b < B_s, crosses the multiples off;
    B_s counts the primes up to min(isqrt(x / L), isqrt(L + span - 1), x^(1/4), isqrt(z))."""
    z, span = x // y, 30 * seg
    top = min(o.isqrt(o.isqrt(x)), o.isqrt(z))
    ps = [int(p) for p in primes_upto(top)]
    cop = [r for r in range(30) if all(r % q for q in (2, 3, 5))]

    def upto(n):   # integers in [1, n] coprime to 30
        return 8 * (n // 30) + sum(1 for r in cop if r <= n % 30)

    total = 0
    for L in range(0, z + 1, span):
        n = L + span - 1
        r = o.isqrt(min(n, x // L) if L else n)
        mine = [p for p in ps if p <= r][:-1]   # b < B_s
        for p in mine:
            if p > 64:
                lo = max((L + p - 1) // p, p)
                hi = n // p
                if hi >= lo:
                    total += upto(hi) - upto(lo - 1)
    return total


@pytest.mark.parametrize("x,alpha,seg", [(10 ** 10, 1, 4096), (10 ** 11, 2, 1024), (10 ** 12, 4, 8192),
                                         (10 ** 13, 8, 32768)])
def test_every_crossing_counted_once(x, alpha, seg):
    y = alpha * o.iroot3(x)
    with pc.Context(0, seg_bytes=seg) as cx:
        cx.s2_hard(x, y, 5)
        assert cx.stats()["clears"] == crossings(x, y, seg)
