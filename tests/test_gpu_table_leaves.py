"""GPU tests of the hard leaves read from the pi table (y <= u < p_b^2) beside those of the
sieve (u >= p_b^2): every part equals the oracle's at y around the fourth root, the cube root
and the square root of x, at segments so small that the rows of the count table start and end
at many different segments, for a truncated tree, and split into shards."""
import pytest

import oracle as o
import paper_1503_01839_gb300 as pc

pytestmark = pytest.mark.gpu

SIZES = [(10 ** 4, 0), (10 ** 6 + 3, 0), (2 ** 31 - 1, 0), (3 * 10 ** 9, 25), (10 ** 10 + 19, 60)]


@pytest.mark.parametrize("x,a", SIZES)
@pytest.mark.parametrize("seg", [1024, 32768])
def test_parts_match_oracle(x, a, seg):
    r2, r3 = o.isqrt(x), o.iroot3(x)
    with pc.Context(0, seg_bytes=seg) as cx:
        for y in sorted({o.isqrt(r2) + 1, r3 - 1, r3, r3 + 1, 2 * r3, (r2 + r3) // 2, r2 - 1, r2}):
            if not 1 <= y <= r2 or x // y > 3 * 10 ** 7:
                continue
            n = o.pi_sieve(y)
            for c in (3, 5, 7):
                if c > n or (a and not c <= a <= n):
                    continue
                want = o.leaf_sums(x, y, c, a)
                got = cx.leaf_sums(x, y, c, a)
                for k in ("S1", "S2_triv", "S2_easy", "S2_hard"):
                    assert got[k] == want[k], (x, y, c, a, seg, k)


@pytest.mark.parametrize("x,alpha", [(10 ** 9, 1), (10 ** 10 + 19, 3), (10 ** 11, 1)])
def test_shards_split_the_table_leaves(x, alpha):
    y = min(alpha * o.iroot3(x), o.isqrt(x))
    with pc.Context(0, seg_bytes=1024) as cx:
        want = o.leaf_sums(x, y, 5)["S2_hard"]
        assert cx.s2_hard(x, y, 5) == want
        leaves = cx.stats()["hard_leaves"]
        for n in (2, 5):
            got, seen = 0, 0
            for k in range(n):
                got += cx.s2_hard_shard(x, y, 5, k, n)
                seen += cx.stats()["hard_leaves"]
            assert (got, seen) == (want, leaves), (x, n)
