"""GPU test of P2 for y < 5: the primes 2, 3 and 5 are terms of the sum too, and the mod-30
bitset that holds the others has no place for them."""
import pytest

import oracle as o
import paper_1503_01839_gb300 as pc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("x", [20, 49, 120, 121, 10 ** 4, 10 ** 6 + 3, 10 ** 8])
@pytest.mark.parametrize("prm", [{}, {"seg_bytes": 1024}, {"p2_bucket": 1, "seg_bytes": 2048}])
def test_p2_at_the_smallest_y(x, prm):
    with pc.Context(0, **prm) as cx:
        for y in range(1, 8):
            if y * y > x:
                break
            want = o.p2(x, o.pi_sieve(y))
            assert cx.leaf_sums(x, y, 0)["P2"] == want, (x, y)
            if y >= o.iroot3(x):
                assert cx.p2(x, y) == want, (x, y)
