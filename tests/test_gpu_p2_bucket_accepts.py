"""GPU test of P2's bucket mode at segments longer than the pi table: a sum without terms, or so
small that it is read from the table, asks for no bucket prime and is answered; where bucket
primes would be looked up beyond the table the call is refused."""
import pytest

import oracle as o
import paper_1503_01839_gb300 as pc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seg", [126976, 131072])
def test_bucket_mode_without_terms(seg):
    with pc.Context(0, p2_bucket=1, seg_bytes=seg) as cx, pc.Context(0) as plain:
        assert cx.p2(10 ** 6, 1000) == 0                     # y = isqrt(x)
        assert cx.leaf_sums(10 ** 6, 1000, 5) == plain.leaf_sums(10 ** 6, 1000, 5)
        assert cx.leaf_sums(10 ** 6 - 1, 998, 5) == plain.leaf_sums(10 ** 6 - 1, 998, 5)   # no prime in (998, 999]
        assert cx.p2(20, 2) == o.p2(20, 1)                   # fewer than three sieving primes
        with pytest.raises(pc.PicountError):
            cx.p2(10 ** 6, 500)
