"""GPU test of segment sizes that sixteen power-of-two sub-ranges cannot tile: odd multiples of
4096 bytes above 65536.  The sieve, whole pi(x), shards and the batch give what 32 KiB
segments give."""
import pytest

import oracle as o
import paper_1503_01839_gb300 as pc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seg", [69632, 77824, 126976])
@pytest.mark.parametrize("warp", [0, 1024, 4096, 8192])
def test_odd_segments_above_64k(seg, warp):
    x = 3 * 10 ** 12
    y = 4 * o.iroot3(x)
    xs = [10 ** 9 + 7, 10 ** 11, 3 * 10 ** 12]
    with pc.Context(0, seg_bytes=32768) as cx, pc.Context(0, seg_bytes=seg, warp_bytes=warp) as odd:
        assert odd.s2_hard(x, y, 5) == cx.s2_hard(x, y, 5)
        assert odd.p2(x, y) == cx.p2(x, y)
        want = [cx.pi_count(v) for v in xs]
        assert [odd.pi_count(v) for v in xs] == want
        assert sum(odd.s2_hard_shard(x, y, 5, k, 3) for k in range(3)) == cx.s2_hard(x, y, 5)
        assert list(odd.pi_count_batch(xs)) == want
