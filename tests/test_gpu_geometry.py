"""GPU test of the sieves' default geometry: just below and just above every line of the rules
that pick segment and sub-range bytes from z, the default gives what fixed 32 KiB segments give."""
import pytest

import oracle as o
import paper_1503_01839_gb300 as pc

pytestmark = pytest.mark.gpu

LINES = [400_000, 12_000_000, 40_000_000, 120_000_000, 280_000_000, 300_000_000, 800_000_000, 1_200_000_000,
         2_000_000_000, 2_200_000_000]


@pytest.mark.parametrize("z", LINES)
def test_default_geometry_at_its_lines(z):
    y = max(1000, int(z ** 0.6))
    with pc.Context(0) as cx, pc.Context(0, seg_bytes=32768, warp_bytes=8192) as fixed:
        for zz in (z - 1, z):
            x = zz * y + y // 2          # floor(x / y) = zz
            assert x // y == zz and o.iroot3(x) <= y <= o.isqrt(x)
            assert cx.s2_hard(x, y, 5) == fixed.s2_hard(x, y, 5), zz
            assert cx.p2(x, y) == fixed.p2(x, y), zz


@pytest.mark.parametrize("x,y,n", [(1136286593, 11662, 3), (11892848023, 81551, 3), (52247375021686, 1075462, 5)])
def test_shard_bounds_do_not_follow_the_rule(x, y, n):
    """Shards are runs of 32 KiB segments at every z."""
    with pc.Context(0) as cx, pc.Context(0, seg_bytes=32768) as fixed:
        got = [cx.s2_hard_shard(x, y, 5, k, n) for k in range(n)]
        assert got == [fixed.s2_hard_shard(x, y, 5, k, n) for k in range(n)]
        assert sum(got) == cx.s2_hard(x, y, 5)
