"""GPU test: easy leaves that do not read the odd-number pi table (the sampled table, or
y >= 2^29) run after the hard-leaf sieve, not beside it, where they are the longer of the two."""
import pytest

import paper_1503_01839_gb300 as pc

pytestmark = pytest.mark.gpu


def test_sampled_leaves_do_not_share_the_chip_with_the_sieve(pi_pow10):
    with pc.Context(0, pi_gather=1) as cx:
        for _ in range(2):
            assert cx.pi_count(10 ** 16) == pi_pow10[16]
        st = cx.stats()
        assert st["ms_hard"] + st["ms_easy"] <= 1.05 * st["ms_total"]


def test_large_y_leaves_do_not_share_the_chip_with_the_sieve():
    x, y = 4 * 10 ** 17, 6 * 10 ** 8
    with pc.Context(0) as cx:
        s = cx.leaf_sums(x, y, 5)
        st = cx.stats()
        assert st["ms_hard"] + st["ms_easy"] <= 1.05 * st["ms_total"]
        assert s["S1"] + s["S2_triv"] + s["S2_easy"] + s["S2_hard"] + st["a"] - 1 - s["P2"] == cx.pi_count(x)
