"""GPU test of pc_table_leaves: the hard leaves (b, q), q a prime in (p_b, y], with
y <= u = x / (p_b q) < p_b^2."""
import pytest

import oracle as o
import paper_1503_01839_gb300 as pc

pytestmark = pytest.mark.gpu


def table_leaves(x, y, c):
    ps = [p for p in range(2, y + 1) if all(p % d for d in range(2, o.isqrt(p) + 1))]
    n = 0
    for b, p in enumerate(ps, 1):
        if b > max(c, 3) and p * p > y:
            n += sum(1 for q in ps[b:] if y <= x // (p * q) < p * p)
    return n


@pytest.mark.parametrize("x,alpha", [(10 ** 8, 1), (10 ** 9, 2), (3 * 10 ** 10, 1)])
def test_table_leaves_counted(x, alpha):
    y = alpha * o.iroot3(x)
    want = table_leaves(x, y, 5)
    with pc.Context(0) as cx:
        cx.s2_hard(x, y, 5)
        assert cx.table_leaves() == want > 0
        assert cx.stats()["hard_leaves"] == o.leaf_sums(x, y, 5)["n_hard"]
        cx.pi_count(1000)
        assert cx.table_leaves() == 0
