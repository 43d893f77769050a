"""GPU test of a tuned context: the tuned segment size is the hard-leaf sieve's, a limit on the size
the rule by z takes, and P2 keeps its own segments."""
import pytest

import paper_1503_01839_gb300 as pc

pytestmark = pytest.mark.gpu

XS = [2 * 10 ** 9, 3 * 10 ** 10, 10 ** 12, 2 * 10 ** 13]


@pytest.fixture(scope="module")
def tuned():
    with pc.Context(0) as cx:
        cx.autotune(min(XS), max(XS), reps=1)
        yield cx


@pytest.mark.parametrize("x", XS)
def test_p2_keeps_its_segments(tuned, x):
    alpha, _ = tuned.tuned(x)
    with pc.Context(0) as plain:
        assert tuned.pi_count(x) == plain.pi_count(x, alpha)
        got, want = tuned.stats(), plain.stats()
    assert got["y"] == want["y"]
    # P2's sieve starts at a bound of its own segments: the same crossings, the same segments
    assert got["p2_clears"] == want["p2_clears"]


@pytest.mark.parametrize("x", XS)
def test_small_z_keep_the_rule(tuned, x):
    """A tuned size of 16 or 32 KiB is a limit on the size the rule by z takes."""
    alpha, seg = tuned.tuned(x)
    with pc.Context(0) as plain:
        assert tuned.pi_count(x) == plain.pi_count(x, alpha)
        rule = plain.stats()["seg_bytes"]
    assert tuned.stats()["seg_bytes"] == (seg if seg > 32768 else min(seg, rule))
