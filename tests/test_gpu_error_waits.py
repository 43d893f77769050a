"""GPU test: a call that fails after it has enqueued work waits for that work before it returns, so
that the caller may switch streams or take the context down at once."""
import pytest

import paper_1503_01839_gb300 as pc

pytestmark = pytest.mark.gpu


def test_refused_s2_hard_leaves_nothing_running():
    import torch
    # count rows beyond 32 bits: found after the schedule's kernels have been enqueued
    x, y = 9_200_000_000_000_000_000, 150_000_000
    s = torch.cuda.Stream()
    with pc.Context(0, seg_bytes=1024) as cx:
        cx.set_stream(s.cuda_stream)
        for _ in range(2):   # the second time the tables are there and nothing else waits
            with pytest.raises(pc.PicountError) as e:
                cx.s2_hard(x, y, 5)
            assert e.value.code == -6
            assert s.query()
        assert cx.pi_count(10 ** 10) == 455052511
