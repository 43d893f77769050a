"""GPU test of the server's scratch estimate: what a query makes the library reserve on the device
stays within pc_server_footprint on both sides of the lines of the segment rules."""
import pytest

import oracle as o
import paper_1503_01839_gb300 as pc

pytestmark = pytest.mark.gpu


def x_for(cx, z):
    """The least power-of-1.01 x whose z = x / y, y as pi_count picks it, reaches z."""
    x = 1 << 20
    while x // min(cx.tuned(x)[0] * o.iroot3(x), o.isqrt(x)) < z:
        x += x // 100
    return x


@pytest.mark.parametrize("z", [4e5, 1.2e7, 4e7, 1.2e8, 2.8e8, 8e8, 2e9, 5e9])
def test_reserved_bytes_stay_within_the_estimate(z):
    import torch
    with pc.Context(0) as cx:
        x = x_for(cx, z)
        assert cx.pi_count(x) > 0   # kernels loaded
    for v, a in ((x - x // 50, 0), (x, 0), (x, 40), (x, 5000)):
        with pc.Context(0, streams=1) as cx:
            with pc.Server(cx, x_max=x, a_max=5000) as srv:
                kind = pc.PC_QUERY_PHI if a else pc.PC_QUERY_PI
                torch.cuda.synchronize()
                before = torch.cuda.mem_get_info()[0]
                srv.submit(kind, v, a)
                assert srv.poll(timeout_ms=-1)[0]["status"] == pc.PC_OK
                assert before - torch.cuda.mem_get_info()[0] <= srv.footprint(kind, v, a), (v, a)
