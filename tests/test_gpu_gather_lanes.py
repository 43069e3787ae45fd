"""The per-pixel back-projection with 1 to 16 lanes per pixel: batches that take
each (images and candidates enough for 243 200 threads on 152 SMs, 516 800 from
32 views on), odd sides, odd batches and fewer views than lanes.  A pixel's views are added up in order
whichever lanes take them, so a batch's images are those of one-candidate
calls, which take other lanes, bit for bit (the operators' tests compare those
with the oracle).  And one view more than a turn of 8 lanes costs a large batch
no second turn."""
import pytest
import torch

from paper_2109_11920_gb300 import Geom, _lib
from paper_2109_11920_gb300 import api as boac

pytestmark = pytest.mark.gpu


# lanes of the batch:                          1             1            2            4           8           16
@pytest.mark.parametrize("n,V,B", [(181, 3, 15), (100, 17, 49), (181, 9, 7), (101, 5, 13), (65, 21, 15), (33, 7, 3),
                                   (201, 33, 29), (181, 33, 15), (181, 32, 7), (65, 33, 31), (65, 45, 9)])
# and from 32 views on:               1              2             4            8            16
def test_lanes_give_the_same_bits(cuda, n, V, B):
    g = Geom.make(n, 25.6 / n, V)
    gen = torch.Generator(device=cuda).manual_seed(n + V)
    mu = 0.3 * torch.rand(B, n, n, device=cuda, generator=gen)
    y = 2.0 * torch.rand(B, V, n, device=cuda, generator=gen)
    z = boac.boac_backproject(g, mu, y)
    for b in (0, B // 2, B - 1):
        assert torch.equal(z[b], boac.boac_backproject(g, mu[b:b + 1].contiguous(), y[b:b + 1].contiguous())[0]), b


def test_views_beyond_a_turn(cuda):
    def time_ms(V):
        g, B, n = Geom.make(200, 0.128, V), 64, 200
        mu, y = torch.full((B, n, n), 0.1, device=cuda), torch.ones(B, V, n, device=cuda)
        out, ws = torch.empty_like(mu), boac.workspace(g, B, _lib.OP_BACKPROJECT, cuda)
        times = []
        for _ in range(10):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            boac.boac_backproject(g, mu, y, out=out, ws=ws)
            end.record()
            torch.cuda.synchronize(cuda)
            times.append(start.elapsed_time(end))
        return min(times[2:])

    assert time_ms(9) < 1.3 * time_ms(8)  # 9 / 8 in views
