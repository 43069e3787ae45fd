"""64 x 64 batches of a little more than one candidate per SM: a whole candidate
per CTA, two CTAs on some SMs, where set-up dominates (one iteration), and an
even split over one CTA per SM where iterations do.  Times against those of two
candidates on every SM (1.2 times as long at one iteration when 200 were split,
0.99 at 20 when 160 were not)."""
import pytest
import torch

from paper_2109_11920_gb300 import Geom, _lib
from paper_2109_11920_gb300 import api as boac

pytestmark = pytest.mark.gpu


def time_ms(g, B, K, dev):
    gen = torch.Generator(device=dev).manual_seed(B)
    mu = 0.15 * torch.rand(B, g.n, g.n, device=dev, generator=gen)
    S = torch.poisson(20 * torch.rand(g.n_views, g.n, device=dev, generator=gen), generator=gen) + 1
    F, L = torch.ones(B, g.n, g.n, device=dev), torch.empty(B, dtype=torch.float64, device=dev)
    ws = boac.workspace(g, B, _lib.OP_MLEM, dev)
    times = []
    for _ in range(12):
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        start.record()
        boac.boac_mlem(g, mu, S, F, K, ws=ws, L=L, check_status=False)
        end.record()
        torch.cuda.synchronize(dev)
        times.append(start.elapsed_time(end))
    return min(times[2:])


@pytest.mark.parametrize("V", [60, 90])
def test_split_where_it_pays(cuda, V):
    g = Geom.make(64, 0.4, V)
    sms = torch.cuda.get_device_properties(cuda).multi_processor_count
    assert time_ms(g, sms * 200 // 152, 1, cuda) < 1.1 * time_ms(g, 2 * sms, 1, cuda)
    assert time_ms(g, sms * 160 // 152, 20, cuda) < 0.9 * time_ms(g, 2 * sms, 20, cuda)


@pytest.mark.parametrize("V,B,K", [(60, 153, 1), (60, 200, 5), (60, 200, 20), (90, 170, 30), (90, 210, 30)])
def test_split_gives_the_same_bits(cuda, V, B, K):
    g = Geom.make(64, 0.4, V)
    gen = torch.Generator(device=cuda).manual_seed(V)
    mu = 0.15 * torch.rand(1, 64, 64, device=cuda, generator=gen)
    S = torch.poisson(20 * torch.rand(V, 64, device=cuda, generator=gen), generator=gen)
    F, L = boac.boac_mlem(g, mu.expand(B, -1, -1).contiguous(), S, torch.ones(B, 64, 64, device=cuda), K)
    assert torch.equal(F, F[:1].expand(B, 64, 64)) and torch.equal(L, L[:1].expand(B))
