"""The SMs a ragged batch's classes get: a class that runs the one-CTA kernel at
256 x 256 (its images in global memory, some ten times the time of the others
per sample) is given enough of them beside another class, so that the batch
takes no longer than its classes one after the other (5 % for the clock)."""
import pytest
import torch

from paper_2109_11920_gb300 import Geom
from paper_2109_11920_gb300 import api as boac

pytestmark = pytest.mark.gpu


def batch(parts, dev):
    gen = torch.Generator(device=dev).manual_seed(7)
    classes, cls, ks, mu, S = [], [], [], [], []
    for i, (n, V, B, K) in enumerate(parts):
        classes.append(Geom.make(n, 25.6 / n, V))
        s = torch.poisson(20 * torch.rand(V, n, device=dev, generator=gen), generator=gen)
        for _ in range(B):
            cls.append(i)
            ks.append(K)
            mu.append(0.15 * torch.rand(n, n, device=dev, generator=gen))
            S.append(s)
    return boac.RaggedBatch(classes, cls, ks, mu, S, device=dev)


def time_ms(parts, dev):
    b = batch(parts, dev)
    b.prepare(None)
    times = []
    for _ in range(4):
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        start.record()
        b.run(True)
        end.record()
        torch.cuda.synchronize(dev)
        times.append(start.elapsed_time(end))
    return min(times[1:])


@pytest.mark.parametrize("parts", [[(256, 90, 64, 6), (128, 120, 152, 20)], [(256, 90, 100, 4), (96, 60, 300, 20)]])
def test_not_slower_than_one_after_the_other(cuda, parts):
    apart = sum(time_ms([p], cuda) for p in parts)
    assert time_ms(parts, cuda) < 1.05 * apart
