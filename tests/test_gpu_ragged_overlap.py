"""The classes of a ragged batch run at once (programmatic dependent launches)
and share the SMs; each class's images and scores are the bits it gives in a
call of its own, whatever runs beside it, on a captured graph too, and work
enqueued after the call sees all of them."""
import pytest
import torch

from paper_2109_11920_gb300 import Geom
from paper_2109_11920_gb300 import api as boac

pytestmark = pytest.mark.gpu


def random_class(n, V, count, k_hi, gen, dev):
    mu = 0.15 * torch.rand(count, n, n, device=dev, generator=gen)
    S = torch.poisson(20 * torch.rand(count, V, n, device=dev, generator=gen), generator=gen)
    K = torch.randint(0, k_hi + 1, (count,), device=dev, generator=gen).tolist()
    return Geom.make(n, 25.6 / n, V), list(mu), list(S), K


@pytest.mark.parametrize("sizes", [
    [(64, 60, 5, 9), (96, 90, 7, 6)],
    [(128, 24, 90, 5), (96, 18, 60, 9), (64, 20, 40, 3)],        # fits together
    [(128, 24, 200, 4), (96, 18, 170, 5), (64, 12, 500, 4)],     # has to share
    [(256, 24, 3, 2), (128, 8, 20, 3), (256, 6, 4, 1), (64, 8, 1, 7)],
])
def test_classes_together_equal_classes_alone(cuda, sizes):
    gen = torch.Generator(device=cuda).manual_seed(len(sizes))
    classes = [random_class(n, V, count, k, gen, cuda) for n, V, count, k in sizes]
    cls, K, mu, S = [], [], [], []
    for j in range(max(c[2] for c in sizes)):      # interleave the classes
        for i, (_, m, s, k) in enumerate(classes):
            if j < len(m):
                cls.append(i), K.append(k[j]), mu.append(m[j]), S.append(s[j])
    batch = boac.RaggedBatch([c[0] for c in classes], cls, K, mu, S, device=cuda)
    batch.prepare()
    batch.run()
    F, L = batch.F_pool.clone(), batch.L.clone()   # enqueued behind the run
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        batch.run()
    batch.F_pool.fill_(1.0)
    graph.replay()
    assert torch.equal(batch.F_pool, F) and torch.equal(batch.L, L)
    assert batch.status() == 0
    for i, (g, m, s, k) in enumerate(classes):
        alone = boac.RaggedBatch([g], [0] * len(m), k, m, s, device=cuda)
        La = boac.boac_mlem_ragged(alone)
        members = [b for b, c in enumerate(cls) if c == i]
        assert torch.equal(L[members], La)
        nn = g.n * g.n
        for j, b in enumerate(members):
            o = batch.cands[b].F_off
            assert torch.equal(F[o:o + nn], alone.F_pool[j * nn:(j + 1) * nn]), (i, j)
