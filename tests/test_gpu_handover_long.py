"""The hand-over wait allows for the time that a cut candidate's first part
takes: the last CTA of the even split may have nothing but a second part, and
waits for all of the first part's iterations, however long they are.  With a
limit of 200 000 cycles (0.1 ms; an iteration takes 0.1 to 1 ms) no candidate
is given up, in uniform and in ragged batches, and the results are the same
bits as with the default limit."""
import pytest
import torch

from paper_2109_11920_gb300 import Geom
from paper_2109_11920_gb300 import api as boac

pytestmark = pytest.mark.gpu

# (side, views, candidates, iterations) of each class, launch configurations
BATCHES = [
    ([(128, 120, 153, 60)], [4]),                                          # last CTA of 151: 30 of 61 units
    ([(256, 60, 33, 12)], None),                                           # clusters
    ([(64, 60, 90, 165), (128, 120, 100, 60)], [4, 4]),                    # classes that share the SMs
    ([(64, 60, 62, 165), (64, 120, 20, 84), (128, 120, 100, 60)], [4, 4, 4]),
]


@pytest.mark.parametrize("parts,config", BATCHES)
def test_long_first_part_is_no_timeout(cuda, parts, config):
    gen = torch.Generator(device=cuda).manual_seed(len(parts))
    classes, cls, ks, mu, S = [], [], [], [], []
    for i, (n, V, B, K) in enumerate(parts):
        classes.append(Geom.make(n, 25.6 / n, V))
        s = torch.poisson(20 * torch.rand(V, n, device=cuda, generator=gen), generator=gen)
        for _ in range(B):
            cls.append(i)
            ks.append(K)
            mu.append(0.15 * torch.rand(n, n, device=cuda, generator=gen))
            S.append(s)
    out = []
    for limit in (0, 200_000):  # 0: the default
        b = boac.RaggedBatch(classes, cls, ks, mu, S, device=cuda)
        torch.cuda.synchronize(cuda)
        old = boac.boac_set_wait_cycles(limit)
        try:
            out.append((boac.boac_mlem_ragged(b, config=config), b.F_pool))  # raises where a wait gave up
        finally:
            boac.boac_set_wait_cycles(old)
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


def test_largest_limit(cuda):
    """The largest limit that can be set never runs out."""
    g, B, K = Geom.make(64, 0.4, 60), 229, 7
    mu = torch.full((64, 64), 0.1, device=cuda)
    S = torch.ones(60, 64, device=cuda)
    b = boac.RaggedBatch([g], [0] * B, [K + i % 3 for i in range(B)], [mu] * B, [S] * B, device=cuda)
    old = boac.boac_set_wait_cycles(2**63 - 1)
    try:
        L = boac.boac_mlem_ragged(b, config=[2])  # raises where a wait gave up
    finally:
        boac.boac_set_wait_cycles(old)
    assert bool(torch.isfinite(L).all())
