"""The scatter schedule's fixed number of rounds per class (n / 2): classes
whose bank-balanced rounds exceed it put the remaining samples into empty
slots.  One MLEM iteration against the oracle shows a sample lost or listed
twice: with V views it changes at least one pixel by about 1/V of its value,
an image error of at least 1/(V n) (V <= 44, n <= 128: 1.8e-4), against
float32 rounding of sums of a few hundred terms (below 1e-5)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2109_11920_gb300 import Geom
from paper_2109_11920_gb300 import api as boac
from problems import make_problem, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,V", [(64, 4), (64, 44), (96, 4), (96, 42), (128, 4), (128, 8), (128, 20), (128, 44)])
def test_every_sample_is_scattered_once(cuda, n, V):
    p = make_problem(n, 25.6 / n, V, 2e5, B=2, seed=61)
    Fo, _, _ = oracle.mlem_batch(p.geom, p.mu, p.S, 1)
    g = Geom.make(n, p.dx, V)
    mu = torch.tensor(p.mu, dtype=torch.float32, device=cuda)
    S = torch.tensor(p.S, dtype=torch.float32, device=cuda)
    for cfg in ((0, 2, 4) if V % 4 == 0 else (1, 3, 5)):
        batch = boac.RaggedBatch([g], [0, 0], [1, 1], list(mu), [S, S], device=cuda)
        boac.boac_mlem_ragged(batch, config=[cfg])
        F = batch.F_pool.view(2, n, n).cpu().numpy()
        for b in range(2):
            assert rel_l2(F[b], Fo[b]) < 1e-5, (cfg, b)
