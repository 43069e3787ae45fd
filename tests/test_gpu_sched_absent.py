"""Geometries whose scatter schedule is too large to be kept (more than 4 MiB:
128 x 128 with 230 views, two per grid; 456 views, four per grid): the operators and the
unfused iteration scatter in lattice order, the fused kernel builds the
schedule into its workspace.  Sums are the same in either order, so the bounds
are those of the kept ones: operators 2e-6 of the oracle's in the 2-norm
(float32 sums of at most 4 V contributions), images 1e-4, scores 1e-6."""
import numpy as np
import pytest
import torch

import oracle
from paper_2109_11920_gb300 import Geom
from paper_2109_11920_gb300 import api as boac
from problems import make_problem, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [230, 456])
def test_no_kept_schedule(cuda, V):
    p = make_problem(128, 0.2, V, 2e5, B=2, seed=V)
    g = Geom.make(p.n, p.dx, V)
    mu = torch.tensor(p.mu, dtype=torch.float32, device=cuda)
    S = torch.tensor(p.S, dtype=torch.float32, device=cuda)
    z = boac.boac_backproject(g, mu, S.expand(2, -1, -1).contiguous()).cpu().numpy()
    Fo, Lo, _ = oracle.mlem_batch(p.geom, p.mu, p.S, 2)
    for unfused in (True, False):
        F, L = boac.boac_mlem(g, mu, S, torch.ones(2, p.n, p.n, device=cuda), 2, unfused=unfused)
        for b in range(2):
            assert rel_l2(F[b].cpu().numpy(), Fo[b]) < 1e-4, (unfused, b)
            assert abs(float(L[b]) - Lo[b]) < 1e-6 * abs(Lo[b]), (unfused, b)
    for b in range(2):
        zo = oracle.backproject(p.geom, np.float32(p.mu[b]).astype(np.float64), np.float32(p.S).astype(np.float64))
        assert rel_l2(z[b], zo) < 2e-6, b
