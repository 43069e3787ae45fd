"""boac_project and boac_backproject on shared sample grids (64, 96, 128 images,
even view counts), at the edges of their split over CTAs and of the view
grouping, against the oracle: one grid, fewer grids than CTAs, two and four
views per grid, one candidate and more than the GPU has SMs.  Bound: float32
sums of at most 128 factors per ray (exp2 to 2^-22) and at most 4 V
contributions per pixel, below 2e-6 of the result in the 2-norm."""
import numpy as np
import pytest
import torch

import oracle
from paper_2109_11920_gb300 import Geom
from paper_2109_11920_gb300 import api as boac
from problems import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,V,B", [(64, 2, 3), (64, 4, 1), (64, 30, 160), (96, 6, 2), (96, 44, 5), (128, 4, 3),
                                   (128, 18, 1), (128, 24, 155), (128, 120, 1)])
def test_operators_on_grids(cuda, n, V, B):
    dx = float(np.float32(25.6 / n))
    rng = np.random.default_rng(n + V)
    m = min(B, 2)
    mu = rng.uniform(0.0, 0.3, (m, n, n)).astype(np.float32)
    F = rng.uniform(0.0, 4.0, (m, n, n)).astype(np.float32)
    y = rng.uniform(0.0, 2.0, (m, V, n)).astype(np.float32)
    which = np.arange(B) % m
    g, go = Geom.make(n, dx, V), oracle.Geometry(n, dx, V)
    put = lambda a: torch.tensor(a[which], device=cuda)  # noqa: E731
    q = boac.boac_project(g, put(mu), put(F)).cpu().numpy()
    z = boac.boac_backproject(g, put(mu), put(y)).cpu().numpy()
    s = boac.boac_backproject(g, put(mu), None).cpu().numpy()
    for k in range(m):
        m64 = mu[k].astype(np.float64)
        qo = oracle.project(go, m64, F[k].astype(np.float64))
        zo = oracle.backproject(go, m64, y[k].astype(np.float64))
        so = oracle.backproject(go, m64, np.ones((V, n)))
        for b in range(k, B, m):
            assert rel_l2(q[b], qo) < 2e-6 and rel_l2(z[b], zo) < 2e-6 and rel_l2(s[b], so) < 2e-6, b
