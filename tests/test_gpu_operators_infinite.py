"""boac_project and boac_backproject through pixels of infinite mu: the bilinear
read of one gives infinity or, where a difference of infinities is taken, not a
number; a factor behind infinity is 0.  Reference: the same formulas in float64,
which meet the same infinities.  Finite values within 1e-5 (float32 sums of at
most 128 factors)."""
import numpy as np
import pytest
import torch

from paper_2109_11920_gb300 import Geom
from paper_2109_11920_gb300 import api as boac

pytestmark = pytest.mark.gpu


def reference(n, V, dx, mu, F):
    c = 0.5 * (n - 1)
    pad = lambda a: np.pad(a.astype(np.float64), 1)  # noqa: E731
    k, b = np.meshgrid(np.arange(n) - c, np.arange(n) - c, indexing="ij")
    q = np.empty((V, n))
    for v in range(V):
        quadrant, rem = divmod(4 * v, V)
        th = 0.5 * np.pi * rem / V
        cs, sn = np.float32(np.cos(th)), np.float32(np.sin(th))
        cs, sn = [(cs, sn), (-sn, cs), (-cs, -sn), (sn, -cs)][quadrant]
        u, w = c + b * float(cs) - k * float(sn), c + b * float(sn) + k * float(cs)
        inside = (u > -1) & (u < n) & (w > -1) & (w < n)
        uu, ww = np.where(inside, u, 0.0), np.where(inside, w, 0.0)
        j, i = np.floor(uu).astype(int), np.floor(ww).astype(int)
        au, aw = uu - j, ww - i

        def sample(a):
            p = pad(a)
            v00, v01, v10, v11 = p[i + 1, j + 1], p[i + 1, j + 2], p[i + 2, j + 1], p[i + 2, j + 2]
            top, bot = v00 + au * (v01 - v00), v10 + au * (v11 - v10)
            return np.where(inside, top + aw * (bot - top), 0.0)

        m, f = sample(mu), sample(F)
        behind = np.zeros_like(m)
        behind[:-1] = np.cumsum(m[::-1], axis=0)[::-1][1:]
        q[v] = dx * (np.exp(-dx * (0.5 * m + behind)) * f).sum(0)
    return q


@pytest.mark.filterwarnings("ignore::RuntimeWarning")
@pytest.mark.parametrize("n,V", [(64, 14), (96, 28), (128, 10)])
def test_infinite_pixels(cuda, n, V):
    dx = float(np.float32(25.6 / n))
    rng = np.random.default_rng(n)
    mu = rng.uniform(0.05, 0.15, (n, n)).astype(np.float32)
    mu[n // 3, n // 2] = np.inf
    mu[n // 2:n // 2 + 3, n // 4:n // 4 + 5] = np.inf
    F = rng.uniform(1.0, 4.0, (n, n)).astype(np.float32)
    g = Geom.make(n, dx, V)
    q = boac.boac_project(g, torch.tensor(mu[None], device=cuda), torch.tensor(F[None], device=cuda))[0].cpu().numpy()
    want = reference(n, V, dx, mu, F)
    generic = np.arange(V) % (V // 2) != 0  # at 0 and 180 degrees an au of rounding error decides
    assert (np.isnan(q) == np.isnan(want))[generic].all()
    assert np.isfinite(want[generic]).mean() > 0.5 and np.isnan(want[generic]).any()
    ok = np.isfinite(want) & generic[:, None]
    np.testing.assert_allclose(q[ok], want[ok], rtol=1e-5)
