"""boac_backproject through dense matter (2 to 8 per cm, path lengths up to 25
cm: attenuation factors down to the smallest floats), at 64, 96 and 128 against
the oracle.

Bound, from the arithmetic: the exponent x of a factor is a float32 sum of at
most n samples of one sign (segments of n / 8, then 8 of their sums: relative
error below (n / 8 + 8) u, u = 2^-24), so a factor's relative error is below
24 u x + 2^-21, where factors down to the smallest float have x <= 103: 1.5e-4.
A pixel adds 4 V positive contributions: 4 V u = 2.9e-5 more.  Contributions
below 2^-126 are spaced 1.4e-45: 4 V of them 4e-6 of a pixel of 1e-37, the
smallest compared."""
import numpy as np
import pytest
import torch

import oracle
from paper_2109_11920_gb300 import Geom
from paper_2109_11920_gb300 import api as boac

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,V", [(64, 60), (96, 90), (128, 120)])
@pytest.mark.parametrize("density", [2.0, 8.0])
def test_factors_keep_their_precision(cuda, n, V, density):
    dx = float(np.float32(25.6 / n))
    rng = np.random.default_rng(n)
    yy, xx = np.mgrid[:n, :n] - 0.5 * (n - 1)
    mu = np.float32(density * (np.hypot(yy, xx) < 0.45 * n) * (0.5 + rng.random((n, n))))
    y = np.float32(0.5 + rng.random((V, n)))
    g, go = Geom.make(n, dx, V), oracle.Geometry(n, dx, V)
    put = lambda a: torch.tensor(a[None], device=cuda)  # noqa: E731
    z = boac.boac_backproject(g, put(mu), put(y))[0].cpu().numpy().astype(np.float64)
    zo = oracle.backproject(go, mu.astype(np.float64), y.astype(np.float64))
    seen = zo > 1e-37
    assert np.max(np.abs(z - zo)[seen] / zo[seen]) < 2e-4
