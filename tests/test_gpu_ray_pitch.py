"""The ray kernels' image pitch in shared memory: sides around the multiples of
32 (where n + 1 is a bad pitch) and at the largest that fit with one and two
images, where the padding right of the image lies in a column of its own; and
lines at 45 degrees cost a multiple of 32 no more than another side.  Images
that are not 0 at the border, so that a sample past the edge shows.  Reference:
the oracle; bound as test_gpu_operators.py's scaled to the longest ray here, 2
(n / 128) 2e-6 in the 2-norm, since a ray's sums grow with n."""
import numpy as np
import pytest
import torch

import oracle
from paper_2109_11920_gb300 import Geom
from paper_2109_11920_gb300 import api as boac
from problems import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 30, 31, 32, 33, 64, 95, 96, 127, 128, 159, 160, 166, 167, 168, 236, 237, 238, 239])
def test_rays_at_every_pitch(cuda, n):
    V = 7  # odd: the ray kernels
    dx = float(np.float32(25.6 / n))
    rng = np.random.default_rng(n)
    mu = rng.uniform(0.1, 0.2, (2, n, n)).astype(np.float32)
    F = rng.uniform(1.0, 4.0, (2, n, n)).astype(np.float32)
    y = rng.uniform(0.5, 2.0, (2, V, n)).astype(np.float32)
    g, go = Geom.make(n, dx, V), oracle.Geometry(n, dx, V)
    put = lambda a: torch.tensor(a, device=cuda)  # noqa: E731
    q = boac.boac_project(g, put(mu), put(F)).cpu().numpy()
    z = boac.boac_backproject(g, put(mu), put(y)).cpu().numpy()
    bound = max(1.0, n / 64) * 2e-6
    for b in range(2):
        m64 = mu[b].astype(np.float64)
        assert rel_l2(q[b], oracle.project(go, m64, F[b].astype(np.float64))) < bound
        assert rel_l2(z[b], oracle.backproject(go, m64, y[b].astype(np.float64))) < bound


@pytest.mark.parametrize("n", [96, 128, 160])
def test_multiples_of_32_are_no_slower(cuda, n):
    def time_ms(n):
        V, B = 75, 16
        g = Geom.make(n, 25.6 / n, V)
        mu, F = torch.full((B, n, n), 0.1, device=cuda), torch.ones(B, n, n, device=cuda)
        q = torch.empty(B, V, n, device=cuda)
        times = []
        for _ in range(12):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            boac.boac_project(g, mu, F, out=q)
            end.record()
            torch.cuda.synchronize(cuda)
            times.append(start.elapsed_time(end))
        return min(times[2:])

    assert time_ms(n) < 1.1 * time_ms(n + 6)  # n + 6: pitch 7 (mod 32), a warp more per view
