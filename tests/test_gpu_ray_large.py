"""The ray kernels on images that do not fit shared memory, around their CTAs of
32 rays and at the sides where one image fits and two do not, against the
oracle (bound as test_gpu_ray_pitch.py); and the views whose rays run along the
image's rows (60 views have them, 90 do not) do not bound a call."""
import numpy as np
import pytest
import torch

import oracle
from paper_2109_11920_gb300 import Geom
from paper_2109_11920_gb300 import api as boac
from problems import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,V", [(169, 5), (223, 4), (224, 3), (225, 8), (240, 7), (255, 6), (256, 12)])
def test_rays_through_large_images(cuda, n, V):
    dx = float(np.float32(25.6 / n))
    rng = np.random.default_rng(n)
    mu = rng.uniform(0.1, 0.2, (2, n, n)).astype(np.float32)
    F = rng.uniform(1.0, 4.0, (2, n, n)).astype(np.float32)
    y = rng.uniform(0.5, 2.0, (2, V, n)).astype(np.float32)
    g, go = Geom.make(n, dx, V), oracle.Geometry(n, dx, V)
    put = lambda a: torch.tensor(a, device=cuda)  # noqa: E731
    q = boac.boac_project(g, put(mu), put(F)).cpu().numpy()
    z = boac.boac_backproject(g, put(mu), put(y)).cpu().numpy()
    for b in range(2):
        m64 = mu[b].astype(np.float64)
        assert rel_l2(q[b], oracle.project(go, m64, F[b].astype(np.float64))) < n / 64 * 2e-6
        assert rel_l2(z[b], oracle.backproject(go, m64, y[b].astype(np.float64))) < n / 64 * 2e-6


def test_views_along_the_rows(cuda):
    def time_ms(V):
        n = 256
        g = Geom.make(n, 0.1, V)
        mu, F = torch.full((1, n, n), 0.1, device=cuda), torch.ones(1, n, n, device=cuda)
        q = torch.empty(1, V, n, device=cuda)
        times = []
        for _ in range(15):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            boac.boac_project(g, mu, F, out=q)
            end.record()
            torch.cuda.synchronize(cuda)
            times.append(start.elapsed_time(end))
        return min(times[2:])

    assert time_ms(60) < 1.15 * time_ms(90)  # 1.25 times as long with 128 rays per CTA
