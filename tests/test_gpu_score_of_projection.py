"""boac_score is boac_loglik of boac_project, bit for bit, on every projector."""
import pytest
import torch

from paper_2109_11920_gb300 import Geom
from paper_2109_11920_gb300 import api as boac

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,V,B", [(64, 60, 3), (96, 90, 2), (128, 120, 70), (128, 75, 2), (100, 60, 2), (256, 36, 1)])
def test_score_is_loglik_of_projection(cuda, n, V, B):
    g = Geom.make(n, 25.6 / n, V)
    gen = torch.Generator(device=cuda).manual_seed(n + V)
    mu = 0.15 * torch.rand(B, n, n, device=cuda, generator=gen)
    F = torch.rand(B, n, n, device=cuda, generator=gen)
    S = torch.poisson(20 * torch.rand(V, n, device=cuda, generator=gen), generator=gen)
    assert torch.equal(boac.boac_score(g, mu, S, F), boac.boac_loglik(g, boac.boac_project(g, mu, F), S))
