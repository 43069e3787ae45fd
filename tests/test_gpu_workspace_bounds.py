"""A call stays inside the workspace it asked for: bytes before and after a
workspace of exactly boac_workspace_bytes keep their pattern.  Covers the
one-CTA kernel with its images in the workspace (256 x 256, view counts not
divisible by 4, more candidates than the unfused kernels take) and the paths
beside it."""
import pytest
import torch

from paper_2109_11920_gb300 import OP_MLEM, Geom
from paper_2109_11920_gb300 import api as boac

pytestmark = pytest.mark.gpu
GUARD = 4 << 20


@pytest.mark.parametrize("n,V,B", [(256, 6, 5), (256, 6, 160), (256, 8, 5), (128, 6, 20), (128, 8, 3), (96, 6, 40)])
def test_workspace_is_large_enough(cuda, n, V, B):
    g = Geom.make(n, 25.6 / n, V)
    gen = torch.Generator(device=cuda).manual_seed(n + V + B)
    mu = 0.2 * torch.rand(B, n, n, device=cuda, generator=gen)
    S = torch.poisson(20 * torch.rand(V, n, device=cuda, generator=gen), generator=gen)
    nbytes = boac.boac_workspace_bytes(g, B, OP_MLEM)
    room = torch.full((nbytes + 2 * GUARD,), 0xA5, dtype=torch.uint8, device=cuda)
    F, L = boac.boac_mlem(g, mu, S, torch.ones(B, n, n, device=cuda), 1, ws=room[GUARD:GUARD + nbytes])
    assert bool((room[:GUARD] == 0xA5).all()) and bool((room[GUARD + nbytes:] == 0xA5).all())
    assert bool(torch.isfinite(F).all()) and bool(torch.isfinite(L).all())
