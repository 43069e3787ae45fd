"""64 x 64 candidates share the SMs: two CTAs of 512 threads each, three of 256
(64 and 80 registers a thread, 57 KB of shared memory, 128 of 512 columns of
tensor memory).  The workspace has a region per resident CTA, which shows how
many the library counts on; and candidates beside each other on an SM keep
their tensor memory apart: equal candidates give equal bits."""
import ctypes

import pytest
import torch

from paper_2109_11920_gb300 import Geom, _lib
from paper_2109_11920_gb300 import api as boac

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [60, 90])
def test_ctas_counted(cuda, V):
    g = Geom.make(64, 0.4, V)
    sms = torch.cuda.get_device_properties(cuda).multi_processor_count
    size = [_lib.load().boac_workspace_bytes(ctypes.byref(g), B, _lib.OP_MLEM) for B in (sms, 2 * sms, 3 * sms)]
    per_cta = (V // 2) * (64 * 64 + 64) * 4 + 64 * 64 * 4  # its exponents and sensitivity image
    assert size[1] >= 2 * sms * per_cta and size[2] >= 3 * sms * per_cta, (size, sms * per_cta)


@pytest.mark.parametrize("V,B", [(60, 304), (90, 200), (60, 456), (90, 700)])
def test_equal_candidates_equal_bits(cuda, V, B):
    g = Geom.make(64, 0.4, V)
    gen = torch.Generator(device=cuda).manual_seed(V)
    mu = 0.15 * torch.rand(2, 64, 64, device=cuda, generator=gen)
    S = torch.poisson(20 * torch.rand(V, 64, device=cuda, generator=gen), generator=gen)
    mu = mu[torch.arange(B, device=cuda) % 2].contiguous()  # two kinds of candidate, side by side
    F, L = boac.boac_mlem(g, mu, S, torch.ones(B, 64, 64, device=cuda), 6)
    for k in range(2):
        assert torch.equal(F[k::2], F[k].expand(len(F[k::2]), 64, 64))
        assert torch.equal(L[k::2], L[k].expand(len(L[k::2])))
