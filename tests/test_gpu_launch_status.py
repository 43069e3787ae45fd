"""A call that returns BOAC_OK has written its scores: boac_mlem_plain,
boac_sysmat_mlem and the unfused gradient return the status of every launch
they make.  The sinograms have 48 960 to 49 152 bins, where the clustered
score kernel's shared memory comes to the 48 KB that a launch may ask for
without an attribute."""
import ctypes

import pytest
import torch

from paper_2109_11920_gb300 import Geom, Tissue, _lib
from paper_2109_11920_gb300 import api as boac

pytestmark = pytest.mark.gpu


def p(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("n,V", [(96, 510), (96, 512), (256, 192)])
@pytest.mark.parametrize("call", ["plain", "sysmat", "grad"])
def test_ok_means_scored(cuda, n, V, call):
    if call == "sysmat" and n == 256:
        pytest.skip("25 M entries: the 96 x 96 cases cover it")
    g = Geom.make(n, 25.6 / n, V)
    lib, ref = _lib.load(), ctypes.byref(g)
    gen = torch.Generator(device=cuda).manual_seed(V)
    B = 2
    mu = 0.15 * torch.rand(B, n, n, device=cuda, generator=gen)
    S = torch.poisson(20 * torch.rand(V, n, device=cuda, generator=gen), generator=gen)
    F = torch.ones(B, n, n, device=cuda)
    L = torch.full((B,), float("nan"), dtype=torch.float64, device=cuda)
    st = boac._stream(cuda)
    if call == "plain":
        ws = boac.workspace(g, B, _lib.OP_MLEM_PLAIN, cuda)
        status = lib.boac_mlem_plain(ref, p(mu), p(S), 0, p(F), 1, B, p(L), 1, p(ws), ws.numel(), st)
    elif call == "sysmat":
        m = boac.SysMat(g, cuda)
        vals = m.values(mu)
        ws = torch.empty(lib.boac_sysmat_mlem_workspace_bytes(m._h, B), dtype=torch.uint8, device=cuda)
        status = lib.boac_sysmat_mlem(m._h, p(vals), p(S), 0, p(F), 1, B, p(L), 1, p(ws), ws.numel(), st)
    else:
        t = Tissue(0.15, 0.25, 0.6)
        c = torch.tensor([[8.0, 0.3, -0.6, 0.2, -0.1, 0.05]] * B, device=cuda)
        dc = torch.empty(B, 6, dtype=torch.float64, device=cuda)
        ws = torch.empty(lib.boac_score_grad_workspace_bytes(ref, B, 1, 1), dtype=torch.uint8, device=cuda)
        status = lib.boac_score_grad_unfused(ref, ctypes.byref(t), p(c), p(S), 0, 1, 1, B, 1, p(L), p(dc), None,
                                             p(ws), ws.numel(), st)
    torch.cuda.synchronize(cuda)
    assert status != _lib.BOAC_OK or bool(torch.isfinite(L).all())
