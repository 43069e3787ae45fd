"""The Eq. 5 score at sinogram sizes around the switch between the clustered
and the one-CTA reduction (6112 terms, 48 896 bins): every caller of the
reduction, L prefilled with NaN, against the oracle (float64 reduction of
float32 expected counts: 1e-6 of the score, as the repository's other score
tests; boac_loglik of given counts 1e-12)."""
import ctypes
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2109_11920_gb300 import Geom, Tissue, _lib
from paper_2109_11920_gb300 import api as boac
from problems import make_problem

pytestmark = pytest.mark.gpu

# n V = 48 896 (clusters), 48 960 and 49 152 (one CTA), and the sides between
SIZES = [(128, 382), (96, 510), (96, 512), (128, 384), (256, 191), (256, 192)]


@pytest.mark.parametrize("n,V", SIZES)
def test_every_caller_scores(cuda, n, V):
    p = make_problem(n, 25.6 / n, V, 2e5, B=2, seed=V, mode=oracle.AREA)
    g = Geom.make(p.n, p.dx, V)
    B, K = 2, 1
    f32 = dict(dtype=torch.float32, device=cuda)
    mu, S, c = torch.tensor(p.mu, **f32), torch.tensor(p.S, **f32), torch.tensor(p.coefs, **f32)
    mu64 = mu.cpu().numpy().astype(np.float64)
    _, Lo, _ = oracle.mlem_batch(p.geom, mu64, p.S, K)
    q = torch.stack([torch.tensor(oracle.project(p.geom, m, np.ones((n, n))), **f32) for m in mu64])
    q64 = q.cpu().numpy().astype(np.float64)
    s64 = p.S.astype(np.float64)
    lg = math.fsum(math.lgamma(v + 1.0) for v in s64.ravel())
    Lq = [float((np.where(s64 > 0, s64 * np.log(np.where(q64[b] > 0, q64[b], 1.0)), 0.0) - q64[b]).sum() - lg)
          for b in range(B)]

    def nan():
        return torch.full((B,), float("nan"), dtype=torch.float64, device=cuda)

    def close(L, ref, tol):
        np.testing.assert_allclose(L.cpu().numpy(), ref, rtol=tol)

    lib = _lib.load()
    ref = ctypes.byref(g)
    L = nan()
    assert lib.boac_loglik(ref, boac._ptr(q), boac._ptr(S), 0, B, 1, boac._ptr(L), boac._stream(cuda)) == 0
    close(L, Lq, 1e-12)
    ones = torch.ones(B, n, n, device=cuda)
    close(boac.boac_score(g, mu, S, ones), Lq, 1e-6)
    for kind in (dict(plain=True), dict(unfused=True)) + ((dict(),) if V % 2 == 0 else ()):
        L = nan()
        boac.boac_mlem(g, mu, S, ones.clone(), K, L=L, **kind)
        close(L, Lo, 1e-6)
    if n < 256:
        m = boac.SysMat(g, cuda)
        _, L = m.mlem(m.values(mu), S, ones.clone(), K)
        close(L, Lo, 1e-6)
    t = Tissue(*p.tissue)
    L, _, _ = boac.boac_score_grad(g, t, c, S, K, ckpt_every=1, unfused=True)
    close(L, Lo, 1e-6)
