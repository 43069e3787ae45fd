"""The calls a user of this library makes, as measurable cases.

A case is one pass through the public entry points at one size: candidate
evaluation inside a Bayesian optimisation (one candidate, a cycle's batch, the
full benchmark batch, ragged batches), 256 x 256 slices, the score gradient,
the bare operators, image sides without a fused kernel, and the explicit
system matrix.  Inputs are drawn from a seed: head phantoms with hot ellipses,
a Poisson sinogram of their attenuated projection, and candidate boundaries
around the true one.  ``exact`` recomputes a case in float64 with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2109_11920_gb300 import Geom, Tissue, api

FIELD_CM = 25.6                     # field of view: n pixels of FIELD_CM / n
TISSUE = (0.15, 0.25, 0.6)          # mu_b, mu_c (1/cm), cranium thickness (cm)
C_TRUE = (8.0, 0.3, -0.6, 0.2, -0.1, 0.05)
RAGGED = ((64, 60), (96, 90), (128, 120))   # (side, views) of a ragged batch
RAGGED_MIX = (1, 1, 2)
MOST_SAMPLES = 2.6e10               # ray samples x iterations of the largest case


def listed():
    return [
        # One proposal of a sequential optimisation at 64 x 64: the smallest
        # call, bound by latency.  Rasterised and scored without the constant
        # ln S! term, as the optimiser calls it; so are the next three.
        dict(name="one_64", kind="bo", n=64, V=60, B=1, K=20),
        # One cycle of the optimiser at its default of 32 proposals.
        dict(name="cycle_128", kind="bo", n=128, V=120, B=32, K=20),
        # A cycle's few proposals on a scanner whose views are not a multiple
        # of four.
        dict(name="cycle_96_v90", kind="bo", n=96, V=90, B=8, K=20),
        # The image-quality study: 72 views, the optimiser's initial set.
        dict(name="study_72_views", kind="bo", n=128, V=72, B=64, K=50),
        # The benchmark: 256 candidates, replayed from a captured graph, with
        # the full score.
        dict(name="batch_256", kind="evaluate", n=128, V=120, B=256, K=50),
        # Candidates of three image sizes and mixed iteration counts at once.
        dict(name="ragged_256", kind="ragged", B=256, k_lo=20, k_hi=80),
        # Fine slices: two slices of 16 candidates, a sinogram per candidate.
        dict(name="slices_256", kind="slices", n=256, V=180, B=32, K=20),
        # Gradients of a batch of candidates through 10 iterations.
        dict(name="grad_64", kind="grad", n=128, V=120, B=64, K=10, ckpt=2, params=False),
        # A polishing step of the incumbent: one gradient of all nine parameters.
        dict(name="polish_1", kind="grad", n=128, V=120, B=1, K=20, ckpt=2, params=True),
        # The bare operators: simulate sinograms of images, back-project
        # sinograms.
        dict(name="operators_64", kind="operators", n=128, V=120, B=64),
        # An image side and view count without a fused kernel, scored as the
        # optimiser does.
        dict(name="odd_100_v75", kind="unfused", n=100, V=75, B=4, K=10),
        # The system matrix written out, for comparison with the above.
        dict(name="matrix_32", kind="sysmat", n=128, V=120, B=32, K=20),
    ]


def draw(rng):
    def log_int(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    kind = rng.choice(("bo", "bo", "bo", "bo", "evaluate", "ragged", "slices", "grad", "grad", "operators",
                       "unfused", "sysmat"))
    if kind == "ragged":
        lo = rng.randint(5, 40)
        return dict(kind=kind, B=log_int(8, 256), k_lo=lo, k_hi=lo + rng.randint(0, 40))
    if kind == "operators":
        case = dict(kind=kind, n=rng.choice((64, 96, 128, rng.randint(40, 160))), V=rng.randint(12, 120), B=log_int(1, 64))
    elif kind == "unfused":
        case = dict(kind=kind, n=rng.randint(24, 180), V=rng.randint(9, 120), B=log_int(1, 8), K=log_int(2, 20))
    elif kind == "grad":
        case = dict(kind=kind, n=rng.choice((64, 96, 128)), V=4 * rng.randint(6, 30), B=log_int(1, 64),
                    K=log_int(3, 20), ckpt=rng.randint(1, 5), params=rng.random() < 0.5)
    elif kind == "sysmat":
        case = dict(kind=kind, n=rng.choice((64, 96, 128)), V=rng.randint(16, 120), B=log_int(3, 40), K=log_int(4, 20))
    elif kind == "slices":
        views = 4 * rng.randint(15, 45) if rng.random() < 0.8 else 2 * rng.randint(30, 90)
        case = dict(kind=kind, n=256, V=views, B=log_int(2, 40), K=log_int(4, 20))
    elif kind == "evaluate":
        case = dict(kind=kind, n=rng.choice((64, 96, 128)), V=4 * rng.randint(6, 30), B=log_int(16, 256),
                    K=log_int(5, 60))
    else:
        views = 4 * rng.randint(6, 30) if rng.random() < 0.7 else 2 * rng.randint(12, 60)
        case = dict(kind=kind, n=rng.choice((64, 96, 128)), V=views, B=log_int(1, 256), K=log_int(5, 60))
    while samples(case) > MOST_SAMPLES:
        case["B"] = case["B"] // 2
    return case


def samples(case):
    """Ray samples x iterations (a gradient counts four per iteration, the
    bare operators one)."""
    if case["kind"] == "ragged":
        K = 0.5 * (case["k_lo"] + case["k_hi"])
        return case["B"] * K * sum(m * n * n * V for m, (n, V) in zip(RAGGED_MIX, RAGGED)) / sum(RAGGED_MIX)
    per = {"grad": 4}.get(case["kind"], 1) * case.get("K", 1)
    return case["B"] * per * case["V"] * case["n"] ** 2


def work(case):
    # 20 operations per ray sample and iteration: the bilinear read (8), the
    # attenuated sum (2), the back-projection weight (2), its transpose (8).
    flops = 20 * samples(case)
    if case["kind"] == "ragged":
        per = sum(m * 4 * (3 * n * n + n * V) for m, (n, V) in zip(RAGGED_MIX, RAGGED)) / sum(RAGGED_MIX)
        return dict(bytes=case["B"] * per, flops=flops)
    n, V, B = case["n"], case["V"], case["B"]
    image, sino = 4 * n * n, 4 * n * V
    if case["kind"] in ("bo", "evaluate"):      # coefficients and a sinogram in, maps and images out
        moved = 24 * B + sino + 2 * B * image
    elif case["kind"] == "grad":                # coefficients and a sinogram in, images and gradients out
        moved = 100 * B + sino + B * image
    elif case["kind"] == "slices":              # maps and sinograms in, images in and out
        moved = B * (3 * image + sino)
    elif case["kind"] == "operators":           # maps and images in, sinograms out, and back
        moved = B * (4 * image + 2 * sino)
    else:                                       # maps and a sinogram in, images in and out
        moved = 3 * B * image + sino
    return dict(bytes=moved, flops=flops)


# ---------------------------------------------------------------- inputs
def _f32(x):
    return float(np.float32(x))


def _tissue():
    return tuple(_f32(t) for t in TISSUE)


def _pixel(n):
    return _f32(FIELD_CM / n)


class _Rays:
    """The ray samples of one geometry in float64: the bilinear sampling
    matrix (rows: view, sample, bin; columns: pixels) and its transpose."""

    def __init__(self, n, V, device="cuda"):
        self.n, self.V, self.dx = n, V, _pixel(n)
        f64 = dict(dtype=torch.float64, device=device)
        c = 0.5 * (n - 1)
        phi = 2 * math.pi * torch.arange(V, **f64) / V
        cs, sn = torch.cos(phi)[:, None, None], torch.sin(phi)[:, None, None]
        t = (torch.arange(n, **f64) - c)[None, :, None]
        s = (torch.arange(n, **f64) - c)[None, None, :]
        u = (c + s * cs - t * sn).reshape(-1)
        w = (c + s * sn + t * cs).reshape(-1)
        j0, i0 = torch.floor(u), torch.floor(w)
        au, aw = u - j0, w - i0
        col, val = [], []
        for di in (0, 1):
            for dj in (0, 1):
                i, j = i0.long() + di, j0.long() + dj
                wt = (aw if di else 1 - aw) * (au if dj else 1 - au)
                ok = (i >= 0) & (i < n) & (j >= 0) & (j < n)
                col.append(torch.where(ok, i * n + j, 0))
                val.append(torch.where(ok, wt, 0.0))
        rows = V * n * n
        col, val = torch.stack(col, 1).reshape(-1), torch.stack(val, 1).reshape(-1)
        ptr = torch.arange(rows + 1, device=device, dtype=torch.int64) * 4
        self.B = torch.sparse_csr_tensor(ptr, col, val, (rows, n * n))
        order = torch.argsort(col, stable=True)
        ptr_t = torch.zeros(n * n + 1, device=device, dtype=torch.int64)
        ptr_t[1:] = torch.cumsum(torch.bincount(col, minlength=n * n), 0)
        self.Bt = torch.sparse_csr_tensor(ptr_t, order // 4, val[order], (n * n, rows))
        self.shape = (V, n, n)

    def factors(self, mu):
        """Attenuation factors of every sample: mu [n n, B] -> [V, n, n, B]."""
        m = _Apply.apply(mu, self.B, self.Bt).view(*self.shape, -1)
        after = torch.flip(torch.cumsum(torch.flip(m, (1,)), 1), (1,)) - m
        return torch.exp(-self.dx * (0.5 * m + after))

    def project(self, a, F):
        """[V, n, B] from F [n n, B]."""
        f = _Apply.apply(F, self.B, self.Bt).view(*self.shape, -1)
        return self.dx * (a * f).sum(1)

    def backproject(self, a, y):
        """[n n, B] from y [V, n, B]."""
        g = self.dx * a * y[:, None]
        return _Apply.apply(g.reshape(-1, g.shape[-1]), self.Bt, self.B)


class _Apply(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x, A, At):
        ctx.At = At
        return A @ x.contiguous()

    @staticmethod
    def backward(ctx, g):
        return ctx.At @ g.contiguous(), None, None


def _pixels(n, device="cuda"):
    x = (torch.arange(n, dtype=torch.float64, device=device) - 0.5 * (n - 1)) * _pixel(n)
    return x[None, :].expand(n, n), x[:, None].expand(n, n)


def _maps(n, coef, tissue, area):
    """Attenuation maps [B, n, n] in float64 of boundaries coef [B, 6];
    tissue: three tensors that broadcast with [B, 1, 1]."""
    x, y = _pixels(n, coef.device)
    r = torch.sqrt(x * x + y * y)
    z = torch.where(r > 0, x / torch.where(r > 0, r, 1.0), 1.0)
    P = [torch.ones_like(z), z]
    for k in range(1, 5):
        P.append(((2 * k + 1) * z * P[k] - k * P[k - 1]) / (k + 1))
    R = sum(coef[:, k, None, None] * P[k] for k in range(6)).clamp(min=0.0)
    mu_b, mu_c, dR = tissue
    if not area:
        return torch.where(r < R, mu_b, torch.where(r < R + dR, mu_c, 0.0))
    dx = _pixel(n)
    f_in = (0.5 + (R - r) / dx).clamp(0.0, 1.0)
    f_out = (0.5 + (R + dR - r) / dx).clamp(0.0, 1.0)
    return mu_b * f_in + mu_c * (f_out - f_in)


def _constant_tissue(device="cuda"):
    return tuple(torch.tensor(t, dtype=torch.float64, device=device) for t in _tissue())


def _candidates(rng, B, c_true):
    c = np.asarray(c_true)
    return (c + rng.normal(size=(B, 6)) * (0.15 * np.abs(c) + 0.05)).astype(np.float32)


def _heads(rng, count):
    """True boundaries of `count` heads."""
    c = np.tile(np.asarray(C_TRUE), (count, 1))
    if count > 1:
        c[:, 0] = rng.uniform(6.0, 9.0, count)
        c[:, 1:] *= rng.uniform(0.5, 1.5, (count, 5))
    return c


def _sinograms(rng, rays, heads, counts):
    """(maps, activities, sinograms) of the heads' phantoms: brain activity 1
    with four ellipses at 4, Poisson counts of the attenuated projection."""
    n, device = rays.n, rays.B.device
    maps = _maps(n, torch.tensor(heads, device=device), _constant_tissue(device), False)
    brain = maps == _constant_tissue(device)[0]
    x, y = _pixels(n, device)
    F = brain.double()
    for _ in range(4):
        rad = 0.5 * heads[:, 0] * np.sqrt(rng.uniform(size=len(heads)))
        ang = rng.uniform(0, 2 * math.pi, len(heads))
        a, b = rng.uniform(0.5, 2.0, (2, len(heads)))
        th = rng.uniform(0, math.pi, len(heads))
        cx, cy, a, b, ct, st = (torch.tensor(v, device=device)[:, None, None] for v in
                                (rad * np.cos(ang), rad * np.sin(ang), a, b, np.cos(th), np.sin(th)))
        inside = (((x - cx) * ct + (y - cy) * st) / a) ** 2 + ((-(x - cx) * st + (y - cy) * ct) / b) ** 2 <= 1
        F = torch.where(inside & brain, 4.0, F)
    q = []
    for part in torch.split(torch.arange(len(heads)), 32):
        a = rays.factors(maps[part].reshape(len(part), -1).T)
        q.append(rays.project(a, F[part].reshape(len(part), -1).T).permute(2, 0, 1))
    q = torch.cat(q)
    lam = (q * (counts / q.sum((1, 2), keepdim=True))).cpu().numpy()
    S = torch.tensor(rng.poisson(lam).astype(np.float32), device=device)
    return maps, F, S


def _counts(n):
    return {64: 2e5, 96: 2e5, 128: 1e6, 256: 5e6}.get(n, 3e5)


_RAYS = {}


def _rays(n, V):
    """The last geometries' rays (input generation and `exact` only)."""
    if (n, V) not in _RAYS:
        while len(_RAYS) >= 3:
            _RAYS.pop(next(iter(_RAYS)))
        _RAYS[n, V] = _Rays(n, V)
    return _RAYS[n, V]


def _inputs(case, seed):
    """Inputs of a case from its seed: dict of device tensors."""
    rng = np.random.default_rng(seed)
    kind, B = case["kind"], case["B"]
    if kind == "ragged":
        cls = np.concatenate([np.full(B * m // sum(RAGGED_MIX), i) for i, m in enumerate(RAGGED_MIX)])
        cls = np.concatenate([cls, np.full(B - cls.size, len(RAGGED_MIX) - 1)])
        rng.shuffle(cls)
        K = rng.integers(case["k_lo"], case["k_hi"] + 1, B)
        mu, S = [None] * B, [None] * B
        for i, (n, V) in enumerate(RAGGED):
            members = np.flatnonzero(cls == i)
            if not members.size:
                continue
            heads = _heads(rng, len(members))
            _, _, Si = _sinograms(rng, _rays(n, V), heads, _counts(n))
            c = np.concatenate([_candidates(rng, 1, h) for h in heads])
            mi = _maps(n, torch.tensor(c, device="cuda").double(), _constant_tissue(), False).float()
            for j, b in enumerate(members):
                mu[b], S[b] = mi[j], Si[j]
        return dict(cls=cls, K=K, mu=mu, S=S)
    n, V = case["n"], case["V"]
    heads = _heads(rng, 2 if kind == "slices" else 1)
    maps, F, S = _sinograms(rng, _rays(n, V), heads, _counts(n))
    which = np.arange(B) * len(heads) // B
    c = np.concatenate([_candidates(rng, 1, heads[i]) for i in which])
    got = dict(c=torch.tensor(c, device="cuda"), S=S[0] if kind != "slices" else S[torch.tensor(which)].contiguous())
    if kind == "grad" and case["params"]:
        t = np.asarray(TISSUE) * rng.uniform(0.8, 1.2, (B, 3))
        got["c"] = torch.tensor(np.concatenate([c, t], 1).astype(np.float32), device="cuda")
    elif kind not in ("bo", "evaluate", "grad"):
        got["mu"] = _maps(n, got["c"].double(), _constant_tissue(), False).float()
    if kind == "operators":
        # images in counts: the true activity, each with its own noise
        noise = torch.tensor(rng.uniform(0.5, 1.5, (B, n, n)), device="cuda")
        q = _rays(n, V).project(_rays(n, V).factors(maps[0].reshape(-1, 1)), F[0].reshape(-1, 1))
        got["F"] = (F[0] * (_counts(n) / q.sum()) * noise).float()
        got["y"] = torch.tensor(rng.uniform(0.0, 2.0, (B, V, n)).astype(np.float32), device="cuda")
    return got


# ------------------------------------------------------------------ a pass
def prepare(case, seed):
    s = dict(case, **_inputs(case, seed))
    if case["kind"] == "ragged":
        geoms = [Geom.make(n, _pixel(n), V) for n, V in RAGGED]
        s["batch"] = api.RaggedBatch(geoms, [int(i) for i in s["cls"]], [int(k) for k in s["K"]], s["mu"], s["S"])
        return s
    s["g"], s["t"] = Geom.make(case["n"], _pixel(case["n"]), case["V"]), Tissue(*_tissue())
    if case["kind"] == "evaluate":
        s["evaluator"] = api.BatchedEvaluator(s["g"], s["t"], s["S"], case["B"], case["K"])
    if case["kind"] == "sysmat":
        s["matrix"] = api.SysMat(s["g"], "cuda")
    return s


def run(s):
    kind = s["kind"]
    if kind == "ragged":
        batch = s["batch"]
        batch.F_pool.fill_(1.0)
        L = api.boac_mlem_ragged(batch)
        return dict(F=batch.F_pool, L=L)
    g, B, n = s["g"], s["B"], s["n"]
    if kind == "evaluate":
        ev = s["evaluator"]
        L = ev.evaluate(s["c"])
        return dict(F=ev.F, L=L, mu=ev.mu)
    if kind == "bo":
        mu = api.boac_rasterize_mu(g, s["t"], s["c"])
        F, L = api.boac_mlem(g, mu, s["S"], torch.ones(B, n, n, device="cuda"), s["K"], include_lgamma=False)
        return dict(F=F, L=L, mu=mu)
    if kind == "grad":
        if s["params"]:
            L, grad, F = api.boac_score_grad_params(g, s["c"], s["S"], s["K"], s["ckpt"], want_image=True)
        else:
            L, grad, F = api.boac_score_grad(g, s["t"], s["c"], s["S"], s["K"], s["ckpt"], want_image=True)
        return dict(L=L, grad=grad, F=F)
    if kind == "operators":
        q = api.boac_project(g, s["mu"], s["F"])
        z = api.boac_backproject(g, s["mu"], s["y"])
        return dict(q=q, z=z)
    F = torch.ones(B, n, n, device="cuda")
    if kind == "sysmat":
        F, L = s["matrix"].mlem(s["matrix"].values(s["mu"]), s["S"], F, s["K"])
    elif kind == "unfused":
        F, L = api.boac_mlem(g, s["mu"], s["S"], F, s["K"], include_lgamma=False, unfused=True)
    else:
        F, L = api.boac_mlem(g, s["mu"], s["S"], F, s["K"])
    return dict(F=F, L=L)


# ------------------------------------------------------- 64-bit reference
def _score64(S, q, lgamma):
    """[B] from S [V, n, B or 1] and q [V, n, B]."""
    term = torch.where(S > 0, S * torch.log(torch.where(S > 0, q, 1.0)), 0.0) - q
    return (term - torch.lgamma(S + 1) if lgamma else term).sum((0, 1))


def _mlem64(rays, mu, S, K, lgamma=True):
    """(F [B, n, n], L [B]) of mu [B, n, n], S [V, n] or [B, V, n], K an
    iteration count or one per candidate."""
    n, B = rays.n, mu.shape[0]
    K = torch.as_tensor(K, device=mu.device).expand(B)
    S = S.double()[None].expand(B, -1, -1) if S.dim() == 2 else S.double()
    Fs, Ls = [], []
    step = max(1, int(1.2e9 / (rays.V * n * n * 8)))
    for at in range(0, B, step):
        m, Sp, Kp = mu[at:at + step].double(), S[at:at + step].permute(1, 2, 0), K[at:at + step]
        a = rays.factors(m.reshape(len(m), -1).T)
        sens = rays.backproject(a, torch.ones_like(Sp))
        F = torch.ones(n * n, len(m), dtype=torch.float64, device=mu.device)
        for it in range(int(Kp.max())):
            q = rays.project(a, F)
            r = torch.where(q > 0, Sp / q, 0.0)
            new = torch.where(sens > 0, F * rays.backproject(a, r) / sens, 0.0)
            F = torch.where(it < Kp, new, F)
        Ls.append(_score64(Sp, rays.project(a, F), lgamma))
        Fs.append(F.T.reshape(-1, n, n))
    return torch.cat(Fs), torch.cat(Ls)


def _grad64(rays, case, c, S):
    n, V = rays.n, rays.V
    S = S.double()[:, :, None]
    Ls, gs, Fs = [], [], []
    step = max(1, int(1.5e10 / (rays.V * n * n * 8 * 6 * case["K"])))
    for at in range(0, case["B"], step):
        p = c[at:at + step].double().requires_grad_(True)
        tissue = tuple(p[:, 6 + k, None, None] for k in range(3)) if case["params"] else _constant_tissue()
        mu = _maps(n, p[:, :6], tissue, True)
        mu = mu + (mu.detach().float().double() - mu.detach())      # maps are stored in 32 bits
        a = rays.factors(mu.reshape(len(p), -1).T)
        sens = rays.backproject(a, torch.ones(V, n, len(p), dtype=torch.float64, device=c.device))
        seen = torch.where(sens > 0, sens, 1.0)
        F = torch.ones(n * n, len(p), dtype=torch.float64, device=c.device)
        for _ in range(case["K"]):
            q = rays.project(a, F)
            r = torch.where(q > 0, S / torch.where(q > 0, q, 1.0), 0.0)
            F = torch.where(sens > 0, F * rays.backproject(a, r) / seen, 0.0)
        L = _score64(S, rays.project(a, F), True)
        L.sum().backward()
        Ls.append(L.detach())
        gs.append(p.grad)
        Fs.append(F.detach().T.reshape(-1, n, n))
    return dict(L=torch.cat(Ls), grad=torch.cat(gs), F=torch.cat(Fs))


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "ragged":
        F, L = [None] * case["B"], torch.empty(case["B"], dtype=torch.float64, device="cuda")
        for i, (n, V) in enumerate(RAGGED):
            members = np.flatnonzero(s["cls"] == i)
            if not members.size:
                continue
            Fi, Li = _mlem64(_rays(n, V), torch.stack([s["mu"][b] for b in members]),
                             torch.stack([s["S"][b] for b in members]), torch.tensor(s["K"][members], device="cuda"))
            L[torch.tensor(members, device="cuda")] = Li
            for j, b in enumerate(members):
                F[b] = Fi[j].reshape(-1)
        return dict(F=torch.cat(F), L=L)
    rays = _rays(case["n"], case["V"])
    if kind == "grad":
        return _grad64(rays, case, s["c"], s["S"])
    if kind == "operators":
        q, z = [], []
        for part in torch.split(torch.arange(case["B"]), 16):
            a = rays.factors(s["mu"][part].double().reshape(len(part), -1).T)
            q.append(rays.project(a, s["F"][part].double().reshape(len(part), -1).T).permute(2, 0, 1))
            z.append(rays.backproject(a, s["y"][part].double().permute(1, 2, 0)).T.reshape(-1, rays.n, rays.n))
        return dict(q=torch.cat(q), z=torch.cat(z))
    if kind in ("bo", "evaluate"):
        mu = _maps(rays.n, s["c"].double(), _constant_tissue(), False)
        F, L = _mlem64(rays, mu, s["S"], case["K"], lgamma=kind == "evaluate")
        return dict(F=F, L=L, mu=mu)
    F, L = _mlem64(rays, s["mu"], s["S"], case["K"], lgamma=kind != "unfused")
    return dict(F=F, L=L)
