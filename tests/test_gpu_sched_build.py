"""The scatter schedule's builder: every build of a geometry gives the same
bytes (two streams may build a kept schedule at the same time), each sample of
a class once; and the schedules' arena: first use of a geometry on two streams
at once, and calls that find no room in it.

Bounds: a sample lost or listed twice changes one MLEM iteration's image by at
least 1 / (V n) (1.8e-4 at 128 x 128 and 44 views), float32 rounding by less
than 1e-5; back-projections 2e-6 of the oracle's in the 2-norm, as
test_gpu_sched_absent.py."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
from paper_2109_11920_gb300 import Geom, _lib
from paper_2109_11920_gb300 import api as boac
from problems import make_problem, rel_l2

pytestmark = pytest.mark.gpu


def build(g, per, pad, dev):
    lib = _lib.load()
    nbytes = lib.boac_test_schedule_bytes(ctypes.byref(g), per)
    out = torch.empty(nbytes, dtype=torch.uint8, device=dev)
    assert lib.boac_test_schedule(ctypes.byref(g), per, pad, boac._ptr(out), nbytes, boac._stream(dev)) == 0
    return out


# 128 x 128 with 44 and 20 views: classes with more samples than rounds hold
@pytest.mark.parametrize("n,V,per,pad", [(64, 4, 4, 4), (64, 42, 2, 1), (96, 60, 4, 4), (96, 90, 2, 1),
                                         (128, 44, 4, 4), (128, 20, 4, 1), (128, 90, 2, 4), (128, 120, 4, 4)])
def test_builds_are_the_same_bytes(cuda, n, V, per, pad):
    g = Geom.make(n, 25.6 / n, V)
    first = build(g, per, pad, cuda)
    torch.cuda.synchronize(cuda)
    streams = [torch.cuda.Stream(cuda) for _ in range(3)]
    others = []
    for i in range(30):  # builds beside each other (and so in varying company)
        with torch.cuda.stream(streams[i % 3]):
            others.append(build(g, per, pad, cuda))
    torch.cuda.synchronize(cuda)
    for o in others:
        assert torch.equal(first, o)
    # each class: its samples that touch the image, once each
    entries = first.cpu().numpy().view(np.uint16)[:V // per * 9 * 16 * n].reshape(V // per, 9, 16 * n)
    k, b = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    c = 0.5 * (n - 1)
    for gi in range(V // per):
        phi = 2 * np.pi * gi / V
        u = c + (b - c) * np.cos(phi) - (k - c) * np.sin(phi)
        w = c + (b - c) * np.sin(phi) + (k - c) * np.cos(phi)
        margin = np.minimum(np.minimum(u + 1, n - u), np.minimum(w + 1, n - w))
        for cls in range(9):
            e = entries[gi, cls]
            e = e[e != 0xFFFF].astype(int)
            listed = set(e.tolist())
            assert len(listed) == e.size, (gi, cls)
            mine = (k % 3 * 3 + b % 3 == cls)
            code = k * 256 + b
            assert set(code[mine & (margin > 1e-3)].tolist()) <= listed, (gi, cls)
            assert listed <= set(code[mine & (margin > -1e-3)].tolist()), (gi, cls)


def check(p, cuda, calls):
    """Each call's first use of p's geometry on a stream of its own, all at
    once; then again, on kept schedules."""
    g = Geom.make(p.n, p.dx, p.V)
    mu = torch.tensor(p.mu, dtype=torch.float32, device=cuda)
    S = torch.tensor(p.S, dtype=torch.float32, device=cuda)
    B = mu.shape[0]
    y = S.expand(B, -1, -1).contiguous()
    run = dict(fused=lambda: boac.boac_mlem(g, mu, S, torch.ones(B, p.n, p.n, device=cuda), 1, check_status=False)[0],
               unfused=lambda: boac.boac_mlem(g, mu, S, torch.ones(B, p.n, p.n, device=cuda), 1, unfused=True,
                                              check_status=False)[0],
               backproject=lambda: boac.boac_backproject(g, mu, y))
    Fo, _, _ = oracle.mlem_batch(p.geom, p.mu, p.S, 1)
    zo = [oracle.backproject(p.geom, np.float32(p.mu[b]).astype(np.float64), np.float32(p.S).astype(np.float64))
          for b in range(B)]
    torch.cuda.synchronize(cuda)
    for attempt in range(2):
        out = []
        for name in calls:
            with torch.cuda.stream(torch.cuda.Stream(cuda)):
                out.append(run[name]())
        torch.cuda.synchronize(cuda)
        for name, r in zip(calls, out):
            for b in range(B):
                err = rel_l2(r[b].cpu().numpy(), zo[b] if name == "backproject" else Fo[b])
                assert err < (2e-6 if name == "backproject" else 1e-5), (p.n, p.V, name, attempt, b, err)


@pytest.mark.parametrize("V", [20, 28, 36, 40, 48, 52, 56, 68])
def test_first_use_on_several_streams(cuda, V):
    p = make_problem(128, 0.2, V, 2e5, B=2, seed=V)
    check(p, cuda, ("fused", "backproject", "unfused", "fused", "backproject", "unfused"))


# run in a process of its own: the arena stays full for the rest of it
def test_arena_exhausted(cuda):
    code = (
        "import sys; sys.path[:0] = ['tests', '.']\n"
        "import torch\n"
        "import test_gpu_sched_build as t\n"
        "from paper_2109_11920_gb300 import Geom, api\n"
        "dev = torch.device('cuda:0')\n"
        "for V in range(392, 456, 4):  # 16 schedules of 3.4 to 4 MiB, 59.3 of the arena's 64 MiB\n"
        "    api.boac_backproject(Geom.make(128, 0.2, V), torch.zeros(1, 128, 128, device=dev),\n"
        "                         torch.ones(1, V, 128, device=dev))\n"
        "for V in (240, 60, 90, 44):  # 240 takes most of what is left, 60 and 90 find no room, 44 finds it once\n"
        "    p = t.make_problem(128, 0.2, V, 2e5, B=2, seed=V)\n"
        "    t.check(p, dev, ('fused', 'unfused', 'backproject'))\n"
        "print('arena checked')\n")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "arena checked" in r.stdout, r.stdout + r.stderr
