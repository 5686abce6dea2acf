"""Equal rays of a point are marched once: caller-built sets with rays that
repeat, nearly repeat, or differ only in a scale, a wall flag, one cell or one
length, against the FP64 march of the same set (which marches every ray).
FP32 tolerance per intensity: the FP32 bar of tests/test_gpu_march_steps.py
(40 segments, 3.8e-5 of the largest emission scale); repeated rays bit for bit.
Sizes: fewer rays than slices are not paired (another kernel), exactly eight,
odd numbers, more than the 2,048 of a point that are compared."""
import numpy as np
import pytest
import torch

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu


def _rays(kind, n, rng, C):
    """Lists of (cells, lengths, scale, wall) of one point's n rays."""
    rays = []
    for i in range(n):
        m = int(rng.integers(1, 41))
        rays.append([rng.integers(0, C, m), rng.uniform(0.01, 1.0, m), float(rng.uniform(0.5, 2.0)), 0])
    if kind == "all equal":
        rays = [list(rays[0]) for _ in range(n)]
    elif kind == "mirrored":
        for i in range(n // 2):
            rays[n - 1 - i] = list(rays[i])
    elif kind == "threes":
        for i in range(0, n - 2, 3):
            rays[i + 1] = list(rays[i])
            rays[i + 2] = list(rays[i])
    elif kind == "near":
        for i in range(0, n - 1, 2):
            c, d, s, w = rays[i]
            c, d = c.copy(), d.copy()
            which = (i // 2) % 5
            if which == 0:
                s = float(np.nextafter(np.float32(s), np.float32(9)))
            elif which == 1:
                w = 1
            elif which == 2:
                c[-1] = (c[-1] + 1) % C
            elif which == 3:
                d[0] = float(np.nextafter(np.float32(d[0]), np.float32(9)))
            else:
                d = d * (1 + 1e-12)     # the same in FP32: equal rays
            rays[i + 1] = [c, d, s, w]
    return rays


@pytest.mark.parametrize("nk", [1, 63, 200, 201])
@pytest.mark.parametrize("kind,n", [("all equal", 8), ("all equal", 33), ("mirrored", 7), ("mirrored", 64), ("threes", 31),
                                    ("near", 40), ("distinct", 17), ("mirrored", 2049), ("mirrored", 2048)])
def test_pairs(kind, n, nk):
    ctx = R.Context(0)
    rng = np.random.default_rng(n)
    C, P = 50, 3 if n < 100 else 1
    pts = [_rays(kind if p != 1 else "distinct", n, rng, C) for p in range(P)]
    flat = [r for p in pts for r in p]
    seg = np.concatenate([[0], np.cumsum([len(r[0]) for r in flat])])
    w = rng.uniform(0.1, 1.0, len(flat))
    rays = R.rays_from_arrays(np.arange(P + 1) * n, seg, np.concatenate([r[0] for r in flat]),
                              np.concatenate([r[1] for r in flat]), np.arange(len(flat) + 1),
                              np.array([r[2] for r in flat]), w, np.array([r[3] for r in flat]), 6000.0, ctx.device)
    g = synth.Grid(300.0, 900.0, 1000)
    kap = torch.as_tensor(10.0 ** rng.uniform(-5, 0.3, (C, nk)), device=ctx.device).float()
    em = torch.as_tensor(rng.uniform(0.5, 2.0, (C, nk)), device=ctx.device).float()
    out = {}
    for prec, dt in ((R.FP32, torch.float32), (R.FP64, torch.float64)):
        q = torch.empty((P, nk), dtype=dt, device=ctx.device)
        I = torch.full((len(flat), nk), float("nan"), dtype=dt, device=ctx.device)
        R.trace_rays(ctx, rays, C, kap.to(dt), em.to(dt), g, 0, nk, prec, q, I)
        ctx.sync()
        out[prec] = q.double().cpu().numpy(), I.double().cpu().numpy()
    (q32, I32), (q64, I64) = out[R.FP32], out[R.FP64]
    scale = np.maximum(np.abs(I64), 2.0 * 40 * 0.01)
    assert np.max(np.abs(I32 - I64) / scale) <= 3.8e-5
    assert np.max(np.abs(q32 / q64 - 1)) <= 3.8e-5
    for i, a in enumerate(flat):     # rays equal in FP32 have equal intensities
        for j in range(max(0, i - 3), i):
            b = flat[j]
            if i // n == j // n and len(a[0]) == len(b[0]) and (a[0] == b[0]).all() and a[3] == b[3] and \
                    np.float32(a[2]) == np.float32(b[2]) and (np.float32(a[1]) == np.float32(b[1])).all():
                assert np.array_equal(I32[i], I32[j])
