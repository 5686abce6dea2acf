"""The search for equal rays, at the sizes from which it runs (segments x
columns past 2^25, 256 columns) and just below: the sets of
tests/test_gpu_march_pairs.py, with its tolerance against the FP64 march, and
equal rays bit for bit."""
import numpy as np
import pytest
import torch

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth
from test_gpu_march_pairs import _rays

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("past", [False, True])
@pytest.mark.parametrize("kind,n", [("all equal", 8), ("all equal", 33), ("mirrored", 64), ("threes", 31), ("near", 40),
                                    ("distinct", 17), ("mirrored", 2049), ("mirrored", 2048), ("threes", 999)])
def test_searched_sets(kind, n, past):
    ctx = R.Context(0)
    rng = np.random.default_rng(n + 1)
    C, P = 50, 3 if n < 100 else 1
    flat = [r for p in range(P) for r in _rays(kind if p != 1 else "distinct", n, rng, C)]
    seg = np.concatenate([[0], np.cumsum([len(r[0]) for r in flat])])
    nk = -(-2 ** 25 // int(seg[-1])) - (0 if past else 1)
    assert nk >= 256
    rays = R.rays_from_arrays(np.arange(P + 1) * n, seg, np.concatenate([r[0] for r in flat]),
                              np.concatenate([r[1] for r in flat]), np.arange(len(flat) + 1),
                              np.array([r[2] for r in flat]), rng.uniform(0.1, 1.0, len(flat)),
                              np.array([r[3] for r in flat]), 6000.0, ctx.device)
    g = synth.Grid(300.0, 900.0, 200_000)
    kap = torch.as_tensor(10.0 ** rng.uniform(-5, 0.3, (C, nk)), device=ctx.device).float()
    em = torch.as_tensor(rng.uniform(0.5, 2.0, (C, nk)), device=ctx.device).float()
    out = {}
    for prec, dt in ((R.FP32, torch.float32), (R.FP64, torch.float64)):
        q = torch.full((P, nk), float("nan"), dtype=dt, device=ctx.device)
        I = torch.full((len(flat), nk), float("nan"), dtype=dt, device=ctx.device)
        R.trace_rays(ctx, rays, C, kap.to(dt), em.to(dt), g, 0, nk, prec, q, I)
        ctx.sync()
        out[prec] = q.double(), I.double()
    (q32, I32), (q64, I64) = out[R.FP32], out[R.FP64]
    assert float(((I32 - I64).abs() / I64.abs().clamp(min=2.0 * 40 * 0.01)).max()) <= 3.8e-5
    assert float((q32 / q64 - 1).abs().max()) <= 3.8e-5
    seen = {}
    for i, (c, d, s, w) in enumerate(flat):   # equal in FP32: equal intensities
        key = (i // n, c.tobytes(), d.astype(np.float32).tobytes(), np.float32(s).tobytes(), w)
        if key in seen:
            assert torch.equal(I32[i], I32[seen[key]])
        seen.setdefault(key, i)
    if kind in ("all equal", "mirrored", "threes"):
        assert len(seen) < len(flat)
