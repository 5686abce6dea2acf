"""The single-direction FP32 march with two and with four columns a lane: few
blocks and enough for four (ten an SM), ranges that end inside a tile, at its
edge and off the vector's multiples, with and without the intensities, against
the FP64 march.  Tolerance as in tests/test_gpu_march_pairs.py: 3.8e-5 of the
largest emission scale for at most 40 segments."""
import numpy as np
import pytest
import torch

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("intensity", [False, True])
@pytest.mark.parametrize("P,n", [(3, 9), (760, 8), (1520, 9), (95, 64)])
@pytest.mark.parametrize("nk", [4, 127, 128, 132, 252, 256, 258, 1028])
def test_columns_a_lane(P, n, nk, intensity):
    ctx = R.Context(0)
    rng = np.random.default_rng(P + nk)
    C, B = 40, P * n
    m = rng.integers(1, 12, B)
    seg = np.concatenate([[0], np.cumsum(m)])
    rays = R.rays_from_arrays(np.arange(P + 1) * n, seg, rng.integers(0, C, seg[-1]), rng.uniform(0.01, 1.0, seg[-1]),
                              np.arange(B + 1), rng.uniform(0.5, 2.0, B), rng.uniform(0.1, 1.0, B),
                              rng.integers(0, 2, B), 6000.0, ctx.device)
    kap = torch.as_tensor(10.0 ** rng.uniform(-5, 0.3, (C, nk)), device=ctx.device).float()
    em = torch.as_tensor(rng.uniform(0.5, 2.0, (C, nk)), device=ctx.device).float()
    out = {}
    for prec, dt in ((R.FP32, torch.float32), (R.FP64, torch.float64)):
        q = torch.full((P, nk), float("nan"), dtype=dt, device=ctx.device)
        I = torch.full((B, nk), float("nan"), dtype=dt, device=ctx.device) if intensity else None
        R.trace_rays(ctx, rays, C, kap.to(dt), em.to(dt), synth.Grid(300.0, 900.0, 2000), 0, nk, prec, q, I)
        ctx.sync()
        out[prec] = q.double(), I.double() if intensity else None
    (q32, I32), (q64, I64) = out[R.FP32], out[R.FP64]
    assert float((q32 / q64 - 1).abs().max()) <= 3.8e-5
    if intensity:
        assert float(((I32 - I64).abs() / I64.abs().clamp(min=0.8)).max()) <= 3.8e-5
