"""Bundles with more directions than their set's max_dirs says (two or more)
are marched whole in every form of the march: in one warp, dealt to several,
with eight bundles a point or fewer, on both sides of the size at which the
form changes.  Against the same set with its true max_dirs, within the march's
rounding (tests/test_gpu_march_steps.py: 7e-14 in FP64, 3.8e-5 in FP32)."""
import numpy as np
import pytest
import torch

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [(R.FP64, 7e-14), (R.FP32, 3.8e-5)])
@pytest.mark.parametrize("bundles,nk", [(1, 70), (1, 152 * 11 * 32 + 1), (3, 33), (9, 70)])
@pytest.mark.parametrize("dirs,claimed", [(18, 17), (18, 2), (35, 17), (40, 18), (65, 17), (65, 5), (64, 63)])
def test_more_directions_than_claimed(dirs, claimed, bundles, nk, precision, tol):
    ctx = R.Context(0)
    rng = np.random.default_rng(dirs)
    C, m = 9, 7
    dt = torch.float64 if precision == R.FP64 else torch.float32
    tk = torch.as_tensor(2.0 ** rng.uniform(-20, -3, (C, nk)), device=ctx.device).to(dt)
    tj = torch.as_tensor(2.0 ** rng.uniform(-3, 3, (C, nk)), device=ctx.device).to(dt)
    n = bundles * dirs
    rays = R.rays_from_arrays([0, bundles], np.arange(bundles + 1) * m, rng.integers(0, C, bundles * m),
                              rng.uniform(0.1, 0.5, bundles * m), np.arange(bundles + 1) * dirs,
                              rng.uniform(1.0, 8.0, n), rng.uniform(0.5, 1.5, n), np.zeros(bundles), 0.0, ctx.device)
    out = []
    for c in (dirs, claimed):
        rays.struct.max_dirs = c
        q = torch.empty((1, nk), dtype=dt, device=ctx.device)
        I = torch.full((n, nk), float("nan"), dtype=dt, device=ctx.device)
        R.trace_rays(ctx, rays, C, tk, tj, synth.Grid(100.0, 200.0, max(nk, 2)), 0, nk, precision, q, I)
        ctx.sync()
        out.append((q.cpu().numpy(), I.cpu().numpy()))
    for a, b in zip(*out):
        assert np.all(np.isfinite(b)) and np.max(np.abs(a / b - 1.0)) <= tol
