"""A line whose strength is past the FP32 range (an Einstein coefficient of
1e80) makes the points of its own window infinite and no others: the points
outside keep the values of the list without it, within the 7e-6 of
tests/test_gpu_line_sum_forms.py (the other lines then lie in other slots and
share other reciprocals).  Narrow and wide lines alternate, so that a slot's
two windows differ.  The window is where FP64, which holds such a strength,
sees the line."""
import numpy as np
import pytest
import torch

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile,pb", [(128, 32), (128, 64), (256, 32), (512, 64)])
@pytest.mark.parametrize("strong", [0, 7, 20, 21, 38])
@pytest.mark.parametrize("profile", [R.PROFILE_WHITING, R.PROFILE_VOIGT])
def test_strength_past_fp32(profile, strong, tile, pb):
    ctx = R.Context(0)
    ctx.set_tiling(tile, 4)
    ctx.set_line_batch(pb)
    ctx.set_profile(profile)
    p = synth.stagnation_line(seed=31, n_cells=3, n_atomic=400, n_molecular=400, n_grid=100_001)
    h = 1950.0 / 100_000
    p.lines = synth.subset_lines(p.lines, np.arange(39))
    p.lines.lam0[:] = 50.0 + h * (2000.3 + 13.7 * np.arange(39))
    p.lines.lamS0[:] = np.where(np.arange(39) % 2 == 0, 0.0, 0.02)
    p.lines.A[:] = 1e6
    k0, nk = 1900, 700
    sp = R.DeviceSpecies(p.species, ctx.device)
    out = {}
    for A in (0.0, 1e80):
        p.lines.A[strong] = A
        ln = R.DeviceLines(p.lines, ctx.device)
        cells = R.DeviceCells(p.cells, sp.S, ctx.device)
        R.populations(ctx, sp, cells)
        for prec, dt in ((R.FP64, torch.float64), (R.FP32, torch.float32)):
            kap = torch.empty((3, nk), dtype=dt, device=ctx.device)
            em = torch.empty_like(kap)
            R.spectral_coeffs(ctx, sp, ln, cells, p.grid, k0, nk, prec, kap, em)
            ctx.sync()
            out[A, prec] = kap.double().cpu().numpy(), em.double().cpu().numpy()
    inside = out[1e80, R.FP64][1] != out[0.0, R.FP64][1]
    assert inside.any() and not inside.all()
    assert np.all(np.isinf(out[1e80, R.FP32][1][inside]))
    for got, ref in zip(out[1e80, R.FP32], out[0.0, R.FP32]):
        a, b = got[~inside], ref[~inside]
        assert np.all(np.isfinite(a))
        big = np.abs(b) >= 1e-6 * np.abs(b).max()
        assert np.max(np.abs(a[big] / b[big] - 1)) <= 7e-6
