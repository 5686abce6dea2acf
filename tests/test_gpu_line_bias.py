"""The FP32 line sum does not lean: the mean signed error of the emission over
many lines, cells and points, against the FP64 path, on spacings that FP32
holds exactly and that it rounds by up to 4e-8.

Every line and cell rounds on its own (2e-7 a point, over a thousand lines and
24 cells: 1e-8 of the mean, twice that where a few hot cells hold most points
above 1e-6 of the maximum), and the approximate functions lean by 5e-9 or are
corrected; an uncorrected constant leans for all: the spacing's rounding by
twice itself, the Gaussian's exponent or ex2 by 5e-8 and more.  Bound: 8e-8.
The root mean square stays below 2.4e-7, twice the FP32 rounding."""
import pytest
import torch

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_grid", [300_001, 524_289, 650_000, 800_003, 1_000_001])
def test_mean_error(n_grid):
    ctx = R.Context(0)
    mean, square, count = 0.0, 0.0, 0
    for seed in (41, 42, 43):
        p = synth.stagnation_line(seed=seed, n_cells=24, n_atomic=4000, n_molecular=60_000, n_grid=n_grid)
        sp, ln = R.DeviceSpecies(p.species, ctx.device), R.DeviceLines(p.lines, ctx.device)
        cells = R.DeviceCells(p.cells, sp.S, ctx.device)
        R.populations(ctx, sp, cells)
        k0, nk = int(0.2 * n_grid), 8000
        em = []
        for prec, dt in ((R.FP64, torch.float64), (R.FP32, torch.float32)):
            kap = torch.empty((24, nk), dtype=dt, device=ctx.device)
            em.append(torch.empty_like(kap))
            R.spectral_coeffs(ctx, sp, ln, cells, p.grid, k0, nk, prec, kap, em[-1])
        ctx.sync()
        a, b = em[1].double(), em[0]
        big = b > 1e-6 * b.max()
        e = a[big] / b[big] - 1.0
        mean, square, count = mean + float(e.sum()), square + float((e * e).sum()), count + e.numel()
    assert abs(mean / count) <= 8e-8, mean / count
    assert (square / count) ** 0.5 <= 2.4e-7, (square / count) ** 0.5
