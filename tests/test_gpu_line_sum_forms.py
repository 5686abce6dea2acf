"""The FP32 line sum's sweeps (whole-tile lines four runs at a time, partial
lines two a slot) where they can go wrong: batches of 0, 1, odd, full and
overflowing line counts, lines broader than many tiles and narrower than the
grid spacing (|u| of a run's far points beyond any window), ragged ranges of
one point to one past a tile, every tiling and batch size, with the optional
terms, against the oracle.

Tolerance on j, all terms positive: widths and Voigt fit 1e-6, strengths 5e-7,
a bracket's roundings 1e-6, a batch of 64 plain terms 64 x 6e-8: 7e-6 of the
value; where the spacing is far above the widths the centre's offset (2^-25
of a point) enters u with h / (2 lamV), and the FP32 path's own bar of 1e-3
above 1e-6 of the maximum holds.  The evaluations counted equal FP64's."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu


def _check(p, k0, nk, tol, tile=0, cpb=0, pb=32, broad=False, floor=1e-6):
    ctx = R.Context(0)
    if tile:
        ctx.set_tiling(tile, cpb)
    ctx.set_line_batch(pb)
    dev = ctx.device
    sp, ln = R.DeviceSpecies(p.species, dev), R.DeviceLines(p.lines, dev)
    cells = R.DeviceCells(p.cells, sp.S, dev)
    R.populations(ctx, sp, cells)
    C = cells.C
    ev = []
    for prec, dt in ((R.FP64, torch.float64), (R.FP32, torch.float32)):
        kap = torch.full((C, nk), float("nan"), dtype=dt, device=dev)
        em = torch.full_like(kap, float("nan"))
        if broad:
            ctx.set_broadening(7, synth.RAD_E_IONIZE, synth.FLOW_MASS)
        ctx.reset_stats()
        R.spectral_coeffs(ctx, sp, ln, cells, p.grid, k0, nk, prec, kap, em)
        ctx.sync()
        ev.append(ctx.get_stats()["evaluations"])
    if broad:
        oracle.set_broadening(7, synth.RAD_E_IONIZE, synth.FLOW_MASS)
    try:
        rk, rj = oracle.spectral_coeffs(p, k0=k0, nk=nk)
    finally:
        oracle.set_broadening(0)
    j, k = em.double().cpu().numpy(), kap.double().cpu().numpy()
    assert np.all(np.isfinite(j)) and np.all(np.isfinite(k))
    assert ev[0] == ev[1]
    big = rj >= floor * rj.max()
    if rj.max() > 0:
        assert np.max(np.abs(j[big] / rj[big] - 1)) <= tol
        kb = np.abs(rk) >= floor * np.abs(rk).max()
        assert np.max(np.abs(k[kb] - rk[kb]) / np.abs(rk[kb])) <= max(tol, 1e-3)   # kappa's terms may cancel
    assert np.all(np.abs(j[rj == 0]) == 0)


def _problem(n_atomic, n_molecular, n_grid, n_cells=3, lam=(50.0, 2000.0)):
    return synth.stagnation_line(seed=31, n_cells=n_cells, n_atomic=n_atomic, n_molecular=n_molecular, n_grid=n_grid,
                                 lam=lam)


@pytest.mark.parametrize("n_lines", [0, 1, 2, 31, 32, 33, 63, 64, 65, 97])
def test_line_counts(n_lines):
    """All lines in one tile: lam0 within 4 points of its middle."""
    p = _problem(400, 400, 4001)
    h = 1950.0 / 4000
    p.lines = synth.subset_lines(p.lines, np.arange(max(n_lines, 1)))
    if n_lines == 0:
        p.lines.lam0[:] = 50.0 + 3990 * h    # out of the range
    else:
        p.lines.lam0[:] = 50.0 + h * (1064.0 + np.linspace(-4, 4, len(p.lines)))
    p.lines.lamS0[:] = np.geomspace(1e-3, 30.0, len(p.lines))
    _check(p, 1000, 130, 1e-3)


@pytest.mark.parametrize("k0,nk", [(0, 1), (5, 127), (640, 128), (640, 129), (3001, 1000)])
@pytest.mark.parametrize("stark", [0.0, 0.05, 20.0])
def test_widths(stark, k0, nk):
    p = _problem(800, 2000, 4001)
    p.lines.lamS0[:] = stark
    _check(p, k0, nk, 1e-3)


@pytest.mark.parametrize("n_grid", [2, 40, 300])
def test_grid_far_coarser_than_the_lines(n_grid):
    p = _problem(400, 400, n_grid)
    p.lines.lam0[::7] = 50.0 + (1950.0 / (n_grid - 1)) * np.minimum(np.arange(len(p.lines.lam0[::7])) % n_grid, n_grid - 1)
    p.lines = synth.subset_lines(p.lines, np.argsort(p.lines.lam0, kind="stable"))
    _check(p, 0, n_grid, 1e-3)


@pytest.mark.parametrize("tile,cpb", [(128, 2), (128, 4), (128, 8), (256, 2), (256, 4), (256, 8), (512, 4)])
@pytest.mark.parametrize("pb", [32, 64])
def test_tilings(tile, cpb, pb):
    _check(_problem(2000, 20_000, 200_001, n_cells=5), 60_000, 5000, 7e-6, tile, cpb, pb)


@pytest.mark.parametrize("tile", [128, 256, 512])
def test_full_lorentz(tile):
    _check(_problem(2000, 10_000, 200_001, n_cells=5), 30_000, 3001, 1.4e-5, tile, 4, 32, broad=True)
