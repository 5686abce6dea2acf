"""Ray sets whose points do not cover all bundles: bundles ahead of the first
point's and after the last point's (a part of a larger set, handed over with
the whole set's lists) belong to no point and are not marched, and nothing is
read for them, whatever an earlier call left in the workspace.  The marched
points' results are those of the set without them, bit for bit in the flux
(the same bundles, in the same groups), and their intensities."""
import numpy as np
import pytest
import torch

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu


def _fill_workspace(ctx):
    """Line records and tile lists of a coefficient call where the march's scratch will lie."""
    p = synth.stagnation_line(seed=3, n_cells=20, n_atomic=4000, n_molecular=20_000, n_grid=20_001)
    sp, ln = R.DeviceSpecies(p.species, ctx.device), R.DeviceLines(p.lines, ctx.device)
    cells = R.DeviceCells(p.cells, sp.S, ctx.device)
    R.populations(ctx, sp, cells)
    kap = torch.empty((20, 4000), dtype=torch.float32, device=ctx.device)
    R.spectral_coeffs(ctx, sp, ln, cells, p.grid, 8000, 4000, R.FP32, kap, torch.empty_like(kap))


@pytest.mark.parametrize("precision", [R.FP32, R.FP64])
@pytest.mark.parametrize("mirrored", [False, True])
@pytest.mark.parametrize("ahead,after", [(1, 0), (0, 1), (37, 0), (0, 5), (11, 300)])
@pytest.mark.parametrize("nk", [130, 40_001])   # without and with the search for equal rays
def test_points_cover_part_of_the_bundles(nk, ahead, after, mirrored, precision):
    ctx = R.Context(0)
    rng = np.random.default_rng(ahead + after)
    C, P, n = 60, 3, 24
    dt = torch.float64 if precision == R.FP64 else torch.float32
    rays = [(rng.integers(0, C, m), rng.uniform(0.01, 1.0, m)) for m in rng.integers(1, 40, ahead + P * n + after)]
    if mirrored:
        for p in range(P):
            for k in range(n // 2):
                rays[ahead + p * n + n - 1 - k] = rays[ahead + p * n + k]
    w = rng.uniform(0.1, 1.0, len(rays))

    def ray_set(part, point_off):
        seg = np.concatenate([[0], np.cumsum([len(r[0]) for r in part])])
        k = len(part)
        return R.rays_from_arrays(point_off, seg, np.concatenate([r[0] for r in part]),
                                  np.concatenate([r[1] for r in part]), np.arange(k + 1), np.ones(k),
                                  w[ahead:ahead + k] if k < len(w) else w, np.zeros(k), 0.0, ctx.device)

    kap = torch.as_tensor(10.0 ** rng.uniform(-5, 0.3, (C, nk)), device=ctx.device).to(dt)
    em = torch.as_tensor(rng.uniform(0.5, 2.0, (C, nk)), device=ctx.device).to(dt)
    g = synth.Grid(300.0, 900.0, 50_000)
    out = []
    for part, off in ((rays, ahead), (rays[ahead:ahead + P * n], 0)):
        s = ray_set(part, off + np.arange(P + 1) * n)
        _fill_workspace(ctx)
        q = torch.full((P, nk), float("nan"), dtype=dt, device=ctx.device)
        I = torch.full((len(part), nk), -1.0, dtype=dt, device=ctx.device)
        R.trace_rays(ctx, s, C, kap, em, g, 0, nk, precision, q, I)
        ctx.sync()
        out.append((q.cpu().numpy(), I.cpu().numpy()))
    (q, I), (q0, I0) = out
    assert np.array_equal(q, q0)
    assert np.array_equal(I[ahead:ahead + P * n], I0)
    assert np.all(I[:ahead] == -1.0) and np.all(I[ahead + P * n:] == -1.0)


@pytest.mark.parametrize("n", [31, 33, 300, 2048])
@pytest.mark.parametrize("claimed", [8, 32, 5000])
@pytest.mark.parametrize("searched", [False, True])
def test_points_larger_than_claimed(searched, n, claimed):
    """max_bundles_per_point sizes launches; a set that states another value has the same intensities, bit for bit."""
    ctx = R.Context(0)
    rng = np.random.default_rng(n)
    C, P = 60, 2
    half = [(rng.integers(0, C, m), rng.uniform(0.01, 1.0, m)) for m in rng.integers(1, 12, P * n)]
    for p in range(P):
        for k in range(n // 3):
            half[p * n + n - 1 - k] = half[p * n + k]
    seg = np.concatenate([[0], np.cumsum([len(r[0]) for r in half])])
    nk = max(256, 2 ** 25 // int(seg[-1]) + 1) if searched else 70
    rays = R.rays_from_arrays(np.arange(P + 1) * n, seg, np.concatenate([r[0] for r in half]),
                              np.concatenate([r[1] for r in half]), np.arange(P * n + 1), np.ones(P * n),
                              rng.uniform(0.1, 1.0, P * n), np.zeros(P * n), 0.0, ctx.device)
    kap = torch.as_tensor(10.0 ** rng.uniform(-5, 0.3, (C, nk)), device=ctx.device).float()
    em = torch.as_tensor(rng.uniform(0.5, 2.0, (C, nk)), device=ctx.device).float()
    out = []
    for m in (n, claimed):
        rays.struct.max_bundles_per_point = m
        q = torch.full((P, nk), float("nan"), dtype=torch.float32, device=ctx.device)
        I = torch.full((P * n, nk), float("nan"), dtype=torch.float32, device=ctx.device)
        R.trace_rays(ctx, rays, C, kap, em, synth.Grid(300.0, 900.0, 200_000), 0, nk, R.FP32, q, I)
        ctx.sync()
        out.append((q.cpu().numpy(), I.cpu().numpy()))
    assert np.array_equal(out[0][1], out[1][1])
    # the bundles' sums: other groups and slices, each compensated; FP32 rounding of up to 16 partial sums
    assert np.max(np.abs(out[0][0] / out[1][0] - 1)) <= 16 * 2.0 ** -24


@pytest.mark.parametrize("precision", [R.FP32, R.FP64])
@pytest.mark.parametrize("nk", [70, 40_001])
def test_points_without_bundles(nk, precision):
    """Segments that no bundle holds and points without bundles: nothing is marched, the flux is zero."""
    ctx = R.Context(0)
    rays = R.rays_from_arrays([0, 0, 0], [0], np.zeros(2000, int), np.ones(2000), [0], np.ones(1), np.ones(1),
                              np.zeros(1), 0.0, ctx.device)
    rays.struct.max_dirs, rays.struct.max_bundles_per_point = 1, 9
    dt = torch.float64 if precision == R.FP64 else torch.float32
    kap = torch.ones((3, nk), dtype=dt, device=ctx.device)
    q = torch.full((2, nk), float("nan"), dtype=dt, device=ctx.device)
    R.trace_rays(ctx, rays, 3, kap, kap, synth.Grid(300.0, 900.0, 50_000), 0, nk, precision, q)
    ctx.sync()
    assert float(q.abs().max()) == 0.0
