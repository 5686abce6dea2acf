"""The march's step at the lengths where its series change: optical depths of
a segment below, at and above each limit, columns of mixed depths (so that
the lanes of a warp take different lengths), negative kappa, one to three
bundles of directions, against a march in extended precision.

FP64 tolerance: a step rounds I, A, B and p a few times, each within 2^-53 of
values no larger than |I| + s (|j| + |kappa I|); 40 steps of at most 16
roundings: 40 x 16 x 1.1e-16 = 7e-14 of the largest intensity on the way.
FP32: the same count with 2^-24, 40 x 16 x 6e-8 = 3.8e-5."""
import numpy as np
import pytest
import torch

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _p(t):
    """(1 - (1 - e^-t)/t)/t, extended precision."""
    small = np.abs(t) < LD(0.6)
    s, term = np.zeros_like(t), np.full_like(t, LD(1) / 2)   # sum of (-t)^n / (n + 2)!
    for n in range(26):
        s = s + term
        term = term * (-t) / (n + 3)
    tt = np.where(small, LD(1), t)
    return np.where(small, s, (1 + np.expm1(-tt) / tt) / tt)


def _march(kap, em, dx, scale):
    kap, em = kap.astype(LD), em.astype(LD)
    I = np.zeros((len(scale), kap.shape[1]), LD)
    big = np.zeros_like(I)
    kf, jf = kap[0], em[0]
    n = kap.shape[0]
    for i in range(n):
        kn, jn = ((kap[i] + kap[i + 1]) / 2, (em[i] + em[i + 1]) / 2) if i + 1 < n else (kap[i], em[i])
        s = LD(dx) * scale.astype(LD)[:, None]
        t = kf[None] * s
        p = _p(t)
        I = I + s * ((1 - t * p) * (jf[None] - kf[None] * I) + p * (jn - jf)[None])
        big = np.maximum(big, np.abs(I) + s * np.abs(jf)[None])
        kf, jf = kn, jn
    return I, big


@pytest.mark.parametrize("precision,tol", [(R.FP64, 7e-14), (R.FP32, 3.8e-5)])
@pytest.mark.parametrize("n_mu", [1, 5, 16, 24, 40])
@pytest.mark.parametrize("depth", [0.0, 2.0 ** -17, 2.0 ** -10, 2.0 ** -5, 2.0 ** -4, 0.5, 4.0, "mixed", "negative"])
def test_slab_steps(precision, tol, n_mu, depth):
    ctx = R.Context(0)
    rng = np.random.default_rng(5)
    C, nk, dx = 40, 333, 0.25
    if depth == "mixed":
        d = 2.0 ** rng.uniform(-24, 1, (C, nk))
    elif depth == "negative":
        d = -2.0 ** rng.uniform(-20, -9, (C, nk))
    else:
        d = depth * (1.0 + 2.0 ** -12 * rng.uniform(-1, 1, (C, nk)))   # both sides of the limit
    kap = d / dx
    em = 2.0 ** rng.uniform(-3, 3, (C, nk))
    dt = torch.float64 if precision == R.FP64 else torch.float32
    tk = torch.as_tensor(kap, device=ctx.device).to(dt)
    tj = torch.as_tensor(em, device=ctx.device).to(dt)
    # directions around mu = 1, so that `depth` is the normal ray's and the others straddle it
    mu = np.linspace(0.55, 1.0, n_mu) if depth != "mixed" else np.linspace(0.02, 1.0, n_mu)
    geo = synth.SlabGeometry(cell_order=np.arange(C, dtype=np.int64), dx=np.full(C, dx), mu=mu,
                             wmu=np.full(n_mu, 1.0 / n_mu))
    rays = R.slab_rays(ctx, geo, ctx.device)
    q = torch.empty((1, nk), dtype=dt, device=ctx.device)
    I = torch.full((rays.n_dirs, nk), float("nan"), dtype=dt, device=ctx.device)
    R.trace_rays(ctx, rays, C, tk, tj, synth.Grid(100.0, 200.0, nk), 0, nk, precision, q, I)
    ctx.sync()
    ref, big = _march(tk.double().cpu().numpy(), tj.double().cpu().numpy(), dx, np.concatenate([[1.0], 1.0 / mu]))
    err = np.max(np.abs(I.double().cpu().numpy().astype(LD) - ref) / np.maximum(big, LD(1e-300)))
    assert err <= tol, float(err)


@pytest.mark.parametrize("precision,tol", [(R.FP64, 7e-14), (R.FP32, 3.8e-5)])
@pytest.mark.parametrize("n_mu", [1, 2, 3, 6, 13, 16, 17, 24])
@pytest.mark.parametrize("nk", [1, 31, 33, 152 * 11 * 32, 152 * 11 * 32 + 1])
def test_split_directions(precision, tol, n_mu, nk):
    """The directions of a bundle in one warp or dealt to several: counts around the multiples of a warp's
    share, ranges at and past the line between the two forms, intensities and their weighted sum."""
    ctx = R.Context(0)
    rng = np.random.default_rng(11)
    C, dx, w = 12, 0.5, min(nk, 97)
    kap = np.tile(2.0 ** rng.uniform(-20, 2, (C, w)), (1, -(-nk // w)))[:, :nk]
    em = np.tile(2.0 ** rng.uniform(-3, 3, (C, w)), (1, -(-nk // w)))[:, :nk]
    dt = torch.float64 if precision == R.FP64 else torch.float32
    tk = torch.as_tensor(kap, device=ctx.device).to(dt)
    tj = torch.as_tensor(em, device=ctx.device).to(dt)
    mu = np.linspace(0.1, 0.9, n_mu)
    wmu = rng.uniform(0.5, 1.5, n_mu)
    geo = synth.SlabGeometry(cell_order=np.arange(C, dtype=np.int64), dx=np.full(C, dx), mu=mu, wmu=wmu)
    rays = R.slab_rays(ctx, geo, ctx.device)
    q = torch.empty((1, nk), dtype=dt, device=ctx.device)
    I = torch.full((rays.n_dirs, nk), float("nan"), dtype=dt, device=ctx.device)
    R.trace_rays(ctx, rays, C, tk, tj, synth.Grid(100.0, 200.0, max(nk, 2)), 0, nk, precision, q, I)
    ctx.sync()
    ref, big = _march(tk[:, :w].double().cpu().numpy(), tj[:, :w].double().cpu().numpy(), dx,
                      np.concatenate([[1.0], 1.0 / mu]))
    got = I.double().cpu().numpy()
    reps = -(-nk // w)
    tile = lambda x: np.tile(x.astype(float), (1, reps))[:, :nk]
    assert np.max(np.abs(got - tile(ref)) / np.maximum(tile(big), 1e-300)) <= tol
    weight = rays.t["dir_weight"].cpu().numpy()[:, None]
    flux = np.abs(weight) * tile(big)
    assert np.max(np.abs(q[0].double().cpu().numpy() - (weight * tile(ref)).sum(0)) /
                  np.maximum(flux.sum(0), 1e-300)) <= tol


@pytest.mark.parametrize("precision", [R.FP64, R.FP32])
@pytest.mark.parametrize("claimed", [2, 5, 17])
def test_bundle_longer_than_claimed(precision, claimed):
    """A bundle of 17 directions in a ray set that claims fewer is marched whole (within the march's rounding, as above)."""
    ctx = R.Context(0)
    rng = np.random.default_rng(3)
    C, nk = 9, 70
    dt = torch.float64 if precision == R.FP64 else torch.float32
    tk = torch.as_tensor(2.0 ** rng.uniform(-20, -8, (C, nk)), device=ctx.device).to(dt)
    tj = torch.as_tensor(2.0 ** rng.uniform(-3, 3, (C, nk)), device=ctx.device).to(dt)
    geo = synth.SlabGeometry(cell_order=np.arange(C, dtype=np.int64), dx=np.full(C, 0.5),
                             mu=np.linspace(0.1, 0.9, 16), wmu=np.full(16, 1.0 / 16))
    rays = R.slab_rays(ctx, geo, ctx.device)
    out = []
    for m in (17, claimed):
        rays.struct.max_dirs = m
        q = torch.empty((1, nk), dtype=dt, device=ctx.device)
        I = torch.full((rays.n_dirs, nk), float("nan"), dtype=dt, device=ctx.device)
        R.trace_rays(ctx, rays, C, tk, tj, synth.Grid(100.0, 200.0, nk), 0, nk, precision, q, I)
        ctx.sync()
        out.append(I.cpu().numpy())
    assert np.all(np.isfinite(out[0])) and np.max(np.abs(out[0] / out[1] - 1.0)) <= (
        7e-14 if precision == R.FP64 else 3.8e-5)
