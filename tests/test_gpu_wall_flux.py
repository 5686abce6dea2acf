"""The spectral integral at the lengths where its slices change: around one and
two slices, a chunk inside the grid and the grid's ends, and past 65,535 slices
of 1,024 points.  Against a 64-bit sum of the same values; all positive, so a
blocked sum of n of them errs by less than (log2 n + 128) 2^-53 = 2e-14."""
import pytest
import torch

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [R.FP32, R.FP64])
@pytest.mark.parametrize("P,nk,k0,extra", [(1, 1, 0, 9), (3, 1023, 0, 0), (2, 1024, 5, 0), (2, 1025, 0, 7), (1, 2049, 3, 4),
                                           (1, 65535 * 1024, 0, 0), (1, 65535 * 1024 + 1, 0, 0),
                                           (1, 65535 * 1024 + 4097, 1, 1), (2, 70_000_001, 0, 5)])
def test_lengths(P, nk, k0, extra, precision):
    ctx = R.Context(0)
    gen = torch.Generator(device=ctx.device)
    gen.manual_seed(nk)
    dt = torch.float64 if precision == R.FP64 else torch.float32
    ql = torch.rand((P, nk), generator=gen, dtype=dt, device=ctx.device) + 0.5
    n = k0 + nk + extra
    g = synth.Grid(100.0, 900.0, n)
    q = torch.full((P,), 2.0, dtype=torch.float64, device=ctx.device)   # added to
    R.wall_flux(ctx, ql, precision, g, k0, nk, P, q)
    ctx.sync()
    s = ql.double().sum(1)
    if k0 == 0:
        s = s - 0.5 * ql[:, 0].double()
    if k0 + nk == n:
        s = s - 0.5 * ql[:, -1].double()
    ref = 2.0 + s * (800.0 / (n - 1) * 1e-3)
    assert float(((q - ref) / ref).abs().max()) <= 2e-14
