"""The planning of the line sum (checks, window tiles and records of the lines
whose window reaches the range) on ranges that most lines miss: lines whose
window ends just inside, just outside or across the range, ranges of one
point, of one tile and a point, and at the grid's end, sorted and unsorted
lists, with and without the optional Lorentz terms.  FP64 against the oracle
to 1e-10 (the bar of the parity tests), and the same (line, cell, point)
evaluations in FP32."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("broad", [False, True])
@pytest.mark.parametrize("shuffle", [False, True])
@pytest.mark.parametrize("k0,nk", [(0, 1), (1537, 129), (4000, 512), (8990, 11)])
def test_range_of_lines(k0, nk, shuffle, broad):
    ctx = R.Context(0)
    p = synth.stagnation_line(seed=11, n_cells=5, n_atomic=2000, n_molecular=6000, n_grid=9001)
    if shuffle:
        order = np.random.default_rng(3).permutation(len(p.lines))
        p.lines = synth.Lines(**{k: np.ascontiguousarray(getattr(p.lines, k)[order])
                                 for k in synth.Lines.__dataclass_fields__})
    dev = ctx.device
    sp, ln = R.DeviceSpecies(p.species, dev), R.DeviceLines(p.lines, dev)
    cells = R.DeviceCells(p.cells, sp.S, dev)
    R.populations(ctx, sp, cells)
    if broad:
        ctx.set_broadening(7, synth.RAD_E_IONIZE, synth.FLOW_MASS)
        oracle.set_broadening(7, synth.RAD_E_IONIZE, synth.FLOW_MASS)
    try:
        rk, rj = oracle.spectral_coeffs(p, k0=k0, nk=nk)
    finally:
        oracle.set_broadening(0)
    counts = []
    for precision, dt in ((R.FP64, torch.float64), (R.FP32, torch.float32)):
        kap = torch.full((5, nk), float("nan"), dtype=dt, device=dev)
        em = torch.full_like(kap, float("nan"))
        ctx.reset_stats()
        R.spectral_coeffs(ctx, sp, ln, cells, p.grid, k0, nk, precision, kap, em)
        ctx.sync()
        counts.append(ctx.get_stats()["evaluations"])
        if precision == R.FP64:
            for got, ref in ((kap, rk), (em, rj)):
                got = got.cpu().numpy()
                assert np.array_equal(ref == 0, got == 0)
                assert np.max(np.abs(got - ref)) <= 1e-10 * max(np.max(np.abs(ref)), 1e-300)
                nz = ref != 0
                assert not nz.any() or np.max(np.abs(got[nz] / ref[nz] - 1)) <= 1e-10
    assert counts[0] == counts[1]
