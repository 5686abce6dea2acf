"""Ground-level weights and per-cell factors of the optional Lorentz terms over
level lists of lengths around a block's threads and cells past one block.

Levels of an energy whose Boltzmann factor is zero are put in front of every
atom's own, which then stand in reverse order: the partition function is the
same sum in another order, apart by at most the count of its nonzero terms
(under 200) times 2^-53 = 2e-14, and the ground weight is a sum of whole
numbers.  The widths and the line strengths follow it: 1e-12 of the result,
on emission, which has no cancellation."""
import copy

import numpy as np
import pytest
import torch

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import solver, synth

pytestmark = pytest.mark.gpu


def _emission(p):
    ctx = R.Context(0)
    ctx.set_broadening(R.BROAD_RESONANCE | R.BROAD_VDW, synth.RAD_E_IONIZE, synth.FLOW_MASS)
    dp = solver.DeviceProblem(p, ctx)
    R.populations(ctx, dp.species, dp.cells)
    kap = torch.empty((dp.C, p.grid.n), dtype=torch.float64, device=ctx.device)
    em = torch.empty_like(kap)
    R.spectral_coeffs(ctx, dp.species, dp.lines, dp.cells, p.grid, 0, p.grid.n, R.FP64, kap, em)
    ctx.sync()
    return em.cpu().numpy()


@pytest.mark.parametrize("cells,pad", [(1, 0), (3, 1), (128, 500), (129, 512), (130, 2049)])
def test_padded_level_lists(cells, pad):
    p = synth.stagnation_line(n_cells=cells, n_atomic=400, n_molecular=0, n_grid=600)
    ref = _emission(p)
    q = copy.copy(p)
    q.species = sp = copy.copy(p.species)
    E, g, off = [], [], [0]
    for s in range(len(p.species.names)):
        a, b = int(p.species.atom_off[s]), int(p.species.atom_off[s + 1])
        n = pad if b > a else 0
        E += [np.full(n, 1e9), p.species.atom_E[a:b][::-1]]
        g += [np.full(n, 3.0), p.species.atom_g[a:b][::-1]]
        off.append(off[-1] + n + b - a)
    sp.atom_E, sp.atom_g, sp.atom_off = np.concatenate(E), np.concatenate(g), np.array(off, np.int64)
    assert max(np.diff(p.species.atom_off)) < 200
    got = _emission(q)
    assert np.all(np.isfinite(ref)) and np.max(ref) > 0
    assert np.max(np.abs(got - ref) / np.maximum(np.abs(ref), 1e-300)) <= 1e-12
