"""Partition functions over the range of the fixed-point exponentials and past
its ends: energies of 0, below its resolution, at and beyond 2^20 cm^-1 and
negative, temperatures from 150 K (exponents past its limit) to 2e6 K (factors
near 1), one cell, three cells and enough for four cells a block.

Tolerance on ln(N/Z), against extended precision with the same b = c2 / T in
64 bits: a term errs by at most 4 x 2^-53 and its energy by 2^-45 b (or, by
exp, by 2^-53 b E <= 8e-14 with b E <= 690), a thread adds at most 40 terms
(40 x 2^-53), the logarithms round |ln N| + |ln Z| <= 800 to 2^-53 each:
8e-14 + 5e-15 + 9e-14 < 2e-13."""
import numpy as np
import pytest

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu
LD = np.longdouble
C2 = (6.626e-27 * 2.998e10) / 1.380e-16


@pytest.mark.parametrize("n_cells", [1, 3, 700])
def test_lnpref_over_the_range(n_cells):
    ctx = R.Context(0)
    p = synth.stagnation_line(seed=21, n_cells=n_cells, n_atomic=3000, n_molecular=500, n_grid=11)
    sp, rng = p.species, np.random.default_rng(4)
    n = len(sp.atom_E)
    for at, E in ((1, 1e-9), (2, 2.0 ** 20), (3, np.nextafter(2.0 ** 20, 0)), (4, 2.5e6), (5, -3.0), (6, 1e-30),
                  (7, 0.1), (8, 2.0 ** -45)):
        sp.atom_E[(at * 97) % n] = E
    p.cells.Tve[:] = np.geomspace(150.0, 2e6, n_cells) if n_cells > 1 else 5000.0
    p.cells.Ttr[:] = np.geomspace(2e6, 150.0, n_cells) if n_cells > 1 else 300.0
    p.cells.n[:] = 10.0 ** rng.uniform(10, 17, p.cells.n.shape)
    dsp = R.DeviceSpecies(sp, ctx.device)
    cells = R.DeviceCells(p.cells, dsp.S, ctx.device)
    got = R.populations(ctx, dsp, cells)
    ctx.sync()
    got = got.cpu().numpy()
    for c in np.unique(np.linspace(0, n_cells - 1, 12).astype(int)):
        bv, bt = LD(C2 / p.cells.Tve[c]), LD(C2 / p.cells.Ttr[c])
        for s in range(dsp.S):
            if sp.kind[s] == 0:
                i0, i1 = sp.atom_off[s], sp.atom_off[s + 1]
                Z = (np.exp(-bv * sp.atom_E[i0:i1].astype(LD)) * sp.atom_g[i0:i1]).sum()
            else:
                Z = LD(0)
                for i in range(sp.st_off[s], sp.st_off[s + 1]):
                    nv, nj = sp.st_nv[i], sp.st_nj[i]
                    vib = sp.vib_E[sp.st_vib_off[i]:][:nv].astype(LD)
                    rot = sp.rot_E[sp.st_rot_off[i]:][:nv * nj].astype(LD).reshape(nv, nj)
                    J = np.arange(nj)
                    w = (2 * J + 1) * sp.st_Lalt.reshape(-1, 2)[i][J % 2]
                    zr = (np.exp(-bt * rot) * w).sum(1)
                    Z += sp.st_g[i] / sp.st_sigma[i] * np.exp(-bv * LD(sp.st_E[i])) * (np.exp(-bv * vib) * zr).sum()
            ref = np.log(LD(p.cells.n[c, sp.density_col[s]])) - np.log(Z)
            assert abs(LD(got[c, s]) - ref) <= 2e-13, (c, s, float(got[c, s]), float(ref))
