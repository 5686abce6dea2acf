"""Partition functions of cold cells, where a level's exponent c2 E / T is of
order one for energies of a wavenumber or less, and on both sides of the
temperature (1,473 K) at which the exponentials change their form.

Tolerance on ln(N/Z), against extended precision with the same c2 / T in 64
bits: a term is a product of at most three exponentials, each with 4 x 2^-53
beside its exponent's own rounding x 2^-53 (averaged over the terms, as the
reference weighs them); 60 additions on the way of a term; the two logarithms
and their difference round |ln N|, |ln Z| and the result."""
import numpy as np
import pytest

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu
LD = np.longdouble
C2 = (6.626e-27 * 2.998e10) / 1.380e-16
T = np.array([0.05, 0.3, 3.0, 20.0, 77.0, 150.0, 300.0, 700.0, 1400.0, 1473.0, 1474.0, 1600.0, 3000.0])


@pytest.mark.parametrize("n_cells", [13, 700])
def test_cold_cells(n_cells):
    ctx = R.Context(0)
    p = synth.stagnation_line(seed=21, n_cells=n_cells, n_atomic=3000, n_molecular=500, n_grid=11)
    sp, rng = p.species, np.random.default_rng(4)
    for s in range(len(sp.kind)):   # fine-structure levels of every atom
        if sp.kind[s] == 0:
            i0, i1 = sp.atom_off[s], sp.atom_off[s + 1]
            at = i0 + 1 + rng.permutation(i1 - i0 - 1)[:60]
            sp.atom_E[at] = 10.0 ** rng.uniform(-2, 3, len(at))
    p.cells.Tve[:] = np.resize(T, n_cells)
    p.cells.Ttr[:] = np.resize(T[::-1], n_cells)
    p.cells.n[:] = 10.0 ** rng.uniform(10, 17, p.cells.n.shape)
    dsp = R.DeviceSpecies(sp, ctx.device)
    cells = R.DeviceCells(p.cells, dsp.S, ctx.device)
    got = R.populations(ctx, dsp, cells)
    ctx.sync()
    got = got.cpu().numpy()
    for c in list(range(13)) + [n_cells - 1]:
        bv, bt = LD(C2 / p.cells.Tve[c]), LD(C2 / p.cells.Ttr[c])
        for s in range(dsp.S):
            if sp.kind[s] == 0:
                i0, i1 = sp.atom_off[s], sp.atom_off[s + 1]
                x = bv * sp.atom_E[i0:i1].astype(LD)
                t = np.exp(-x) * sp.atom_g[i0:i1]
                Z, X = t.sum(), (t * x).sum()
            else:
                Z = X = LD(0)
                for i in range(sp.st_off[s], sp.st_off[s + 1]):
                    nv, nj = sp.st_nv[i], sp.st_nj[i]
                    vib = sp.vib_E[sp.st_vib_off[i]:][:nv].astype(LD)
                    rot = sp.rot_E[sp.st_rot_off[i]:][:nv * nj].astype(LD).reshape(nv, nj)
                    J = np.arange(nj)
                    w = (2 * J + 1) * sp.st_Lalt.reshape(-1, 2)[i][J % 2]
                    x = bv * (LD(sp.st_E[i]) + vib)[:, None] + bt * rot
                    t = sp.st_g[i] / sp.st_sigma[i] * np.exp(-x) * w
                    Z, X = Z + t.sum(), X + (t * x).sum()
            if Z < LD(2.0) ** -900:   # past FP64's range (a molecule's zero-point energy at 0.05 K)
                continue
            lnN, lnZ = np.log(LD(p.cells.n[c, sp.density_col[s]])), np.log(Z)
            tol = (12 + float(X / Z) + 60 + abs(float(lnN)) + abs(float(lnZ)) + abs(float(lnN - lnZ))) * 2.0 ** -53
            assert abs(LD(got[c, s]) - (lnN - lnZ)) <= tol, (c, s, float(abs(LD(got[c, s]) - (lnN - lnZ)) / tol))
