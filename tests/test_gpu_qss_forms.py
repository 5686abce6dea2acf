"""Row assembly of the QSS systems: level counts around the unrolled parts,
models in which pairs of levels have several transitions (their rates are
added) or none, one cell and more cells than one pass of the grid; against
the oracle, FP64 within 1e-10 relative per level, the bar of the other QSS
tests (condition 2e-14 for a relative change of 1e-15 of every entry; the sums
of up to 496 rates here round by 496 x 1.1e-16 = 6e-14 of their terms)."""
import numpy as np
import pytest
import torch

from oracle import qss
from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels", [2, 3, 5, 17, 31, 32])
@pytest.mark.parametrize("several", [False, True])
@pytest.mark.parametrize("cells", [1, 3, 2600])
def test_rows(levels, several, cells):
    ctx = R.Context(0)
    m = synth.cr_model(species="N", n_levels=levels, n_lumped=levels % 3, seed=77 + levels)
    if several:   # every third transition moved onto the pair of the one before it
        for k in range(2, len(m["lo"]), 3):
            m["lo"][k], m["up"][k] = m["lo"][k - 1], m["up"][k - 1]
    p = synth.stagnation_line(n_cells=min(cells, 30), n_atomic=10, n_molecular=10, n_grid=11)
    at = np.arange(cells) % len(p.cells.Ttr)
    c = synth.Cells(Ttr=p.cells.Ttr[at], Tve=p.cells.Tve[at], n=p.cells.n[at])
    dm, dc = R.DeviceCrModel(m, ctx.device), R.DeviceCells(c, 8, ctx.device)
    out = torch.empty((cells, dm.l), dtype=torch.float64, device=ctx.device)
    R.qss_populations(ctx, dm, dc, out)
    ctx.sync()
    got = out.cpu().numpy()
    ref = qss.solve_cells(m, p.cells, ion_col=m["ion_col"])
    assert np.max(np.abs(got[:len(ref)] - ref) / np.abs(ref)) <= 1e-10
    assert np.array_equal(got, got[at])
