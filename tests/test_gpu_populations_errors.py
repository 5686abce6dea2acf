"""Refused cells: a temperature or density that fails its check, in the first,
a middle or the last cell, over one cell a block and four, few and many blocks.
The call is EINVAL, and the context computes the good cells afterwards, to the
same bits."""
import numpy as np
import pytest

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cells", [1, 5, 611, 12_000])
def test_refused_cells(n_cells):
    ctx = R.Context(0)
    p = synth.stagnation_line(seed=21, n_cells=n_cells, n_atomic=400, n_molecular=500, n_grid=11)
    dsp = R.DeviceSpecies(p.species, ctx.device)

    def run(cells):
        d = R.DeviceCells(cells, dsp.S, ctx.device)
        R.populations(ctx, dsp, d)
        ctx.sync()
        return d.lnpref.cpu().numpy()

    good = run(p.cells)
    for at in sorted({0, n_cells // 2, n_cells - 1}):
        for kind in ("Ttr", "Tve", "n"):
            c = synth.Cells(Ttr=p.cells.Ttr.copy(), Tve=p.cells.Tve.copy(), n=p.cells.n.copy())
            if kind == "n":
                c.n[at, 3] = -1.0
            else:
                getattr(c, kind)[at] = np.nan if at else 0.0
            with pytest.raises(R.RapralError) as e:
                run(c)
            assert e.value.code == R.EINVAL
            ctx.clear_status()
            assert np.array_equal(run(p.cells), good)
