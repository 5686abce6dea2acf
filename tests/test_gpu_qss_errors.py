"""Refused QSS models: a transition outside the levels, in any warp's share of
the list, and systems without a pivot, over one cell and over more cells than
the grid holds at once, so that blocks start while others report.  The call is
EINVAL, and the context solves the good model afterwards, to the same bits."""
import numpy as np
import pytest
import torch

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu


def _solve(ctx, m, cells):
    dm, dc = R.DeviceCrModel(m, ctx.device), R.DeviceCells(cells, 8, ctx.device)
    out = torch.empty((len(cells.Ttr), dm.l), dtype=torch.float64, device=ctx.device)
    R.qss_populations(ctx, dm, dc, out)
    ctx.sync()
    return out.cpu().numpy()


@pytest.mark.parametrize("cells", [1, 700, 20_000])
@pytest.mark.parametrize("kind", ["upper", "order", "lower", "singular"])
def test_refused_models(kind, cells):
    ctx = R.Context(0)
    m = synth.cr_model(species="N", n_levels=32, seed=5)
    p = synth.stagnation_line(n_cells=30, n_atomic=10, n_molecular=10, n_grid=11)
    at = np.arange(cells) % 30
    c = synth.Cells(Ttr=p.cells.Ttr[at], Tve=p.cells.Tve[at], n=p.cells.n[at])
    good = _solve(ctx, m, c)
    bads = []
    if kind == "singular":   # nothing moves between the levels
        bads.append(dict(m, **{k: np.zeros_like(m[k]) for k in ("hp_C", "e_C", "A", "ii_C")}))
    else:
        for t in (0, 33, 70, 127, 128, 495):   # shares of all four warps, the list's ends
            key, v = {"upper": ("up", 255), "order": ("up", int(m["lo"][t])), "lower": ("lo", -1)}[kind]
            b = dict(m, **{key: m[key].copy()})
            b[key][t] = v
            bads.append(b)
    for b in bads:
        with pytest.raises(R.RapralError) as e:
            _solve(ctx, b, c)
        assert e.value.code == R.EINVAL
        ctx.clear_status()
        assert np.array_equal(_solve(ctx, m, c), good)
