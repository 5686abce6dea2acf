"""Photoionisation tables from far sparser to far denser than the grid, so that
a warp's first points lie in one table interval, in a few, or in hundreds (the
lanes then search for themselves), on ragged ranges, against the oracle: FP64
to 1e-10 relative, FP32 to 1e-3 above 1e-6 of a row's maximum, the bars of
tests/test_gpu_continuum.py."""
import numpy as np
import pytest
import torch

import oracle
from oracle import continuum as ct
from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nodes", [2, 5, 34, 512, 514, 5000])
@pytest.mark.parametrize("n_grid,k0,nk", [(301, 0, 301), (1001, 13, 700), (20_001, 3000, 257)])
def test_node_densities(nodes, n_grid, k0, nk):
    ctx = R.Context(0)
    p = synth.stagnation_line(n_cells=3, n_atomic=400, n_molecular=1000, n_grid=n_grid)
    ms = [synth.continuum_model(species=s, n_levels=12, n_nodes=nodes, seed=1007 + i) for i, s in enumerate("NO")]
    sp = R.DeviceSpecies(p.species, ctx.device)
    cells = R.DeviceCells(p.cells, sp.S, ctx.device)
    R.populations(ctx, sp, cells)
    dm = R.DeviceContinuum(ms, ctx.device)
    ref = ct.continuum(ms, p.cells, oracle.lnpref(p), p.grid, k0, nk)
    for prec, dt in ((R.FP64, torch.float64), (R.FP32, torch.float32)):
        kap = torch.zeros((3, nk), dtype=dt, device=ctx.device)
        em = torch.zeros_like(kap)
        R.continuum_coeffs(ctx, dm, sp.S, cells, p.grid, k0, nk, prec, kap, em)
        ctx.sync()
        for got, r in zip((kap, em), ref):
            err = np.abs(got.double().cpu().numpy() - r) / np.maximum(np.abs(r), 1e-300)
            if prec == R.FP64:
                assert err.max() <= 1e-10
            else:
                assert err[r >= 1e-6 * r.max(axis=1, keepdims=True)].max() <= 1e-3
