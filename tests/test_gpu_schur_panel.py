"""The blocked inverse and the sheet's entry order at the edges of their tiles:
panels of 32 columns with remainders, warps of eight rows (up to 256 points) and
of 32, several bodies' worth of points; S^-1 through f0 = S^-1 1, whose residual
a refined solve leaves at a few FP64 roundings, and R_s f against the sum of its
stencils."""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf
from oracle import body as OB
from oracle import vic as OV

pytestmark = pytest.mark.gpu

GRID = (700, 690, 0.01, -3.5, -3.45)


@pytest.mark.parametrize("ns", [4, 31, 32, 33, 64, 65, 255, 256, 257, 288, 520])
def test_factor_and_entry_order(ns):
    plan = pf.Plan(*GRID, pf.PF_FP64)
    r = 1.7 * GRID[2] * ns / (2 * np.pi) + 0.02
    th = 2 * np.pi * np.arange(ns) / ns + 0.05
    x, y, ds = r * np.cos(th), 0.8 * r * np.sin(th), np.full(ns, 2 * np.pi * r / ns)
    if ns > 8:                                # points in an order that is not the grid's, some of them on one another's nodes
        perm = np.random.default_rng(ns).permutation(ns)
        x, y = x[perm], y[perm]
    sch = pf.pf_schur_factor(plan, x, y, ds)
    g0, f0, S = pf.pf_schur_info(sch)
    scale = np.abs(S).sum(1).max() * np.abs(f0).max()
    assert np.abs(S @ f0 - 1.0).max() < 1e-13 * max(1.0, scale)
    assert abs(np.dot(ds, f0) - g0) < 1e-13 * np.dot(ds, np.abs(f0))
    assert np.abs(S * ds[:, None] - (S * ds[:, None]).T).max() < 1e-13 * np.abs(S).max() * ds.max()
    f = np.random.default_rng(3).normal(0.0, 1.0, ns)
    w = torch.zeros(GRID[1], GRID[0], dtype=torch.float64, device="cuda")
    pf.pf_sheet_regularize(plan, sch, torch.from_numpy(f).cuda(), w)
    og = OV.Grid(*GRID)
    ref = OB.regularize_surface(og, OB.SurfaceStencil(og, x, y), f, ds)
    assert np.abs(w.cpu().numpy() - ref).max() < 1e-13 * np.abs(ref).max()
    pf.pf_sync(plan)
