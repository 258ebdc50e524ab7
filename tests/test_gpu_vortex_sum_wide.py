"""The right-hand side summed from the vortices on grids so wide that the
lattice Green's function exceeds one, where the fixed-point sums over seven table
entries come closest to 64 bits.

S f of the sheet with s0 = 0 in a fluid at rest is E_s L^-1 R_v Gamma; the same
sum in FP64 on the host, from the plan's table.  Points two cells apart on a
circle keep |S| |f| below 1e3 of the right-hand side, and a refined solve leaves a few roundings of
that: 1e-12 of the largest entry.  (One sum of seven that wrapped around would be off by
2^-27 times a weight and a strength, 1e-10 of it.)"""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf
from oracle.kernels import m4prime, yang3
from oracle.vic import stencil_1d

pytestmark = pytest.mark.gpu


def _offset_weights(isurf, wsurf, ivort, wvort):
    """First node offset and the seven weights of a point against each vortex, one axis."""
    c = np.zeros((len(ivort), 7))
    for a in range(4):
        for b in range(4):
            c[:, a + 3 - b] += wsurf[a] * wvort[:, b]
    return isurf[0] - ivort[:, 0] - 3, c


def _host_sum(plan, grid, x, y, X, Y, G):
    nx, ny, dx, x0, y0 = grid
    table = pf.pf_lgf_table(plan)                                        # [n, m]
    sx, sy = stencil_1d(x, x0, dx, nx, yang3), stencil_1d(y, y0, dx, ny, yang3)
    vx, vy = stencil_1d(X, x0, dx, nx, m4prime), stencil_1d(Y, y0, dx, ny, m4prime)
    k = np.arange(7)
    out = np.empty(len(x))
    for p in range(len(x)):
        bx, cx = _offset_weights(sx[0][p], sx[1][p], *vx)
        by, cy = _offset_weights(sy[0][p], sy[1][p], *vy)
        m, n = np.abs(bx[:, None] + k), np.abs(by[:, None] + k)
        out[p] = np.dot(G, np.einsum("qa,qb,qba->q", cx, cy, table[n[:, :, None], m[:, None, :]]))
    return out


@pytest.mark.parametrize("prec", [pf.PF_FP64, pf.PF_MIXED])
@pytest.mark.parametrize("nx,ny,ns,nv", [(1024, 1024, 130, 4500), (2048, 1800, 256, 3500), (2048, 2048, 40, 3000)])
def test_the_vortex_sum_on_wide_grids(nx, ny, ns, nv, prec):
    dx = 2.0 / (max(nx, ny) - 1)
    grid = (nx, ny, dx, -0.5 * (nx - 1) * dx, -0.5 * (ny - 1) * dx)
    plan = pf.Plan(*grid, prec)
    r = 2.0 * dx * ns / (2 * np.pi)
    # the circle in a corner of the grid: offsets up to the whole of it
    th = 2 * np.pi * np.arange(ns) / ns + 0.1
    x, y = r * np.cos(th) + grid[3] + r + 4.3 * dx, r * np.sin(th) + grid[4] + r + 4.6 * dx
    sch = pf.pf_schur_factor(plan, x, y, np.full(ns, 2 * np.pi * r / ns))
    _, _, S = pf.pf_schur_info(sch)
    rng = np.random.default_rng(ns)
    X = grid[3] + dx * (1.5 + (nx - 4.5) * rng.random(nv))
    Y = grid[4] + dx * (1.5 + (ny - 4.5) * rng.random(nv))
    G = rng.normal(0.0, 0.1, nv)
    f, _, _ = pf.pf_sheet_solve_vortices(plan, sch, *(torch.from_numpy(a).cuda() for a in (X, Y, G)), (0, 0, 0, 0, 0),
                                         pf.PF_SHEET_GIVEN_S0)
    pf.pf_sync(plan)
    got = (S.astype(np.longdouble) @ f.cpu().numpy().astype(np.longdouble)).astype(np.float64)
    want = _host_sum(plan, grid, x, y, X, Y, G)
    assert np.abs(got - want).max() < 1e-12 * np.abs(want).max()
