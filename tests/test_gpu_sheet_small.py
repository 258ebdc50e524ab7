"""The one-cluster sheet solve and the vortex right-hand side at the sizes where
they could go wrong: fewer points than blocks, the last size one cluster solves
and the first that it does not, every mode; vortex counts around a round of 64,
none, some off the grid.

The sheet is held to its own equations with the plan's S: the residual of a
refined solve is a few FP64 roundings of |S| |f| (1e-13 covers 256 terms), the
constraint rows the same.  Two right-hand sides that differ by roundings give
sheets within cond(S) 1e-14."""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu

GRID = (400, 380, 0.01, -2.0, -1.9)


def _circle(ns):
    """ns points about 1.6 cells apart."""
    r = 1.6 * GRID[2] * ns / (2 * np.pi) if ns > 8 else 0.05
    th = 2 * np.pi * np.arange(ns) / ns + 0.1
    return r * np.cos(th), r * np.sin(th), np.full(ns, 2 * np.pi * r / ns)


def _vortices(n, seed, outside=0):
    rng = np.random.default_rng(seed)
    a, r = rng.uniform(0, 2 * np.pi, n), rng.uniform(0.9, 1.7, n)
    X, Y, G = r * np.cos(a), r * np.sin(a), rng.normal(0.0, 0.1, n)
    X[:outside] = 9.0
    return [torch.from_numpy(v).cuda() for v in (X, Y, G)]


@pytest.mark.parametrize("prec", [pf.PF_FP64, pf.PF_MIXED])
@pytest.mark.parametrize("ns", [4, 7, 9, 64, 255, 256, 257])
def test_every_mode_satisfies_its_equations(ns, prec):
    plan = pf.Plan(*GRID, prec)
    x, y, ds = _circle(ns)
    sch = pf.pf_schur_factor(plan, x, y, ds)
    g0, f0, S = pf.pf_schur_info(sch)
    X, Y, G = _vortices(150, ns)
    motion = (0.1, -0.2, 0.3, 1.0, 0.25)
    sb = (0.1 - 1.0) * y - (-0.2 - 0.25) * x - 0.5 * 0.3 * (x * x + y * y)
    Xn, Yn = [1.3 * x[0] + 0.03, 1.3 * x[ns // 2] - 0.04], [1.3 * y[0] + 0.02, 1.3 * y[ns // 2] - 0.01]

    def ew(vx, vy, vg):            # E L^-1 w of a vortex set, from the sheet it gives with s0 = 0 in a flow at rest
        f, _, _ = pf.pf_sheet_solve_vortices(plan, sch, vx, vy, vg, (0, 0, 0, 0, 0), pf.PF_SHEET_GIVEN_S0)
        return S @ f.cpu().numpy()

    e = ew(X, Y, G)
    unit = [ew(*(torch.tensor([v], dtype=torch.float64, device="cuda") for v in (a, b, 1.0))) for a, b in zip(Xn, Yn)]
    scale = np.abs(S).sum(1).max()

    shift = float(np.dot(ds * f0, sb)) / g0          # the Kutta modes' s0 is that of P^Gamma s'_b (Eq. kuttasystem)

    def check(f, s0, gam, circ, edges):
        f = f.cpu().numpy()
        rhs = sb - s0 - (shift if edges else 0.0) + e + sum(g * u for g, u in zip(gam, unit))
        tol = 1e-13 * (scale * np.abs(f).max() + np.abs(rhs).max())
        assert np.abs(S @ f - rhs).max() < tol
        if circ is not None:
            assert abs(np.dot(ds, f) + sum(gam) - circ) < 1e-13 * (np.dot(ds, np.abs(f)) + abs(s0 * g0) + 1.0)
        for k in edges:
            assert abs(f[k]) < 1e-12 * (np.abs(f).max() + abs(s0) * np.abs(f0).max())

    solve = lambda *a, **k: pf.pf_sheet_solve_vortices(plan, sch, X, Y, G, motion, *a, **k)     # noqa: E731
    f, _, s0 = solve(pf.PF_SHEET_GIVEN_S0, 0.4)
    assert s0 == 0.4
    check(f, s0, [], None, [])
    f, _, s0 = solve(pf.PF_SHEET_CIRCULATION, -0.7)
    check(f, s0, [], -0.7, [])
    k = (0, ns // 2)
    f, _, s0 = solve(pf.PF_SHEET_KUTTA_STEADY, edges=k[:1])
    assert abs(f[k[0]].item()) < 1e-12 * (float(f.abs().max()) + abs(s0) * np.abs(f0).max())
    gw = float(G.sum())
    f, gam, s0 = solve(pf.PF_SHEET_KUTTA_SHED, gw, edges=k[:1], Xnew=Xn[:1], Ynew=Yn[:1])
    check(f, s0, gam, -gw, k[:1])
    f, gam, s0 = solve(pf.PF_SHEET_KUTTA_SHED, gw, edges=k, Xnew=Xn, Ynew=Yn)
    check(f, s0, gam, -gw, k)
    pf.pf_sync(plan)


@pytest.mark.parametrize("n,outside", [(0, 0), (1, 0), (63, 3), (64, 0), (65, 1), (1000, 20), (5000, 0)])
def test_vortex_sum_equals_the_field_sum(n, outside):
    plan = pf.Plan(*GRID, pf.PF_FP64)
    x, y, ds = _circle(90)
    sch = pf.pf_schur_factor(plan, x, y, ds)
    _, _, S = pf.pf_schur_info(sch)
    X, Y, G = _vortices(n, 5 + n, outside)
    f, _, s0 = pf.pf_sheet_solve_vortices(plan, sch, X, Y, G, (0, 0, 0, 1.0, 0), pf.PF_SHEET_CIRCULATION, 0.1)
    w = pf.pf_regularize(plan, X, Y, G)
    for route in (pf.PF_RHS_FFT, pf.PF_RHS_SPARSE):
        pf.pf_plan_set_rhs_route(plan, route)
        fw, _, s0w = pf.pf_sheet_solve(plan, sch, w, (0, 0, 0, 1.0, 0), pf.PF_SHEET_CIRCULATION, 0.1)
        tol = np.linalg.cond(S) * 1e-14
        assert float((f - fw).norm()) <= tol * float(fw.norm()) and abs(s0 - s0w) <= tol * max(1.0, abs(s0w))
