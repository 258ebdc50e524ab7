"""The mixed path's interpolation at arbitrary points, eight lanes a point,
against the stencil sum in numpy."""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu


def _m4p(f):
    return np.stack([-0.5 * f * (1 - f) ** 2, 1 - 2.5 * f ** 2 + 1.5 * f ** 3,
                     1 - 2.5 * (1 - f) ** 2 + 1.5 * (1 - f) ** 3, -0.5 * (1 - f) * f ** 2])


# a lone point, less and more than a warp and a block, more than one round of the largest grid (152 x 16 blocks of 128)
@pytest.mark.parametrize("nq", [1, 31, 33, 129, 152 * 16 * 128 + 45])
def test_mixed_points(nq):
    nx, ny, dx = 70, 51, 0.01
    plan = pf.Plan(nx, ny, dx, -0.1, 0.2, pf.PF_MIXED)
    rng = np.random.default_rng(nq)
    uv = rng.normal(size=(ny, nx, 2)).astype(np.float32)
    gx, gy = 1 + (nx - 3) * rng.random(nq), 1 + (ny - 3) * rng.random(nq)
    gx[0], gy[0] = nx - 3 + 0.75, 1.0                              # last and first cells
    bad = rng.random(nq) < (0.2 if nq > 1 else 0)
    gx[bad] = rng.choice([-1e9, 0.5, nx - 1.5, np.nan, np.inf, 1e300], int(bad.sum()))
    out = [torch.empty(nq + 8, dtype=torch.float32, device="cuda").fill_(7.0) for _ in range(2)]
    u, v = pf.pf_interpolate(plan, torch.from_numpy(uv).cuda(), torch.from_numpy(-0.1 + dx * gx).cuda(),
                             torch.from_numpy(0.2 + dx * gy).cuda(), out[0][:nq], out[1][:nq])
    if bad.any():
        with pytest.raises(pf.GridPfError, match=rf"\b{int(bad.sum())}\b"):
            pf.pf_sync(plan)
    else:
        assert pf.pf_sync(plan) == 0
    assert all(bool((o[nq:] == 7.0).all()) for o in out)
    ok = ~bad
    X, Y = (-0.1 + dx * gx[ok] + 0.1) / dx, (0.2 + dx * gy[ok] - 0.2) / dx
    ci, cj = np.floor(X).astype(int), np.floor(Y).astype(int)
    wx, wy = _m4p(X - ci), _m4p(Y - cj)
    for o, c in ((u, 0), (v, 1)):
        o = o.cpu().numpy()
        ref = sum(wx[a] * wy[b] * uv[cj - 1 + b, ci - 1 + a, c] for a in range(4) for b in range(4))
        # weights |w| <= 1 to 6 roundings of terms up to 2.5 each, 16 terms of |uv| < 6, and the fraction's 2^-24
        assert np.abs(o[ok] - ref).max() <= 6 * 16 * 2 * 15 * 2.0 ** -24
        assert (o[bad] == 0).all()
