"""The one-launch R_v and E_v of small sets against the binned passes: the same
w bitwise (the sums are integers), the same velocities to rounding (the stencil's
rows are added in pairs), at the edges of the rule that chooses them."""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu


def _set(n, nx, ny, dx, seed, clustered):
    rng = np.random.default_rng(seed)
    X = dx * (0.3 + (nx - 1.6) * rng.random(n))                # some stencils leave the grid
    Y = dx * (0.3 + (ny - 1.6) * rng.random(n))
    if clustered:
        X[: n // 2], Y[: n // 2] = dx * (33.0 + 6.0 * rng.random(n // 2)), dx * (20.0 + rng.random(n // 2))
    return X, Y, rng.normal(0.0, 0.3, n)


def _oob(plan):
    try:
        return pf.pf_sync(plan)
    except pf.GridPfError as e:
        return int(str(e).split("PF_ERR_OUT_OF_DOMAIN")[-1].split(":")[-1].split()[0])


# the largest direct counts (4096 mixed, 2048 FP64) and the ones next to them; one vortex; a cluster of
# more than 256 records a tile; tiles x vortices at 2^20 and past it (32 x 33 tiles)
@pytest.mark.parametrize("prec", [pf.PF_FP64, pf.PF_MIXED])
@pytest.mark.parametrize("nx,ny,n,tile,clustered", [(70, 50, 1, 32, False), (100, 131, 2047, 32, True), (100, 131, 2048, 16, True),
                                                    (100, 131, 4096, 32, True), (100, 131, 4097, 32, False),
                                                    (1024, 1040, 992, 32, False), (1024, 1040, 993, 32, False)])
def test_direct_equals_binned(prec, nx, ny, n, tile, clustered):
    dx = 0.01
    plan = pf.Plan(nx, ny, dx, 0.0, 0.0, prec)
    pf.pf_launch_config_set(plan, tile=tile)
    X, Y, G = _set(n, nx, ny, dx, n + nx, clustered)
    # the same set with vortices of strength zero outside the grid appended takes the binned passes
    m = 4200
    far = np.full(m, -5.0)
    small = [torch.from_numpy(a).cuda() for a in (X, Y, G)]
    large = [torch.from_numpy(np.concatenate([a, b])).cuda() for a, b in ((X, far), (Y, far), (G, np.zeros(m)))]
    w = pf.pf_regularize(plan, *small)
    outside = _oob(plan)
    ref = pf.pf_regularize(plan, *large)
    assert _oob(plan) == outside + m
    assert torch.equal(w, ref)
    u, v = pf.pf_vic_velocity(plan, *small, 1.0, -0.5)
    assert _oob(plan) == outside
    ru, rv = pf.pf_vic_velocity(plan, *large, 1.0, -0.5)
    _oob(plan)
    tol = 1e-14 if prec == pf.PF_FP64 else 1e-6               # 8 roundings of a row sum and the weights' forms
    for a, b in ((u, ru[:n]), (v, rv[:n])):
        assert float((a - b).double().norm()) <= tol * float(b.double().norm())
        assert torch.equal(a == 0, b == 0)                     # those off the grid


@pytest.mark.parametrize("prec", [pf.PF_FP64, pf.PF_MIXED])
def test_tuning_a_small_set_after_a_large_one(prec):
    """The tuner times the route that the set takes: nothing of the larger set's bins is read."""
    plan = pf.Plan(100, 90, 0.01, 0.0, 0.0, prec)
    pf.pf_regularize(plan, *[torch.from_numpy(a).cuda() for a in _set(20000, 100, 90, 0.01, 3, False)])
    _oob(plan)
    pf.pf_autotune(plan, 300, reps=1)
    assert pf.pf_sync(plan) == 0
