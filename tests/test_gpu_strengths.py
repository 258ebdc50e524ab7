"""Strengths that are not finite, by every route of R_v: the tiles that hold the
vortex's stencil are NaN, the other nodes are as they are without it, to the
rounding of their fixed-point sums (1e-13 FP64, 1e-6 mixed, as against the
oracle), and the velocities, which every node reaches, are NaN."""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu

GRID = (300, 200, 0.01, 0.0, 0.0)


def _dev(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


def _set(n, bad):
    rng = np.random.default_rng(n)
    X, Y, G = rng.uniform(0.05, 2.9, n), rng.uniform(0.05, 1.9, n), rng.normal(0.0, 1.0, n)
    X[1], Y[1], G[1] = 1.105, 0.505, bad                     # cell (110, 50): its stencil lies in one tile
    return X, Y, G


# one launch, one-pass binning, three passes; a double beyond FP32 is an infinity to a mixed plan
@pytest.mark.parametrize("n", [2, 5000, 70000])
@pytest.mark.parametrize("prec,bad", [(p, b) for p in (pf.PF_FP64, pf.PF_MIXED) for b in (np.nan, np.inf, -np.inf)] +
                         [(pf.PF_MIXED, -1e39)])
def test_strengths_that_are_not_finite(prec, bad, n):
    plan = pf.Plan(*GRID, prec)
    X, Y, G = _set(n, bad)
    w = pf.pf_regularize(plan, *_dev(X, Y, G)).cpu().numpy()
    keep = np.arange(n) != 1
    ref = pf.pf_regularize(plan, *_dev(X[keep], Y[keep], G[keep])).cpu().numpy()
    hit = np.zeros(w.shape, dtype=bool)
    hit[32:64, 96:128] = True
    assert np.array_equal(np.isnan(w), hit)
    assert np.linalg.norm((w - ref)[~hit]) <= (1e-13 if prec == pf.PF_FP64 else 1e-6) * np.linalg.norm(ref[~hit])
    for q in pf.pf_vic_velocity(plan, *_dev(X, Y, G), 1.0, 0.0):
        assert bool(torch.isnan(q).all())
    pf.pf_sync(plan)


@pytest.mark.parametrize("prec", [pf.PF_FP64, pf.PF_MIXED])
def test_in_the_tile_ordered_state(prec):
    n = 3000
    plan = pf.Plan(*GRID, prec)
    state = pf.VicState(plan, n)
    pf.pf_vic_state_set(state, *_dev(*_set(n, np.nan)))
    u, v = (torch.zeros(n, dtype=plan.dtype, device="cuda") for _ in range(2))
    pf.pf_vic_step(state, 0.0, 1.0, 0.0, u, v)
    torch.cuda.synchronize()
    assert bool(torch.isnan(u).all()) and bool(torch.isnan(v).all())
