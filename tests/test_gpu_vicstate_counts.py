"""The state's tile counts are cleared by the step that read them last: after a
set call, whatever number of steps came before it, a state goes on as a new one
does, bitwise.  The mixed advance packs the moved records of a tile: sets whose
tiles hold one record, whole and partial rows of 32, and more than one chunk."""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu


def _set(n, seed, nx, ny, dx):
    rng = np.random.default_rng(seed)
    return [torch.from_numpy(a).cuda() for a in (dx * (8 + (nx - 16) * rng.random(n)), dx * (8 + (ny - 16) * rng.random(n)),
                                                 rng.normal(0.0, 1e-4, n))]


def _run(st, plan, vortices, steps):
    pf.pf_vic_state_set(st, *vortices)
    for _ in range(steps):
        pf.pf_vic_step(st, 0.02, 0.3, -0.2)
    X, Y, G, nv, _ = pf.pf_vic_state_get(st)
    assert pf.pf_sync(plan) == 0 and nv == len(vortices[0])
    return X.clone(), Y.clone(), G.clone()


@pytest.mark.parametrize("prec", [pf.PF_FP64, pf.PF_MIXED])
@pytest.mark.parametrize("before", [0, 1, 2])
@pytest.mark.parametrize("n", [1, 33, 2500, 40000])
def test_a_set_after_any_number_of_steps(prec, before, n):
    nx, ny, dx = 131, 100, 0.01
    plan = pf.Plan(nx, ny, dx, 0.0, 0.0, prec)
    used, fresh = pf.VicState(plan, 40000), pf.VicState(plan, 40000)
    _run(used, plan, _set(3000, 5, nx, ny, dx), before)
    v = _set(n, n, nx, ny, dx)
    got, ref = _run(used, plan, v, 3), _run(fresh, plan, v, 3)
    for a, b in zip(got, ref):
        assert torch.equal(a, b)
    # the first step against the stateless velocity: 24-bit cell fractions (mixed) or FP64 rounding of the move
    one = _run(used, plan, v, 1)
    u, w = pf.pf_vic_velocity(plan, *v, 0.3, -0.2)
    tol = dx * 2.0 ** -22 if prec == pf.PF_MIXED else 1e-13
    for a, x, d in ((one[0], v[0], u), (one[1], v[1], w)):
        assert float((a - x - 0.02 * d.double()).abs().max()) <= tol + 0.02 * (1e-5 if prec == pf.PF_MIXED else 1e-12)
