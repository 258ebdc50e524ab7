"""Steps of small sets at the edges of what they take: no vortices at all, and
vortices off the grid, whose count is the same by every route of a step."""
import numpy as np
import pytest

import paper_2102_11910_gb300 as pf
from paper_2102_11910_gb300 import inputs

pytestmark = pytest.mark.gpu


def _plan(prec):
    g = inputs.centred_grid(72, 72, 0.025)
    return pf.Plan(g.nx, g.ny, g.dx, g.x0, g.y0, prec)


def _ellipse(edges=()):
    e = inputs.ellipse(40, 0.45, 0.15)
    return pf.BodyKinematics(e.x, e.y, e.ds, edges, amp=0.1, omega=1.0, Uinf=1.0)


@pytest.mark.parametrize("prec", [pf.PF_FP64, pf.PF_MIXED])
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("body", ["none", "one", "multi"])
def test_a_step_without_vortices(prec, scheme, body):
    plan = _plan(prec)
    state = pf.State(plan, 64)
    pf.pf_state_set(state, np.zeros(0), np.zeros(0), np.zeros(0), 0.0)
    if body == "multi":
        pf.pf_step_multi(plan, state, 0.01, [_ellipse()], scheme)
    else:
        pf.pf_step(plan, state, 0.01, _ellipse() if body == "one" else None, scheme)
    assert pf.pf_sync(plan) == 0
    X, _, _, t = pf.pf_state_get(state)
    assert len(X) == 0 and t == 0.01


# capacities: the vortex sum with the one-launch transfers, the field's right-hand side with them (ns x
# capacity past the sum's limit), the same with binned ones
@pytest.mark.parametrize("prec", [pf.PF_FP64, pf.PF_MIXED])
@pytest.mark.parametrize("multi", [False, True])
@pytest.mark.parametrize("capacity", [256, 2048, 1 << 14, 1 << 17])
def test_vortices_off_the_grid_are_counted_alike(prec, multi, capacity):
    plan = _plan(prec)
    rng = np.random.default_rng(8)
    a = rng.uniform(0, 2 * np.pi, 130)
    X, Y = 0.7 * np.cos(a), 0.7 * np.sin(a)
    X[[3, 64, 129]], Y[70] = 5.0, -7.0                             # four of them
    state = pf.State(plan, capacity)
    pf.pf_state_set(state, X, Y, rng.normal(0.0, 0.02, 130), 0.0)
    if multi:
        pf.pf_step_multi(plan, state, 0.01, [_ellipse()], 1)
    else:
        pf.pf_step(plan, state, 0.01, _ellipse(), 1)
    with pytest.raises(pf.GridPfError, match=" 16 points"):        # R_v twice in each of two stages
        pf.pf_sync(plan)
