"""The tile-ordered state on plans of every launch configuration: it bins in its
own tiles and blocks, so its steps are those of a plan left at the default, and
the plan's buffers have to have room for them."""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu

GRID = (300, 260, 0.01, 0.0, 0.0)


def _steps(plan, nv):
    rng = np.random.default_rng(nv)
    X, Y = (0.01 * (2.0 + (n - 6.0) * rng.random(nv)) for n in GRID[:2])
    state = pf.VicState(plan, nv)
    pf.pf_vic_state_set(state, *(torch.from_numpy(a).cuda() for a in (X, Y, rng.normal(0.0, 1e-3, nv))))
    for _ in range(2):
        pf.pf_vic_step(state, 1e-4, 1.0, 0.0)
    pf.pf_sync(plan)
    return [t.clone() for t in pf.pf_vic_state_get(state)[:3]]


@pytest.mark.parametrize("prec", [pf.PF_FP64, pf.PF_MIXED])
@pytest.mark.parametrize("tile,span", [(32, 256), (32, 4096), (16, 2048), (16, 4096)])
@pytest.mark.parametrize("nv", [1500, 100000])
def test_states_do_not_depend_on_the_plans_configuration(prec, tile, span, nv):
    want = _steps(pf.Plan(*GRID, prec), nv)
    plan = pf.Plan(*GRID, prec)
    pf.pf_launch_config_set(plan, tile=tile, min_span=span)
    clone = pf.pf_plan_clone(plan, prec, torch.cuda.Stream())       # takes the configuration, with buffers of its own
    for p in (plan, clone):
        torch.cuda.synchronize()
        for a, b in zip(_steps(p, nv), want):
            assert torch.equal(a, b)
        pf.pf_sync(p)
        torch.cuda.synchronize()
