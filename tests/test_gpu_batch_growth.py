"""A batch's captured steps go on after their plan has binned a set that outgrew
its buffers: they hold the addresses of those it had."""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu

N = 200
DX = 2.54 / (N - 1)


def _instance(nv, prec):
    plan = pf.Plan(N, N, DX, -1.27, -1.27, prec, stream=torch.cuda.Stream())
    pf.pf_plan_set_rhs_route(plan, pf.PF_RHS_FFT)
    rng = np.random.default_rng(nv)
    state = pf.State(plan, nv + 16)
    pf.pf_state_set(state, rng.uniform(0.6, 1.1, nv), rng.uniform(-0.5, 0.5, nv), rng.normal(0.0, 1e-4, nv))
    xi = -1.0 + (2.0 * np.arange(1, 41) - 1.0) / 40
    return plan, state, pf.BodyKinematics(0.5 * xi, np.zeros(40), np.full(40, 1.0 / 40), (0, 39), 0.2, Uinf=1.0)


# states of the one-pass binning and of the three passes (FP64: the three passes for both)
@pytest.mark.parametrize("prec", [pf.PF_FP64, pf.PF_MIXED])
@pytest.mark.parametrize("nv", [6000, 70000])
def test_captured_steps_outlive_the_buffers_growth(nv, prec):
    plan, state, body = _instance(nv, prec)
    other, twin, _ = _instance(nv, prec)
    batch = pf.Batch([plan], [state], [body], 0.1 * DX)
    batch.step(1)
    pf.pf_sync(plan)
    rng = np.random.default_rng(1)
    big = [torch.from_numpy(rng.uniform(-1.0, 1.0, 400000)).cuda() for _ in range(3)]
    torch.cuda.synchronize()
    pf.pf_vic_velocity(plan, *big)
    pf.pf_sync(plan)
    batch.step(2)
    pf.pf_sync(plan)
    for _ in range(3):
        pf.pf_step(other, twin, 0.1 * DX, body, 0)
    pf.pf_sync(other)
    for a, b in zip(pf.pf_state_get(state)[:3], pf.pf_state_get(twin)[:3]):
        assert np.array_equal(a, b)
