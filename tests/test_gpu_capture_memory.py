"""A captured step reserves what its own route reads: one that sums from the
vortices allocates no streamfunction and spectra for the field's route."""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu

N = 1024
SPECTRUM = (N + 1) * N * 16                              # bytes of one 64-bit half spectrum of the padded torus


def _batch(route):
    dx = 2.54 / (N - 1)
    plan = pf.Plan(N, N, dx, -1.27, -1.27, pf.PF_MIXED, stream=torch.cuda.Stream())
    if route is not None:
        pf.pf_plan_set_rhs_route(plan, route)
    rng = np.random.default_rng(0)
    state = pf.State(plan, 2000)
    pf.pf_state_set(state, rng.uniform(0.7, 1.1, 1900), rng.uniform(-0.5, 0.5, 1900), rng.normal(0.0, 1e-3, 1900))
    xi = -1.0 + (2.0 * np.arange(1, 65) - 1.0) / 64
    body = pf.BodyKinematics(0.5 * xi, np.zeros(64), np.full(64, 1.0 / 64), (0, 63), 0.2, Uinf=1.0)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    batch = pf.Batch([plan], [state], [body], 0.1 * dx)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    batch.step(2)
    pf.pf_sync(plan)
    assert len(pf.pf_state_get(state)[0]) == 1904
    return used, batch


def test_vortex_sums_reserve_no_spectra():
    keep = _batch(None)                                   # the library's one-time allocations
    used, b1 = _batch(None)
    field, b2 = _batch(pf.PF_RHS_FFT)
    assert field >= 2 * SPECTRUM > SPECTRUM > used
    assert keep and b1 and b2
