"""The node velocity written to a slice of a larger buffer, at any word: the same
values as in a buffer of its own, and nothing beside them."""
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [pf.PF_FP64, pf.PF_MIXED])
@pytest.mark.parametrize("nx,ny", [(20, 17), (140, 131)])                    # shared-memory and register passes
def test_outputs_at_any_word(prec, nx, ny):
    plan = pf.Plan(nx, ny, 0.02, 0.0, 0.0, prec)
    g = torch.Generator(device="cuda")
    g.manual_seed(nx)
    w = torch.randn(ny, nx, dtype=plan.dtype, device="cuda", generator=g)
    want = pf.pf_velocity_solve(plan, w, 1.0, -0.5).reshape(-1).clone()
    for off in range(4):
        buf = torch.full((2 * nx * ny + 8,), 7.0, dtype=plan.dtype, device="cuda")
        pf.pf_velocity_solve(plan, w, 1.0, -0.5, buf[off:off + 2 * nx * ny])
        pf.pf_sync(plan)
        assert torch.equal(buf[off:off + 2 * nx * ny], want)
        assert bool((buf[:off] == 7.0).all()) and bool((buf[off + 2 * nx * ny:] == 7.0).all())
