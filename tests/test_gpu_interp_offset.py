"""E_v of a caller's field that does not start on a pair of words: a slice of a
larger buffer is a field like any other, and gives the same velocities."""
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [pf.PF_FP64, pf.PF_MIXED])
@pytest.mark.parametrize("nq", [1, 31, 4099])
def test_fields_at_any_word(prec, nq):
    nx, ny, dx = 90, 61, 0.02
    plan = pf.Plan(nx, ny, dx, 0.0, 0.0, prec)
    g = torch.Generator(device="cuda")
    g.manual_seed(nq)
    buf = torch.randn(2 * nx * ny + 4, dtype=plan.dtype, device="cuda", generator=g)
    r = torch.rand(2, nq, dtype=torch.float64, device="cuda", generator=g)
    X, Y = dx * (1.5 + (nx - 4.5) * r[0]), dx * (1.5 + (ny - 4.5) * r[1])
    for off in range(4):
        uv = buf[off:off + 2 * nx * ny]
        got, want = pf.pf_interpolate(plan, uv, X, Y), pf.pf_interpolate(plan, uv.clone(), X, Y)
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    pf.pf_sync(plan)
