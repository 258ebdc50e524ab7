"""E_v of FP64 plans on vortices in a stream: the component across the stream
is as it would be without it, to the last bit, however small beside it, and both
components are those of E_v at points (FP64 sums) to 1e-14 of their own norm."""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu


# one launch for small sets, tiles for larger ones
@pytest.mark.parametrize("n", [1500, 5000])
@pytest.mark.parametrize("strength", [1e-6, 1e-3, 1e12])
@pytest.mark.parametrize("tile", [16, 32])
def test_a_stream_along_one_axis_leaves_the_other_component(n, strength, tile):
    nx, ny, dx = 256, 200, 0.01
    plan = pf.Plan(nx, ny, dx, -1.28, -1.0, pf.PF_FP64)
    pf.pf_launch_config_set(plan, tile=tile)
    rng = np.random.default_rng(n)
    dev = [torch.from_numpy(a).cuda() for a in (rng.uniform(-1.2, 1.2, n), rng.uniform(-0.9, 0.9, n),
                                                strength * rng.normal(0.0, 1.0, n))]
    w = pf.pf_regularize(plan, *dev)

    def both(U, V):
        q = [t.clone() for t in pf.pf_vic_velocity(plan, *dev, U, V)]
        p = pf.pf_interpolate(plan, pf.pf_velocity_solve(plan, w, U, V), *dev[:2])
        pf.pf_sync(plan)
        for a, b in zip(q, p):
            assert float((a - b).norm()) <= 1e-14 * float(b.norm())
        return q

    rest, along_x, along_y = both(0.0, 0.0), both(1.0, 0.0), both(0.0, 1.0)
    assert torch.equal(along_x[1], rest[1]) and torch.equal(along_y[0], rest[0])
