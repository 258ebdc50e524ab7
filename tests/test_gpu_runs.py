"""The one-pass binning of middling mixed sets against the three passes of
larger ones: the same w and the same velocities, bitwise (the sums are integers
and a record's stencil does not depend on where the record is kept)."""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu


def _dev(*a):
    return [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in a]


def _oob(plan):
    try:
        return pf.pf_sync(plan)
    except pf.GridPfError as e:
        return int(str(e).split("PF_ERR_OUT_OF_DOMAIN")[-1].split(":")[-1].split()[0])


# the smallest and largest counts of the route; last blocks of one and of many vortices; spans from the
# plan's least to above it; sets within one tile and over all, on a grid of ragged tiles
@pytest.mark.parametrize("nv,tile,min_span,spread", [(4097, 32, 1024, 1.0), (4097, 16, 4096, 0.02), (8193, 32, 256, 1.0),
                                                     (20011, 16, 1024, 1.0), (20011, 32, 2048, 0.02), (65535, 32, 4096, 1.0),
                                                     (65536, 32, 1024, 0.3)])
def test_runs_equal_the_three_passes(nv, tile, min_span, spread):
    nx, ny, dx = 150, 131, 0.01
    plan = pf.Plan(nx, ny, dx, 0.0, 0.0, pf.PF_MIXED)
    pf.pf_launch_config_set(plan, tile=tile, min_span=min_span)
    rng = np.random.default_rng(nv + tile)
    X, Y = (dx * (0.3 + 0.5 * (1 - spread) * n + spread * (n - 1.6) * rng.random(nv)) for n in (nx, ny))
    G = rng.normal(0.0, 0.3, nv)
    m = 65537                                            # off the grid, of no strength: with them the set is a large one
    far, none = np.full(m, -5.0), np.zeros(m)
    small, large = _dev(X, Y, G), _dev(*(np.concatenate(p) for p in ((X, far), (Y, far), (G, none))))
    w = pf.pf_regularize(plan, *small)
    outside = _oob(plan)
    assert torch.equal(w, pf.pf_regularize(plan, *large))
    assert _oob(plan) == outside + m
    u, v = pf.pf_vic_velocity(plan, *small, 1.0, -0.5)
    assert _oob(plan) == outside
    ru, rv = pf.pf_vic_velocity(plan, *large, 1.0, -0.5)
    _oob(plan)
    assert torch.equal(u, ru[:nv]) and torch.equal(v, rv[:nv])
    assert torch.equal(pf.pf_vic_velocity(plan, *small, 1.0, -0.5)[0], u)          # after the other layout
    _oob(plan)
