"""Launch configurations by each route of R_v: one launch, the one-pass binning of
middling mixed sets, the three passes of larger ones (100,000).  Span and threads of
the plan change no bit of any; each matches the oracle to the precision's tolerance."""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf
from oracle import vic as OV
from paper_2102_11910_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL_W = {pf.PF_FP64: 1e-13, pf.PF_MIXED: 1e-6}
TOL_U = {pf.PF_FP64: 1e-12, pf.PF_MIXED: 1e-5}


def _rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("prec", [pf.PF_FP64, pf.PF_MIXED])
@pytest.mark.parametrize("nv", [2000, 50000, 100000])
@pytest.mark.parametrize("tile,fft", [(32, 0), (16, 0), (16, 1)])
def test_configurations_by_route(prec, nv, tile, fft):
    g = inputs.centred_grid(300, 200, 2.0 / 299)                          # ragged last tiles
    rng = np.random.default_rng(nv)
    X, Y, G = inputs.uniform_vortices(rng, nv, -0.85, 0.85, 1e-4, -0.55, 0.55)
    og = OV.Grid(g.nx, g.ny, g.dx, g.x0, g.y0)
    w_ref = OV.regularize(og, X, Y, G)
    _, _, ur, vr = OV.vortex_velocity(og, X, Y, G, 0.25, -0.1)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (X, Y, G)]
    plan = pf.Plan(g.nx, g.ny, g.dx, g.x0, g.y0, prec)
    first = None
    for span in (256, 512, 1024, 2048, 4096):
        for threads in (128, 256):
            pf.pf_launch_config_set(plan, tile=tile, min_span=span, tile_threads=threads, fft=fft)
            out = [pf.pf_regularize(plan, *dev).clone()]
            out += [t.clone() for t in pf.pf_vic_velocity(plan, *dev, 0.25, -0.1)]
            pf.pf_sync(plan)
            if first is None:
                first = out
                assert _rel(out[0].cpu().numpy(), w_ref) < TOL_W[prec]
                assert _rel(torch.cat(out[1:]).cpu().numpy(), np.concatenate([ur, vr])) < TOL_U[prec]
            assert all(torch.equal(a, b) for a, b in zip(out, first))
