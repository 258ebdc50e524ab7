"""The mixed deposit adds the FP32 product of strength and weights, rounded, as an
integer: w is the exact sum of those products, rounded once.  (A state's FP64
positions follow w's bits, so the terms' rounding is part of the result.)"""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pairs", [1, 40, 400])           # tiles below and above the count that is sorted
def test_w_is_the_sum_of_rounded_products(pairs):
    n = 132
    plan = pf.Plan(n, n, 1.0, 0.0, 0.0, pf.PF_MIXED)       # dx = 1: w in the deposit's own units
    rng = np.random.default_rng(pairs)
    # two vortices at the centres of cells six apart, where the weights are -1/16, 9/16, 9/16, -1/16, exactly
    ci, cj = np.meshgrid(4 + 6 * np.arange(20), 4 + 6 * np.arange(20))
    ci, cj = ci.ravel()[:pairs], cj.ravel()[:pairs]
    g = rng.uniform(0.5, 1.0, (2, pairs)).astype(np.float32)
    X, Y = np.tile(ci + 0.5, 2), np.tile(cj + 0.5, 2)
    w = pf.pf_regularize(plan, *[torch.from_numpy(a).cuda() for a in (X, Y, g.ravel().astype(np.float64))]).cpu().numpy()
    assert pf.pf_sync(plan) == 0
    m = np.array([-1, 9, 9, -1], dtype=np.float32) / np.float32(16)
    for b in range(4):
        gy = g * m[b]                                      # rounded to FP32
        for a in range(4):
            if a in (0, 3) and b in (0, 3):
                continue                                   # |x| < 2^-8: may have bits below the tile's unit, 2^-31 here
            x = (gy * m[a]).astype(np.float64)             # rounded to FP32
            ref = (x[0] + x[1]).astype(np.float32)
            assert np.array_equal(w[cj - 1 + b, ci - 1 + a], ref)
