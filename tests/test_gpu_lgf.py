"""The plan's LGF table at the edges of the tiles that form it and of the square
that is mirrored, against the oracle's own quadrature (sums of some 500 positive
terms on both sides: 500 roundings of the largest value cover them)."""
import numpy as np
import pytest

import paper_2102_11910_gb300 as pf
from oracle.lgf import lgf_table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(8, 8), (8, 200), (200, 8), (31, 31), (32, 31), (31, 32), (33, 40), (40, 33), (63, 64),
                                   (95, 301), (301, 95)])
def test_table(nx, ny):
    plan = pf.Plan(nx, ny, 0.1, 0.0, 0.0, pf.PF_FP64)
    G = pf.pf_lgf_table(plan)                                  # [n, m]
    ref = lgf_table(nx, ny).T
    assert G.shape == ref.shape and G[0, 0] == 0.0
    assert np.abs(G - ref).max() <= 500 * 2.0 ** -53 * ref.max()
    k = min(nx, ny) + 1
    assert np.array_equal(G[:k, :k], G[:k, :k].T)
