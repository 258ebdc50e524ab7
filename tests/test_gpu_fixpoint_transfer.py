"""The 64-bit transfers in fixed point (R_v and E_v of FP64 plans) where they
could go wrong: cell fractions at both ends, one record and many in a tile,
strengths of very different size, values that are not finite, positions whose
quotient (X - x0)/dx is hard to round.

R_v rounds a node's sum to 2^-58 of count x max|Gamma|, E_v a velocity to 2^-57
of the tile's largest, both on top of the weights' 2^-60 and of the FP64
reference's own 2^-52 a term: 1e-14 in the 2-norm covers all of it here."""
import numpy as np
import pytest
import torch

import paper_2102_11910_gb300 as pf
from oracle import vic as OV

pytestmark = pytest.mark.gpu

TOL = 1e-14


def _rel(a, b):
    m = np.abs(b).max()                          # squares of 1e-200 would vanish
    return float(np.linalg.norm((np.asarray(a) - b) / m) / np.linalg.norm(b / m))


def _dev(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


def _check(nx, ny, dx, x0, y0, X, Y, G, tile=None):
    plan = pf.Plan(nx, ny, dx, x0, y0, pf.PF_FP64)
    if tile:
        pf.pf_launch_config_set(plan, tile=tile)
    og = OV.Grid(nx, ny, dx, x0, y0)
    w = pf.pf_regularize(plan, *_dev(X, Y, G))
    assert _rel(w.cpu().numpy(), OV.regularize(og, X, Y, G)) < TOL
    uq, vq = pf.pf_vic_velocity(plan, *_dev(X, Y, G), 1.0, 0.5)         # E_v by tiles
    uv = pf.pf_velocity_solve(plan, w, 1.0, 0.5)
    up, vp = pf.pf_interpolate(plan, uv, *_dev(X, Y))                   # E_v at points, FP64 arithmetic
    pf.pf_sync(plan)
    assert _rel(uq.cpu().numpy(), up.cpu().numpy()) < TOL and _rel(vq.cpu().numpy(), vp.cpu().numpy()) < TOL


@pytest.mark.parametrize("tile", [16, 32])
@pytest.mark.parametrize("n", [1, 7, 8, 255, 3000])
def test_counts_a_tile(n, tile):
    rng = np.random.default_rng(n)
    X, Y = rng.uniform(0.02, 0.3, n), rng.uniform(0.02, 0.3, n)          # one or a few tiles of a 96 x 70 grid
    _check(96, 70, 0.01, 0.0, 0.0, X, Y, rng.normal(0.0, 1.0, n), tile)


def test_fractions_at_both_ends_of_a_cell():
    i = np.arange(1.0, 60.0)
    X = np.concatenate([i, np.nextafter(i + 1, 0), i + 2.0 ** -40, i + 0.5])
    Y = np.concatenate([np.nextafter(i + 1, 0), i, i + 0.5, i + 2.0 ** -40])[::-1].copy()
    X, Y = np.clip(X, 1.0, 61.0), np.clip(Y, 1.0, 61.0)
    _check(64, 64, 1.0, 0.0, 0.0, X, Y, np.linspace(-1.0, 2.0, len(X)))


@pytest.mark.parametrize("dx", [1.0 / 3.0, 2.0 / 1023, 0.1, np.nextafter(1.0, 0.0), np.nextafter(0.5, 1.0)])
def test_quotients_match_the_division(dx):
    """A position's cell and fraction are those of (X - x0)/dx rounded once: compared
    with the oracle, whose weights come from that quotient, to the last bits."""
    rng = np.random.default_rng(9)
    n, x0 = 4000, -0.7
    k = rng.integers(1, 120, n).astype(float)
    X = x0 + dx * np.where(np.arange(n) % 2, k, k + rng.random(n))
    Y = x0 + dx * rng.uniform(1.0, 120.0, n)
    g = (X - x0) / dx
    ok = (g >= 1.0) & (g < 122.0)
    _check(124, 124, dx, x0, x0, X[ok], Y[ok], rng.normal(0.0, 1.0, int(ok.sum())))


def test_strengths_of_very_different_size():
    rng = np.random.default_rng(4)
    n = 500
    G = rng.normal(0.0, 1.0, n) * 10.0 ** rng.integers(-30, 31, n)
    _check(80, 80, 0.02, -0.8, -0.8, rng.uniform(-0.7, 0.7, n), rng.uniform(-0.7, 0.7, n), G)
    _check(80, 80, 0.02, -0.8, -0.8, rng.uniform(-0.7, 0.7, n), rng.uniform(-0.7, 0.7, n), 1e-200 * rng.normal(0.0, 1.0, n))


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_strengths_that_are_not_finite_show(bad):
    plan = pf.Plan(128, 128, 0.02, -1.28, -1.28, pf.PF_FP64)
    X, Y, G = np.array([-0.5, 0.61]), np.array([-0.4, 0.63]), np.array([1.0, bad])
    w = pf.pf_regularize(plan, *_dev(X, Y, G)).cpu().numpy()
    assert np.isnan(w[96, 96]) and np.isnan(w).sum() <= 4 * 32 * 32       # its own tiles
    u, v = pf.pf_vic_velocity(plan, *_dev(X, Y, G))
    assert bool(torch.isnan(u).all()) and bool(torch.isnan(v).all())
    u, v = pf.pf_vic_velocity(plan, *_dev(X, Y, np.ones(2)), float("inf"), 0.0)   # an infinite stream: FP64 sums
    assert not bool(torch.isfinite(u).any()) and bool(torch.isfinite(v).all())
