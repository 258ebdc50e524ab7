"""The 64-bit convolution passes (block fixed point) against torch's FP64 FFT.

psi = -dx^2 G * w and the centred differences of G, with G the plan's own table,
convolved by torch.fft in FP64 on the same padded torus.  Both sides round to
about 2^-52 of the largest value a pass; 40 such roundings over the two
transforms of either side bound the difference by 2e-14 in the 2-norm."""
import pytest
import torch

import paper_2102_11910_gb300 as pf

pytestmark = pytest.mark.gpu

TOL = 2e-14


def _reference(plan, w, dx):
    """psi and the node velocity by torch.fft in FP64 from the plan's table."""
    G = torch.from_numpy(pf.pf_lgf_table(plan)).cuda()               # [n, m], 0 <= n <= ny, 0 <= m <= nx
    m = torch.arange(plan.P, device="cuda")
    m = torch.where(m <= plan.P // 2, m, m - plan.P)
    n = torch.arange(plan.Q, device="cuda")
    n = torch.where(n <= plan.Q // 2, n, n - plan.Q)
    mc, nc = m.clamp(-plan.nx + 1, plan.nx - 1)[None, :], n.clamp(-plan.ny + 1, plan.ny - 1)[:, None]

    def conv(k):
        f = torch.fft.irfft2(torch.fft.rfft2(k) * torch.fft.rfft2(w, s=(plan.Q, plan.P)), s=(plan.Q, plan.P))
        return f[:plan.ny, :plan.nx]

    def g(i, j):
        return G[j.abs(), i.abs()]

    return (-dx * dx * conv(g(mc, nc)), -0.5 * dx * conv(g(mc, nc + 1) - g(mc, nc - 1)),
            0.5 * dx * conv(g(mc + 1, nc) - g(mc - 1, nc)))


def _rel(a, b):
    return float((a - b).norm() / b.norm())


# every transform length in each direction: the last pass is radix 4 (256), absent (512), radix 2, 4 and 8;
# odd row counts, a grid that fills its torus and one that leaves it nearly empty
@pytest.mark.parametrize("nx,ny", [(128, 128), (65, 129), (130, 256), (500, 67), (513, 300), (100, 1025), (1024, 511),
                                   (2048, 70), (66, 2047)])
def test_fp64_passes_match_torch_fft(nx, ny):
    dx = 2.0 / max(nx, ny)
    g = torch.Generator(device="cuda")
    g.manual_seed(nx * 4096 + ny)
    w = torch.randn(ny, nx, dtype=torch.float64, device="cuda", generator=g)
    w *= torch.rand(ny, nx, device="cuda", generator=g) < 0.3           # sparse, as a vortex set's field
    plan = pf.Plan(nx, ny, dx, 0.0, 0.0, pf.PF_FP64)
    psi, u, v = _reference(plan, w, dx)
    assert _rel(pf.pf_poisson_solve(plan, w), psi) < TOL
    uv = pf.pf_velocity_solve(plan, w, 0.5, -0.25)
    assert _rel(uv[..., 0] - 0.5, u) < 20 * TOL and _rel(uv[..., 1] + 0.25, v) < 20 * TOL   # differences of G: cancellation
    alias = w.clone()
    pf.pf_poisson_solve(plan, alias, alias)
    assert torch.equal(alias, pf.pf_poisson_solve(plan, w))
    pf.pf_sync(plan)


@pytest.mark.parametrize("scale", [1e-300, 2.0 ** -1060, 1e290])
def test_the_exponent_range_is_that_of_doubles(scale):
    plan = pf.Plan(140, 90, 1.0, 0.0, 0.0, pf.PF_FP64)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    w = torch.randn(90, 140, dtype=torch.float64, device="cuda", generator=g)
    psi = pf.pf_poisson_solve(plan, w)
    got = pf.pf_poisson_solve(plan, w * scale)
    tol = TOL if scale >= 1e-300 else 1e-3                              # 2^-1060: inputs are denormals of 14 bits
    back = scale ** -0.5                                                # 1 / scale itself would overflow
    assert _rel(got * back * back, psi) < tol


def test_rows_of_very_different_size_and_empty_rows():
    plan = pf.Plan(200, 150, 0.01, 0.0, 0.0, pf.PF_FP64)
    w = torch.zeros(150, 200, dtype=torch.float64, device="cuda")
    w[3, 7], w[40, 100], w[41, 5], w[149, 199] = 1e12, 1.0, -1e-12, 2e-300
    psi, _, _ = _reference(plan, w, 0.01)
    assert _rel(pf.pf_poisson_solve(plan, w), psi) < TOL
    assert float(pf.pf_poisson_solve(plan, torch.zeros_like(w)).abs().max()) == 0.0
    uv = pf.pf_velocity_solve(plan, torch.zeros_like(w), 1.5, -2.0)
    assert torch.equal(uv[..., 0], torch.full_like(w, 1.5)) and torch.equal(uv[..., 1], torch.full_like(w, -2.0))


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_a_value_that_is_not_finite_reaches_every_output(bad):
    plan = pf.Plan(160, 130, 0.01, 0.0, 0.0, pf.PF_FP64)
    w = torch.ones(130, 160, dtype=torch.float64, device="cuda")
    w[77, 3] = bad
    assert bool(torch.isnan(pf.pf_poisson_solve(plan, w)).all())
    assert bool(torch.isnan(pf.pf_velocity_solve(plan, w)).all())
    w[77, 3] = 1.0                                                      # and leaves nothing behind
    assert bool(torch.isfinite(pf.pf_poisson_solve(plan, w)).all())
