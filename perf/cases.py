"""The work a user of this package has it do, as cases that can be timed and checked.

Every case goes through the package's public entry points.  The ranges are those
of the workload generators in ``paper_2102_11910_gb300/inputs.py`` and of the
tests: grids of 128^2 to 2048 x 1800 nodes (also ones that are no power of two
and not square), 100 to 4e6 vortices, plates and ellipses of 32 to 256 surface
points, both precisions.

  vic     the body-free velocity of a vortex set at its own vortices
  psi     the streamfunction of a node field
  probe   the node velocity of a field and its values at given points
  vstate  a vortex set loaded into the tile-ordered state, stepped, read back
  plate   one step of a plate in a stream built from the single operators
  steps   a vortex set loaded, stepped around a body, read back
  serve   a burst of requests through the server
"""
import math

import numpy as np
import torch

import paper_2102_11910_gb300 as pf

PREC = {"mixed": pf.PF_MIXED, "fp64": pf.PF_FP64}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: the plate workload's grid and vortex count without its body
        dict(name="vic_128_256", path="vic", nx=128, ny=128, nv=256, prec="mixed"),
        # a middle-sized instance of the batch recipe on a grid that is no power of two; odd count
        dict(name="vic_700x333_20011", path="vic", nx=700, ny=333, nv=20011, prec="mixed"),
        # the benchmark workload, in both precisions
        dict(name="vic_1024_1e6", path="vic", nx=1024, ny=1024, nv=1000000, prec="mixed"),
        dict(name="vic_1024_1e6_fp64", path="vic", nx=1024, ny=1024, nv=1000000, prec="fp64"),
        # the largest grid of the tests
        dict(name="vic_2048x1800_4e6", path="vic", nx=2048, ny=1800, nv=4000000, prec="mixed"),
        # a streamfunction for output or for the pressure, in the precision a plot needs and in FP64
        dict(name="psi_512x384_fp64", path="psi", nx=512, ny=384, nv=5000, prec="fp64"),
        # velocities of a field at measuring points that are not the vortices
        dict(name="probe_768x512", path="probe", nx=768, ny=512, nv=4000, nq=200003, prec="mixed"),
        # body-free time stepping on the state made for it
        dict(name="vstate_1024_1e6", path="vstate", nx=1024, ny=1024, nv=1000000, nsteps=8, prec="mixed"),
        # the single-step plate workload: regularize, sheet with Kutta at both edges, velocity, interpolate
        dict(name="plate_128_fp64", path="plate", nx=128, ny=128, nv=256, ns=64, prec="fp64"),
        # the same plate stepped in time (Euler, two vortices released a step)
        dict(name="steps_plate_128", path="steps", nx=128, ny=128, nv=256, ns=64, nsteps=16, scheme=0, pitch=False,
             prec="mixed"),
        # the pitching plate half way through its run (RK2, a factor of S for every pose)
        dict(name="steps_pitch_768x512", path="steps", nx=768, ny=512, nv=2000, ns=64, nsteps=6, scheme=1, pitch=True,
             prec="mixed"),
        # uneven requests as the server gets them: small ones, and one in ten at 1024^2 with 1e5 vortices
        dict(name="serve_20", path="serve", requests=20, most_steps=6, prec="mixed"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _points_of(rng, nodes):
    """Surface points of a plate `nodes` cells long: 32 to 256, one to four cells apart where that allows it."""
    lo = max(32, math.ceil(nodes / 4.0))
    return rng.randint(lo, max(lo, min(256, int(nodes))))


def draw(rng):
    path = rng.choice(["vic", "vic", "vic", "psi", "probe", "vstate", "plate", "steps", "serve"])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    nx, ny = _log(rng, 100, 2048), _log(rng, 100, 1800)
    if path == "vic":
        return dict(path=path, nx=nx, ny=ny, nv=_log(rng, 100, 4000000 if prec == "mixed" else 1000000), prec=prec)
    if path == "psi":
        return dict(path=path, nx=nx, ny=ny, nv=_log(rng, 100, 100000), prec=prec)
    if path == "probe":
        return dict(path=path, nx=nx, ny=ny, nv=_log(rng, 100, 100000), nq=_log(rng, 100, 1000000), prec=prec)
    if path == "vstate":
        return dict(path=path, nx=nx, ny=ny, nv=_log(rng, 1000, 1000000), nsteps=rng.randint(1, 10), prec="mixed")
    if path == "plate":
        n = _log(rng, 112, 512)
        return dict(path=path, nx=n, ny=n - rng.randint(0, n // 4), nv=_log(rng, 100, 5000), ns=_points_of(rng, n / 2.54),
                    prec=prec)
    if path == "steps":
        pitch = rng.random() < 0.5
        n = _log(rng, 256 if pitch else 128, 512)
        nx = n + n // 2 if pitch else n
        return dict(path=path, nx=nx, ny=n, nv=_log(rng, 100, 20000), ns=_points_of(rng, nx / (7.68 if pitch else 2.54)),
                    nsteps=rng.randint(4, 16), scheme=rng.randint(0, 1), pitch=pitch, prec="mixed")
    return dict(path="serve", requests=rng.randint(8, 20), most_steps=rng.randint(1, 6), prec="mixed")


# -------------------------------------------------------------------- inputs
def _grid(case):
    """nx x ny nodes centred on the origin, 2 units along the longer direction (around a plate 2.54); the
    pitching plate's grid is 7.68 long and begins 1.5 chords upstream of mid-chord."""
    nx, ny = case["nx"], case["ny"]
    if case.get("pitch"):
        dx = 0.01 * 768 / nx
        return dx, -1.5, -0.5 * (ny - 1) * dx
    if case["path"] in ("plate", "steps"):
        dx = 2.54 / (max(nx, ny) - 1)
    else:
        dx = 2.0 / (max(nx, ny) - 1)
    return dx, -0.5 * (nx - 1) * dx, -0.5 * (ny - 1) * dx


def _vortices(case, seed):
    """nv vortices uniform in the grid's central 80 %, strengths N(0, 1e-4), on the device."""
    dx, x0, y0 = _grid(case)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    r = torch.rand(2, case["nv"], dtype=torch.float64, device="cuda", generator=g)
    X = x0 + (case["nx"] - 1) * dx * (0.1 + 0.8 * r[0])
    Y = y0 + (case["ny"] - 1) * dx * (0.1 + 0.8 * r[1])
    G = 0.01 * torch.randn(case["nv"], dtype=torch.float64, device="cuda", generator=g)
    return X.contiguous(), Y.contiguous(), G


def _points(case, seed):
    """nq measuring points over the whole grid but for the two nodes' rim that a stencil needs."""
    dx, x0, y0 = _grid(case)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 1000003)
    r = torch.rand(2, case["nq"], dtype=torch.float64, device="cuda", generator=g)
    return ((x0 + dx * (1.5 + (case["nx"] - 4.5) * r[0])).contiguous(),
            (y0 + dx * (1.5 + (case["ny"] - 4.5) * r[1])).contiguous())


def _body_case(case, seed):
    """Plate of chord 1 through the origin and vortices away from it, on the host."""
    dx, x0, y0 = _grid(case)
    rng = np.random.default_rng(seed)
    ns, nv = case["ns"], case["nv"]
    xi = -1.0 + (2.0 * np.arange(1, ns + 1) - 1.0) / ns
    alpha0 = math.radians(30.0 if case.get("pitch") else 20.0)
    amp, omega = (math.radians(10.0), 1.0) if case.get("pitch") else (0.0, 0.0)
    X, Y = np.empty(0), np.empty(0)
    hx, hy = (case["nx"] - 1) * dx, (case["ny"] - 1) * dx
    while len(X) < nv:
        # pitching: a wake behind the plate; else all around it
        lo, hi = (0.27, 0.85) if case.get("pitch") else (0.1, 0.9)
        x = x0 + hx * rng.uniform(lo, hi, 2 * nv)
        y = y0 + hy * rng.uniform(0.15, 0.85, 2 * nv)
        keep = (np.abs(x) > 0.56) | (np.abs(y) > 0.35)
        X, Y = np.concatenate([X, x[keep]]), np.concatenate([Y, y[keep]])
    # strengths N(0, 0.01) for 256 vortices, smaller as they get more, so that speeds stay near the stream's
    G = rng.normal(0.0, 0.1 * math.sqrt(256.0 / max(256, nv)) * (0.3 if case.get("pitch") else 1.0), nv)
    return dict(xb=0.5 * xi, yb=np.zeros(ns), ds=np.full(ns, 1.0 / ns), edges=(0, ns - 1), alpha0=alpha0, amp=amp,
                omega=omega, X=X[:nv].copy(), Y=Y[:nv].copy(), G=G, dt=(0.25 if case.get("pitch") else 0.1) * dx)


def _requests(case, seed):
    """Requests of the batch recipe: grids of 128^2 to 512^2, a plate that releases at both edges or an ellipse, 100 to
    20000 vortices; every tenth at 1024^2 with 1e5 vortices.  1 to most_steps steps of half a cell at the fastest."""
    rng = np.random.default_rng(seed)
    shape_rng = np.random.default_rng(case["requests"] * 100 + case["most_steps"])   # the sizes belong to the case
    out = []
    for i in range(case["requests"]):
        big = i % 10 == 5
        nx, ny = (1024, 1024) if big else ((128, 128), (256, 256), (512, 384), (512, 512))[shape_rng.integers(4)]
        dx = 2.0 / (max(nx, ny) - 1)
        plate = shape_rng.random() < 0.5
        if plate:
            perim = 1.0
        else:
            a, b = 0.5, 0.5 / shape_rng.uniform(2.0, 10.0)
            t = np.linspace(0.0, 2 * np.pi, 20001)
            s = np.concatenate([[0.0], np.cumsum(np.hypot(a * np.diff(np.cos(t)), b * np.diff(np.sin(t))))])
            perim = float(s[-1])
        lo = max(32, int(math.ceil(perim / (4.0 * dx))))
        ns = int(shape_rng.integers(lo, max(lo, min(256, int(perim / dx))) + 1))
        nv = 100000 if big else int(round(math.exp(shape_rng.uniform(math.log(100), math.log(20000)))))
        if plate:
            xb, yb, ds = 0.5 * (-1.0 + (2.0 * np.arange(1, ns + 1) - 1.0) / ns), np.zeros(ns), np.full(ns, 1.0 / ns)
            edges, alpha = (0, ns - 1), math.radians(rng.uniform(5.0, 30.0))
        else:
            tp = np.interp(perim * np.arange(ns) / ns, s, t)
            xb, yb, ds, edges, alpha = a * np.cos(tp), b * np.sin(tp), np.full(ns, perim / ns), (), rng.uniform(0.0, math.pi)
        h = 0.5 * (nx - 1) * dx
        hy = 0.5 * (ny - 1) * dx - 0.35
        X, Y = np.empty(0), np.empty(0)
        while len(X) < nv:
            x, y = rng.uniform(-0.8 * h, 0.4 * h, 2 * nv), rng.uniform(-hy, hy, 2 * nv)
            keep = np.hypot(x, y) > 0.55
            X, Y = np.concatenate([X, x[keep]]), np.concatenate([Y, y[keep]])
        G = rng.normal(0.0, math.sqrt(1e-3), nv)
        out.append(dict(nx=nx, ny=ny, grid=(dx, -h, -0.5 * (ny - 1) * dx), xb=xb, yb=yb, ds=ds, edges=edges, alpha0=alpha,
                        amp=0.0, omega=0.0, X=X[:nv].copy(), Y=Y[:nv].copy(), G=G, dt=min(0.002, 0.5 * dx / (1.0 + 0.069 * math.sqrt(nv))),
                        nsteps=int(shape_rng.integers(1, case["most_steps"] + 1))))
    return out


# --------------------------------------------------------------- the program
def _plan(case):
    dx, x0, y0 = _grid(case)
    return pf.Plan(case["nx"], case["ny"], dx, x0, y0, PREC[case["prec"]])


def prepare(case, seed):
    path = case["path"]
    s = dict(case=case)
    if path == "serve":
        s["server"] = pf.Server(max_slots=16, hbm_budget_bytes=8 << 30, precision=PREC[case["prec"]])
        s["requests"] = []
        for r in _requests(case, seed):
            body = pf.BodyKinematics(r["xb"], r["yb"], r["ds"], r["edges"], r["alpha0"], Uinf=1.0)
            s["requests"].append(((r["nx"], r["ny"]) + r["grid"], r["X"], r["Y"], r["G"], r["nsteps"], r["dt"], body))
        return s
    plan = s["plan"] = _plan(case)
    if path in ("plate", "steps"):
        b = s["b"] = _body_case(case, seed)
        if path == "steps":
            s["body"] = pf.BodyKinematics(b["xb"], b["yb"], b["ds"], b["edges"], b["alpha0"], b["amp"], b["omega"], Uinf=1.0)
            s["state"] = pf.pf_state_create(plan, case["nv"] + 2 * case["nsteps"])
            return s
        xs, ys = _turned(b, b["alpha0"])
        s["schur"] = pf.pf_schur_factor(plan, xs, ys, b["ds"])
        new = [_release(xs, ys, k, None, b["dt"]) for k in b["edges"]]
        s["new"] = [p[0] for p in new], [p[1] for p in new]
        s["X"], s["Y"], s["G"] = (torch.from_numpy(b[k]).cuda() for k in ("X", "Y", "G"))
        s["Xall"], s["Yall"] = (torch.cat([s[k], torch.tensor(p, dtype=torch.float64, device="cuda")])
                                for k, p in zip(("X", "Y"), s["new"]))
        s["gamma_w"] = float(b["G"].sum())
        return s
    s["X"], s["Y"], s["G"] = _vortices(case, seed)
    if path == "vic":
        s["u"], s["v"] = (torch.empty(case["nv"], dtype=plan.dtype, device="cuda") for _ in range(2))
    elif path == "vstate":
        s["state"] = pf.VicState(plan, case["nv"])
    else:
        s["w"] = pf.pf_regularize(plan, s["X"], s["Y"], s["G"])
        if path == "probe":
            s["Xq"], s["Yq"] = _points(case, seed)
    return s


def run(s):
    case, path = s["case"], s["case"]["path"]
    if path == "serve":
        tickets = [pf.pf_server_submit(s["server"], *r) for r in s["requests"]]
        left = set(tickets)
        while left:
            left.difference_update(pf.pf_server_progress(s["server"]))
        return [_frame(case, pf.pf_server_result(s["server"], t, len(r[1]) + 2 * r[4])) for t, r in zip(tickets, s["requests"])]
    plan = s["plan"]
    if path == "vic":
        return pf.pf_vic_velocity(plan, s["X"], s["Y"], s["G"], 1.0, 0.0, s["u"], s["v"])
    if path == "psi":
        return pf.pf_poisson_solve(plan, s["w"])
    if path == "probe":
        uv = pf.pf_velocity_solve(plan, s["w"], 1.0, 0.0)
        return (uv,) + tuple(pf.pf_interpolate(plan, uv, s["Xq"], s["Yq"]))
    if path == "vstate":
        pf.pf_vic_state_set(s["state"], s["X"], s["Y"], s["G"])
        for _ in range(case["nsteps"]):
            pf.pf_vic_step(s["state"], VSTATE_DT, 1.0, 0.0)
        return pf.pf_vic_state_get(s["state"])[:4]
    if path == "plate":
        w = pf.pf_regularize(plan, s["X"], s["Y"], s["G"])
        f, gn, s0 = pf.pf_sheet_solve(plan, s["schur"], w, (0.0, 0.0, 0.0, 1.0, 0.0), pf.PF_SHEET_KUTTA_SHED, s["gamma_w"],
                                      s["b"]["edges"], *s["new"])
        gn = torch.tensor(gn, dtype=torch.float64)
        pf.pf_regularize(plan, s["Xall"], s["Yall"], torch.cat([s["G"], gn.cuda()]), w)
        pf.pf_sheet_regularize(plan, s["schur"], f, w)
        uv = pf.pf_velocity_solve(plan, w, 1.0, 0.0)
        return (f, gn, s0) + tuple(pf.pf_interpolate(plan, uv, s["Xall"], s["Yall"]))
    b = s["b"]
    pf.pf_state_set(s["state"], b["X"], b["Y"], b["G"])
    for _ in range(case["nsteps"]):
        pf.pf_step(plan, s["state"], b["dt"], s["body"], case["scheme"])
    return _frame(case, pf.pf_state_get(s["state"]))


def _frame(case, out):
    """Positions and strengths as a program stores them for a movie or a restart: in the plan's precision."""
    return [a.astype(np.float32 if case["prec"] == "mixed" else np.float64) for a in out[:3]]


VSTATE_DT = 1e-5      # a small part of a cell a step at the benchmark's vortex density


# ---------------------------------------------------------------------- work
def _conv_flops(nx, ny, inverses):
    p, q = 1 << (2 * nx - 1).bit_length(), 1 << (2 * ny - 1).bit_length()
    return (1 + inverses) * 2.5 * p * q * math.log2(p * q)


def work(case):
    """Inputs once, outputs once; the padded convolution, 16 nodes a vortex and transfer, and the sheet's dense solves."""
    path, e = case["path"], 4 if case["prec"] == "mixed" else 8
    if path == "serve":
        b = f = 0
        for r in _requests(case, 0):
            n, nv = r["nsteps"], len(r["X"])
            b += 48 * nv
            f += n * (_conv_flops(r["nx"], r["ny"], 2) + 300 * nv + 6 * len(r["xb"]) ** 2) + 2 * len(r["xb"]) ** 3
        return {"bytes": b, "flops": f}
    nodes, nv = case["nx"] * case["ny"], case["nv"]
    if path == "vic":
        return {"bytes": (24 + 2 * e) * nv, "flops": _conv_flops(case["nx"], case["ny"], 2) + 220 * nv}
    if path == "psi":
        return {"bytes": 2 * e * nodes, "flops": _conv_flops(case["nx"], case["ny"], 1)}
    if path == "probe":
        return {"bytes": 3 * e * nodes + (16 + 2 * e) * case["nq"], "flops": _conv_flops(case["nx"], case["ny"], 2) + 120 * case["nq"]}
    if path == "vstate":
        return {"bytes": 48 * nv, "flops": case["nsteps"] * (_conv_flops(case["nx"], case["ny"], 2) + 240 * nv)}
    ns = case["ns"]
    stages = 1 if path == "plate" else case["nsteps"] * (1 + case["scheme"])
    factor = 0 if path == "plate" else (stages if case["pitch"] else 1) * 2 * ns ** 3
    return {"bytes": 48 * nv + (0 if path == "plate" else 48 * case["nsteps"]),
            "flops": stages * (_conv_flops(case["nx"], case["ny"], 2) + 500 * nv + 18 * ns ** 2) + factor}


# --------------------------------------------------------- the same in 64 bits
# Plain torch on the device, FP64 throughout: the lattice Green's function by
# quadrature of its one-dimensional integral, the convolution by torch.fft, M4'
# and the smoothed three-point function written out, dense solves.
_TABLES = {}


def _lgf(n):
    """G(m, k), 0 <= m, k <= n: (1/2 pi) int_0^pi (1 - exp(-2 m u) cos(k t)) / sinh(2 u) dt, sinh u = sin(t/2), m >= k."""
    if n not in _TABLES:
        x, wt = np.polynomial.legendre.leggauss(20)
        e = np.concatenate([[0.0], np.pi * 1.4 ** np.arange(-72.0, 1.0)])
        h = 0.5 * np.diff(e)
        t = torch.from_numpy((e[:-1, None] + h[:, None] * (1.0 + x)).ravel()).cuda()
        wt = torch.from_numpy((h[:, None] * wt).ravel()).cuda()
        u = torch.asinh(torch.sin(0.5 * t))
        c = wt / torch.sinh(2.0 * u) / (2.0 * math.pi)
        k = torch.arange(n + 1, dtype=torch.float64, device="cuda")
        G = torch.empty(n + 1, n + 1, dtype=torch.float64, device="cuda")
        half = 2.0 * torch.sin(0.5 * t[:, None] * k[None, :]) ** 2
        for i in range(0, n + 1, 256):
            decay = -2.0 * k[i:i + 256, None] * u[None, :]
            G[i:i + 256] = ((-torch.expm1(decay)) @ c)[:, None] + (torch.exp(decay) * c) @ half
        low = torch.tril(G)
        _TABLES.clear()
        _TABLES[n] = low + torch.tril(G, -1).T
    return _TABLES[n]


class _Flow:
    def __init__(self, nx, ny, dx, x0, y0):
        self.nx, self.ny, self.dx, self.x0, self.y0 = nx, ny, dx, x0, y0
        self.G = _lgf(max(nx, ny) + 1)
        self.P, self.Q = (1 << (2 * n + 1).bit_length() for n in (nx, ny))

    def _conv(self, w, kernel):
        """sum over the grid's nodes of kernel(i - i', j - j') w(i', j')."""
        m = torch.arange(self.P, device="cuda")
        m = torch.where(m < self.P // 2, m, m - self.P)
        n = torch.arange(self.Q, device="cuda")
        n = torch.where(n < self.Q // 2, n, n - self.Q)
        k = kernel(m.clamp(-self.nx, self.nx)[None, :], n.clamp(-self.ny, self.ny)[:, None])
        out = torch.fft.irfft2(torch.fft.rfft2(k) * torch.fft.rfft2(w, s=(self.Q, self.P)), s=(self.Q, self.P))
        return out[:self.ny, :self.nx].contiguous()

    def at(self, m, n):
        return self.G[m.abs(), n.abs()]

    def psi(self, w):
        return -self.dx ** 2 * self._conv(w, self.at)

    def velocity(self, w, U, V):
        """Central differences of psi, as differences of G."""
        u = -0.5 * self.dx * self._conv(w, lambda m, n: self.at(m, n + 1) - self.at(m, n - 1)) + U
        v = 0.5 * self.dx * self._conv(w, lambda m, n: self.at(m + 1, n) - self.at(m - 1, n)) + V
        return u, v

    def _stencil(self, X, Y, weight):
        ix, wx, iy, wy = [], [], [], []
        for Z, z0, i, wz in ((X, self.x0, ix, wx), (Y, self.y0, iy, wy)):
            g = (Z - z0) / self.dx
            for a in range(-1, 3):
                i.append(torch.floor(g) + a)
                wz.append(weight((g - i[-1]).abs()))
        ix, iy = (torch.stack(i, -1).long() for i in (ix, iy))
        wx, wy = torch.stack(wx, -1), torch.stack(wy, -1)
        return ((ix[:, None, :].expand(-1, 4, 4)).reshape(-1, 16), (iy[:, :, None].expand(-1, 4, 4)).reshape(-1, 16),
                (wy[:, :, None] * wx[:, None, :]).reshape(-1, 16))

    @staticmethod
    def m4p(r):
        return torch.where(r <= 1, 1 - 2.5 * r ** 2 + 1.5 * r ** 3, torch.where(r <= 2, 0.5 * (2 - r) ** 2 * (1 - r), 0 * r))

    @staticmethod
    def three(r):
        s3 = math.sqrt(3.0)
        a, b = r.clamp(max=1.0), r.clamp(1.0, 2.0)
        inner = (17 / 48 + s3 * math.pi / 108 + a / 4 - a ** 2 / 4 + (1 - 2 * a) / 16 * (-12 * a ** 2 + 12 * a + 1).clamp(min=0).sqrt()
                 - s3 / 12 * torch.asin(s3 / 2 * (2 * a - 1)))
        outer = (55 / 48 - s3 * math.pi / 108 - 13 * b / 12 + b ** 2 / 4
                 + (2 * b - 3) / 48 * (-12 * b ** 2 + 36 * b - 23).clamp(min=0).sqrt() + s3 / 36 * torch.asin(s3 / 2 * (2 * b - 3)))
        return torch.where(r <= 1, inner, torch.where(r < 2, outer, 0 * r))

    def regularize(self, X, Y, G):
        i, j, w = self._stencil(X, Y, self.m4p)
        out = torch.zeros(self.ny * self.nx, dtype=torch.float64, device="cuda")
        out.index_add_(0, (j * self.nx + i).reshape(-1), (w * G[:, None]).reshape(-1))
        return out.reshape(self.ny, self.nx) / self.dx ** 2

    def interpolate(self, field, X, Y):
        i, j, w = self._stencil(X, Y, self.m4p)
        return (w * field[j, i]).sum(-1)

    # surface points (xs, ys, ds): S, E_s and R_s with the smoothed three-point function
    def surface(self, xs, ys, ds):
        s = _Surface()
        s.x, s.y, s.ds = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (xs, ys, ds))
        s.i, s.j, s.w = self._stencil(s.x, s.y, self.three)
        s.S = -self._pairs(s, s.i, s.j, s.w) * s.ds[None, :]
        s.lu = torch.linalg.lu_factor(s.S)
        s.f0 = s.solve(torch.ones_like(s.x))
        s.f0h = s.ds * s.f0
        s.g0 = s.f0h.sum()
        return s

    def _pairs(self, s, i, j, w):
        out = torch.empty(len(s.x), len(i), dtype=torch.float64, device="cuda")
        for p in range(len(s.x)):
            g = self.at(s.i[p][:, None, None] - i[None], s.j[p][:, None, None] - j[None])
            out[p] = torch.einsum("a,aqb,qb->q", s.w[p], g, w)
        return out

    def sheet(self, s, w, Omega, U, V, edges, Xn, Yn):
        """The sheet, the new strengths and s0: Kutta at the two edges and Kelvin, or Kelvin alone without edges.
        Gamma_w is the circulation of w."""
        gw = w.sum() * self.dx ** 2
        sb = -U * s.y + V * s.x - 0.5 * Omega * (s.x ** 2 + s.y ** 2)
        e = -(s.w * self.psi(w)[s.j, s.i]).sum(-1)
        if not len(edges):
            f = s.solve(sb + e)
            s0 = ((s.ds * f).sum() + gw) / s.g0
            return f - s0 * s.f0, gw.new_zeros(0), s0
        one = s.solve(sb + e)
        i, j, m = self._stencil(Xn, Yn, self.m4p)
        each = s.solve(self._pairs(s, i, j, m))                       # a column for each new vortex
        # unknowns (s0, strengths): f = one + each Gamma - s0 f0; f = 0 x f0 at the edges; circulation zero
        n = len(edges)
        A = torch.zeros(n + 1, n + 1, dtype=torch.float64, device="cuda")
        b = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
        for r, k in enumerate(edges):
            A[r, 0], A[r, 1:], b[r] = -1.0, each[k] / s.f0[k], -one[k] / s.f0[k]
        A[n, 0], A[n, 1:], b[n] = -s.g0, 1.0 + (s.ds[:, None] * each).sum(0), -gw - (s.ds * one).sum()
        z = torch.linalg.solve(A, b)
        return one + each @ z[1:] - z[0] * s.f0, z[1:], z[0]

    def sheet_field(self, s, f):
        out = torch.zeros(self.ny * self.nx, dtype=torch.float64, device="cuda")
        out.index_add_(0, (s.j * self.nx + s.i).reshape(-1), (s.w * (s.ds * f)[:, None]).reshape(-1))
        return out.reshape(self.ny, self.nx) / self.dx ** 2

    def at_vortices(self, X, Y, G, s, f):
        w = self.regularize(X, Y, G)
        u, v = self.velocity(w if s is None else w + self.sheet_field(s, f), 1.0, 0.0)
        return self.interpolate(u, X, Y), self.interpolate(v, X, Y)

    def steps(self, b, nsteps, scheme):
        """The vortices after nsteps steps around the body b in the stream (1, 0)."""
        X, Y, G = (torch.from_numpy(b[k]).cuda() for k in ("X", "Y", "G"))
        last = [None] * len(b["edges"])
        surf, dt = None, b["dt"]

        def at(t):
            return b["alpha0"] + b["amp"] * math.sin(b["omega"] * t), -b["amp"] * b["omega"] * math.cos(b["omega"] * t)

        for n in range(nsteps):
            a, Omega = at(n * dt)
            xs, ys = _turned(b, a)
            if surf is None or b["amp"]:
                surf = self.surface(xs, ys, b["ds"])
            w = self.regularize(X, Y, G)
            new = [_release(xs, ys, k, None if q is None else (float(X[q]), float(Y[q])), dt) for k, q in zip(b["edges"], last)]
            Xn, Yn = (torch.tensor([p[c] for p in new], dtype=torch.float64, device="cuda") for c in (0, 1))
            f, gn, _ = self.sheet(surf, w, Omega, 1.0, 0.0, b["edges"], Xn, Yn)
            last = [len(X) + k for k in range(len(new))]
            X, Y, G = torch.cat([X, Xn]), torch.cat([Y, Yn]), torch.cat([G, gn])
            u, v = self.at_vortices(X, Y, G, surf, f)
            if scheme == 0:
                X, Y = X + dt * u, Y + dt * v
                continue
            Xs, Ys = X + dt * u, Y + dt * v
            a, Omega = at((n + 1) * dt)
            if b["amp"]:
                surf = self.surface(*_turned(b, a), b["ds"])
            f, _, _ = self.sheet(surf, self.regularize(Xs, Ys, G), Omega, 1.0, 0.0, (), None, None)
            u2, v2 = self.at_vortices(Xs, Ys, G, surf, f)
            X, Y = X + 0.5 * dt * (u + u2), Y + 0.5 * dt * (v + v2)
        return X, Y, G


class _Surface:
    def solve(self, r):
        x = torch.linalg.lu_solve(*self.lu, r.reshape(len(self.x), -1))
        x = x + torch.linalg.lu_solve(*self.lu, r.reshape(len(self.x), -1) - self.S @ x)
        return x.reshape(r.shape)


def _turned(b, alpha):
    ca, sa = math.cos(alpha), math.sin(alpha)
    return ca * b["xb"] + sa * b["yb"], -sa * b["xb"] + ca * b["yb"]


def _release(xs, ys, k, last, dt):
    """Where the vortex of the edge at point k starts: half a segment beyond it, then 10 dt along the normal that faces the
    stream (1, 0), or one third of the way to the last one released."""
    m = k + 1 if k == 0 else k - 1
    tx, ty = xs[k] - xs[m], ys[k] - ys[m]
    ex, ey = xs[k] + 0.5 * tx, ys[k] + 0.5 * ty
    if last is not None:
        return ex + (last[0] - ex) / 3.0, ey + (last[1] - ey) / 3.0
    n = math.hypot(tx, ty) * (1.0 if -ty >= 0.0 else -1.0)
    return ex - 10.0 * dt * ty / n, ey + 10.0 * dt * tx / n


def exact(case, seed):
    path = case["path"]
    if path == "serve":
        out = []
        for r in sorted(enumerate(_requests(case, seed)), key=lambda r: r[1]["nx"]):
            q = r[1]
            out.append((r[0], _Flow(q["nx"], q["ny"], *q["grid"]).steps(q, q["nsteps"], 0)))
        return [o for _, o in sorted(out, key=lambda o: o[0])]
    flow = _Flow(case["nx"], case["ny"], *_grid(case))
    if path == "steps":
        return flow.steps(_body_case(case, seed), case["nsteps"], case["scheme"])
    if path == "plate":
        b = _body_case(case, seed)
        xs, ys = _turned(b, b["alpha0"])
        surf = flow.surface(xs, ys, b["ds"])
        X, Y, G = (torch.from_numpy(b[k]).cuda() for k in ("X", "Y", "G"))
        new = [_release(xs, ys, k, None, b["dt"]) for k in b["edges"]]
        Xn, Yn = (torch.tensor([p[c] for p in new], dtype=torch.float64, device="cuda") for c in (0, 1))
        f, gn, s0 = flow.sheet(surf, flow.regularize(X, Y, G), 0.0, 1.0, 0.0, b["edges"], Xn, Yn)
        X, Y, G = torch.cat([X, Xn]), torch.cat([Y, Yn]), torch.cat([G, gn])
        return (f, gn, float(s0)) + flow.at_vortices(X, Y, G, surf, f)
    X, Y, G = _vortices(case, seed)
    if path == "vic":
        return flow.at_vortices(X, Y, G, None, None)
    if path == "vstate":
        for _ in range(case["nsteps"]):
            u, v = flow.at_vortices(X, Y, G, None, None)
            X, Y = X + VSTATE_DT * u, Y + VSTATE_DT * v
        return X, Y, G, None
    w = flow.regularize(X, Y, G)
    if path == "psi":
        return flow.psi(w)
    u, v = flow.velocity(w, 1.0, 0.0)
    Xq, Yq = _points(case, seed)
    return torch.stack([u, v], -1), flow.interpolate(u, Xq, Yq), flow.interpolate(v, Xq, Yq)
