"""Workloads of the solver as its users run them, through its public entry points.

Each case names one kind of call:

  tube     one 1D problem advanced on its own (``Solver.set_state``,
           ``advance``, ``get_state``): the smallest calls, a few hundred
           cells, where latency and launches count
  grid     one 2D problem advanced a few CFL steps the same way
  batch    thousands of independent 1D Riemann problems (``Batch.run``)
  boxes    many independent 2D explosions (``Batch2D.run``)
  rhs      one evaluation of the semi-discrete operator (``Solver.rhs``)
  grad     the operator and its reverse (``rhs_autograd`` and its backward)

Grids, boundary conditions and end times are those of
``paper_1908_02464_gb300.problems`` (the test problems, the benchmark and its
batches); the states are drawn from the seed: the problem's own data with
random amplitudes, phases and contact discontinuities, so that smooth flow
and discontinuities meet in about the proportion of a developed run.
"""
import math

import numpy as np
import torch

from paper_1908_02464_gb300 import problems as P
from paper_1908_02464_gb300 import weno

GAMMA = 1.4


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # a shock tube solved once, start to end: the smallest run a user makes
        dict(name="sod_200_fp64", kind="tube", problem="riemann", n=200, precision="fp64", steps=0),
        # the shock / entropy-wave interaction at 400 cells to its end time, in
        # the reduced precision it is compared in
        dict(name="shu_osher_400_fp32", kind="tube", problem="shu_osher", n=400, precision="fp32", steps=0),
        # ten steps of the double Mach reflection on the 512 x 128 grid: an
        # ordinary 2D run that does not fill the chip for long
        dict(name="dmr_512x128_fp64", kind="grid", problem="double_mach", nx=512, ny=128, precision="fp64", steps=10),
        # the benchmark grid in FP64 and in the mixed precision meant for it
        dict(name="dmr_2048x512_fp64", kind="grid", problem="double_mach", nx=2048, ny=512, precision="fp64", steps=4),
        dict(name="dmr_2048x512_mixed", kind="grid", problem="double_mach", nx=2048, ny=512, precision="mixed",
             steps=10),
        # global Lax-Friedrichs splitting (the rule of the 2D test problems) with
        # walls, at the jet's 640 x 160 cut to an odd size
        dict(name="walls_637x159_lf_fp64", kind="grid", problem="walls_lf", nx=637, ny=159, precision="fp64", steps=10),
        # batches of uneven sizes: 1D in FP64, the benchmark's 4096 instances
        # in FP32, 2D boxes in FP64, each over a part of its usual time
        dict(name="riemann_1024_fp64", kind="batch", count=1024, n_lo=100, n_hi=2000, span=0.02, precision="fp64"),
        dict(name="riemann_4096_fp32", kind="batch", count=4096, n_lo=100, n_hi=4000, span=0.05, precision="fp32"),
        dict(name="explosions_1024_fp64", kind="boxes", count=1024, n_lo=16, n_hi=64, span=0.05, precision="fp64"),
        # the 256^3 vortex: operator alone, and with its reverse, in FP32
        dict(name="vortex_256_rhs_fp32", kind="rhs", dim=3, problem="vortex", nx=256, ny=256, nz=256, precision="fp32"),
        dict(name="vortex_256_grad_fp32", kind="grad", dim=3, problem="vortex", nx=256, ny=256, nz=256,
             precision="fp32"),
        # a ragged 3D box with discontinuities, operator and reverse in FP64
        dict(name="mixed_121x97x113_grad_fp64", kind="grad", dim=3, problem="mixed", nx=121, ny=97, nz=113,
             precision="fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tube", "grid", "grid", "batch", "boxes", "rhs", "grad"])
    prec = rng.choice(["fp64", "fp64", "fp32", "mixed"])
    if kind == "tube":
        return dict(kind=kind, problem=rng.choice(["riemann", "shu_osher"]), n=_log_int(rng, 60, 3000), precision=prec,
                    steps=rng.randint(60, 160))
    if kind == "grid":
        return dict(kind=kind, problem=rng.choice(["double_mach", "walls_lf", "mixed"]), nx=_log_int(rng, 120, 2100),
                    ny=_log_int(rng, 40, 520), precision=prec, steps=rng.randint(2, 5))
    if kind == "batch":
        return dict(kind=kind, count=_log_int(rng, 64, 1500), n_lo=rng.randint(60, 200), n_hi=rng.randint(500, 2000),
                    span=0.02, precision=prec)
    if kind == "boxes":
        return dict(kind=kind, count=_log_int(rng, 64, 1024), n_lo=rng.randint(12, 24), n_hi=rng.randint(40, 72),
                    span=0.05, precision=prec)
    dim = rng.choice([2, 3, 3])
    n = [_log_int(rng, 100, 1100) for _ in range(2)] + [1] if dim == 2 else [_log_int(rng, 24, 200) for _ in range(3)]
    problem = "mixed" if dim == 2 else rng.choice(["mixed", "vortex"])
    return dict(kind=kind, dim=dim, problem=problem, nx=n[0], ny=n[1], nz=n[2], precision=prec)


# ------------------------------------------------------------ seeded problems

def _cons(rho, vel, p):
    E = p / (GAMMA - 1.0) + 0.5 * rho * sum(u * u for u in vel)
    return torch.stack([rho] + [rho * u for u in vel] + [E])


def _coords(n, lo, hi):
    """Cell centres, x last: one broadcastable tensor per direction (x, y, z)."""
    out = []
    for d, m in enumerate(n):
        h = (hi[d] - lo[d]) / m
        c = lo[d] + (torch.arange(m, dtype=torch.float64, device="cuda") + 0.5) * h
        out.append(c.reshape([-1] + [1] * d))
    return out


def _waves(rs, xs, lo, hi, base, amp, count=3):
    f = torch.full([1] * len(xs), base, dtype=torch.float64, device="cuda")
    for _ in range(count):
        arg = rs.uniform(0, 2 * math.pi)
        for d, x in enumerate(xs):
            arg = arg + 2 * math.pi * int(rs.randint(1, 4)) * (x - lo[d]) / (hi[d] - lo[d])
        f = f + amp / count * rs.uniform(0.3, 1.0) * torch.sin(arg)
    return f


def _slab(rs, xs, lo, hi):
    """A slab across one direction, as a mask."""
    d = int(rs.randint(len(xs)))
    x0 = rs.uniform(0.1, 0.5)
    x0, x1 = (lo[d] + f * (hi[d] - lo[d]) for f in (x0, x0 + rs.uniform(0.2, 0.4)))
    return (xs[d] >= x0) & (xs[d] < x1)


def _problem(case, seed):
    """Problem description (grid, boundaries, constants), state in float64 on the GPU, start time."""
    rs = np.random.RandomState(seed % (1 << 31))
    kind = case["problem"]
    if kind == "riemann":
        j = 1.0 + rs.uniform(-0.1, 0.1, 4)
        prob, U = P.riemann_1d(case["n"], (j[0], 0.0, j[1]), (0.125 * j[2], 0.0, 0.1 * j[3]), 0.2)
        return prob, torch.from_numpy(U).cuda(), 0.0
    if kind == "shu_osher":
        prob, U = P.shu_osher(case["n"])
        x = P.centers(-5.0, 5.0, case["n"])
        wave = 1.0 + rs.uniform(0.15, 0.25) * np.sin(5.0 * x + rs.uniform(0, 2 * math.pi))
        U[0] = np.where(x < -4.0, U[0], wave)
        return prob, torch.from_numpy(U).cuda(), 0.0
    if kind == "double_mach":
        # the Mach 10 shock on its way at t = 0.05, smooth waves behind it and
        # contact discontinuities on both sides
        nx, ny, t = case["nx"], case["ny"], 0.05
        prob = P.double_mach(8, 8)[0]
        prob["n"] = [nx, ny]
        lo, hi = prob["lo"], prob["hi"]
        xs = _coords([nx, ny], lo, hi)
        post = xs[0] < 1.0 / 6.0 + (xs[1] + 20.0 * t) / math.sqrt(3.0)
        one = torch.ones([ny, nx], dtype=torch.float64, device="cuda")
        rho, u, v, p = (torch.where(post, a, b) * one for a, b in zip(P.DMR_POST, P.DMR_PRE))
        rho = rho * torch.where(post, _waves(rs, xs, lo, hi, 1.0, 0.1), 1.0)
        p = p * torch.where(post, _waves(rs, xs, lo, hi, 1.0, 0.1), 1.0)
        for _ in range(12):
            cx, cy, r = rs.uniform(0.1, 3.0), rs.uniform(0.0, 1.0), rs.uniform(0.08, 0.22)
            inside = (xs[0] - cx) ** 2 + (xs[1] - cy) ** 2 < r * r
            rho = torch.where(inside, rho * rs.uniform(0.7, 1.5), rho)
        return prob, _cons(rho, [u, v], p), t
    n = [case["nx"], case["ny"], case.get("nz", 1)]
    dim = case.get("dim", 2)
    n = n[:dim]
    if kind == "vortex":
        prob = P.vortex3d(8)[0]
        prob["n"] = n
        lo, hi = prob["lo"], prob["hi"]
        X, Y, Z = (x + rs.uniform(0, 2 * math.pi) for x in _coords(n, lo, hi))
        a = rs.uniform(0.8, 1.2)
        one = torch.ones([n[2], n[1], n[0]], dtype=torch.float64, device="cuda")
        u = a * torch.sin(X) * torch.cos(Y) * torch.cos(Z) * one
        v = -a * torch.cos(X) * torch.sin(Y) * torch.cos(Z) * one
        p = 100.0 + a * a * (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2.0) / 16.0
        return prob, _cons(one, [u, v, 0.0 * one], p * one), 0.0
    prob = P.random_state(dim, [8] * dim, 1)[0]
    prob["n"] = n
    if kind == "walls_lf":
        prob["splitting"] = "lf"
        prob["bc_lo"], prob["bc_hi"] = [P.BC_REFLECT] * dim, [P.BC_TRANSMISSIVE] + [P.BC_REFLECT] * (dim - 1)
    lo, hi = prob["lo"], prob["hi"]
    xs = _coords(n, lo, hi)
    one = torch.ones(n[::-1], dtype=torch.float64, device="cuda")
    slab = _slab(rs, xs, lo, hi)
    rho = _waves(rs, xs, lo, hi, 1.0, 0.2) * torch.where(slab, rs.uniform(1.2, 1.6), 1.0) * one
    p = _waves(rs, xs, lo, hi, 1.0, 0.2) * torch.where(slab, rs.uniform(0.6, 1.4), 1.0) * one
    vel = [(_waves(rs, xs, lo, hi, 0.0, 0.4) + torch.where(slab, rs.uniform(-0.2, 0.2), 0.0)) * one for _ in range(dim)]
    return prob, _cons(rho, vel, p), 0.0


def _rows(n, starts):
    """Instance and position within it of every cell of ``len(n)`` instances laid back to back."""
    inst = torch.repeat_interleave(torch.arange(len(n), device=n.device), n)
    return inst, torch.arange(int(n.sum()), device=n.device) - starts[inst]


def _log_uniform(rs, lo, hi, shape):
    return np.exp(rs.uniform(math.log(lo), math.log(hi), shape))


def _batch_sizes(case):
    """Cells of each instance: the batch's sizes belong to the case, its states to the seed."""
    rs = np.random.RandomState(1000 + case["count"])
    shape = (case["count"],) if case["kind"] == "batch" else (case["count"], 2)
    return rs.randint(case["n_lo"], case["n_hi"] + 1, shape).astype(np.int64)


def _batch_state(case, seed, dtype):
    """Riemann problems of the benchmark's ranges: rho and p log-uniform per side, u uniform, no near-vacuum draws."""
    N, rs, g = _batch_sizes(case), np.random.RandomState(seed % (1 << 31)), GAMMA
    W = np.zeros((len(N), 2, 3))
    todo = np.arange(len(N))
    while len(todo):
        rho, p = _log_uniform(rs, 0.01, 10.0, (len(todo), 2)), _log_uniform(rs, 0.01, 10.0, (len(todo), 2))
        u = rs.uniform(-2.0, 2.0, (len(todo), 2))
        c, z = np.sqrt(g * p / rho), (g - 1.0) / (2.0 * g)
        W[todo] = np.stack([rho, u, p], axis=2)
        du = u[:, 1] - u[:, 0]
        star = np.maximum(c.sum(1) - 0.5 * (g - 1.0) * du, 0.0) / (c * p ** -z).sum(1)
        bad = (2.0 * c.sum(1) / (g - 1.0) <= 2.0 * du) | (star ** (1.0 / z) < 1e-3 * p.min(1))
        todo = todo[bad]
    t_end = case["span"] / (np.abs(W[:, :, 1]) + np.sqrt(g * W[:, :, 2] / W[:, :, 0])).max(1)
    Nd = torch.from_numpy(N).cuda()
    starts = torch.cumsum(Nd, 0) - Nd
    inst, i = _rows(Nd, starts)
    left = (i + 0.5) / Nd[inst] < 0.5
    Wd = torch.from_numpy(W).cuda()[inst]
    V = torch.where(left[:, None], Wd[:, 0], Wd[:, 1])
    vals = _cons(V[:, 0], [V[:, 1]], V[:, 2])
    flat = torch.empty(3 * int(N.sum()), dtype=torch.float64, device="cuda")
    for v in range(3):
        flat[3 * starts[inst] + v * Nd[inst] + i] = vals[v]
    return N, t_end, flat.to(dtype)


def _boxes_state(case, seed, dtype):
    """Discs of gas at rest in gas at rest (explosions and implosions), square cells of 1/64."""
    size, rs, h = _batch_sizes(case), np.random.RandomState(seed % (1 << 31)), 1.0 / 64.0
    count, L = len(size), size.min(1) * h
    rho, p = _log_uniform(rs, 0.1, 10.0, (count, 2)), _log_uniform(rs, 0.1, 10.0, (count, 2))
    ratio = rho[:, 0] / rho[:, 1]
    rho[:, 0] = rho[:, 1] * np.clip(ratio, 1 / 15.0, 15.0)
    t_end = case["span"] * L / np.sqrt(GAMMA * p / rho).max(1)
    r = torch.from_numpy(rs.uniform(0.15, 0.35, count) * L).cuda()
    mid = torch.from_numpy(rs.uniform(0.4, 0.6, (count, 2)) * size * h).cuda()
    rho, p = torch.from_numpy(rho).cuda(), torch.from_numpy(p).cuda()
    NX, cells = (torch.from_numpy(a).cuda() for a in (size[:, 0], size[:, 0] * size[:, 1]))
    starts = torch.cumsum(cells, 0) - cells
    inst, i = _rows(cells, starts)
    x = (i % NX[inst] + 0.5) * h
    y = (torch.div(i, NX[inst], rounding_mode="floor") + 0.5) * h
    inside = (x - mid[inst, 0]) ** 2 + (y - mid[inst, 1]) ** 2 < r[inst] ** 2
    rho, p = (torch.where(inside, a[inst, 0], a[inst, 1]) for a in (rho, p))
    vals = _cons(rho, [0.0 * rho, 0.0 * rho], p)
    flat = torch.empty(4 * int(cells.sum()), dtype=torch.float64, device="cuda")
    for v in range(4):
        flat[4 * starts[inst] + v * cells[inst] + i] = vals[v]
    return size[:, 0], size[:, 1], size * h, t_end, flat.to(dtype)


# ------------------------------------------------------------- prepare and run

def prepare(case, seed):
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    kind = case["kind"]
    if kind == "batch":
        N, t_end, U0 = _batch_state(case, seed, dtype)
        b = weno.Batch(N, 0.0, 1.0, t_end, case["precision"])
        return dict(kind=kind, batch=b, U0=U0, U=torch.empty_like(U0))
    if kind == "boxes":
        NX, NY, hi, t_end, U0 = _boxes_state(case, seed, dtype)
        b = weno.Batch2D(NX, NY, (0.0, 0.0), hi, t_end, case["precision"])
        return dict(kind=kind, batch=b, U0=U0, U=torch.empty_like(U0))
    prob, U, t = _problem(case, seed)
    U = U.to(dtype).contiguous()
    state = dict(kind=kind, solver=weno.Solver(prob, case["precision"]), U=U, t=t)
    if kind in ("tube", "grid"):
        state["t_end"] = prob["t_end"]
        state["steps"] = case["steps"] or 2 ** 31 - 1
    elif kind == "rhs":
        state["out"] = torch.empty_like(U)
    else:
        g = torch.Generator(device="cuda").manual_seed(seed)
        state["U"] = U.requires_grad_(True)
        state["w"] = torch.randn(U.shape, dtype=dtype, device="cuda", generator=g)
    return state


def run(state):
    kind = state["kind"]
    if kind in ("batch", "boxes"):
        # the solver works in place: the initial states go in first
        state["U"].copy_(state["U0"])
        state["batch"].run(state["U"])
        status, steps, t = state["batch"].results()
        return dict(U=state["U"], status=status, steps=steps, t=t)
    s = state["solver"]
    if kind in ("tube", "grid"):
        s.set_state(state["U"], state["t"])
        steps = s.advance(state["t_end"], state["steps"])
        U, t = s.get_state(device=True)
        return dict(U=U, t=t, steps=steps)
    if kind == "rhs":
        return s.rhs(state["U"], state["t"], out=state["out"])
    out = weno.rhs_autograd(s, state["U"], state["t"])
    (g,) = torch.autograd.grad(out, state["U"], state["w"])
    return dict(rhs=out.detach(), grad=g)


# ------------------------------------------------------------------------ work

# floating-point operations of the method per cell, per linear upwind face and
# per WENO face, by dimension; a few percent of the faces take the WENO flux
OPS = {1: (17, 151, 1060), 2: (21, 203, 1451), 3: (25, 255, 1842)}
WENO_SHARE = 0.03


def _flops_per_cell(dim):
    cell, ups, wen = OPS[dim]
    return cell + 2 * (dim + 2) * dim + dim * (ups + WENO_SHARE * (wen - ups))


def work(case):
    size = 8 if case["precision"] == "fp64" else 4
    kind = case["kind"]
    if kind == "batch":
        # mean over N ~ U[lo, hi] of N and of N steps, steps = span N / 0.5
        lo, hi = case["n_lo"], case["n_hi"]
        m1, m2 = (lo + hi) / 2, (lo * lo + lo * hi + hi * hi) / 3
        cells, updates = case["count"] * m1, case["count"] * m2 * 3 * case["span"] / 0.5
        return dict(bytes=2 * 3 * size * cells, flops=updates * _flops_per_cell(1))
    if kind == "boxes":
        lo, hi = case["n_lo"], case["n_hi"]
        m = (lo + hi) / 2
        cells = case["count"] * m * m
        # steps ~ span min(NX, NY) h / c over dt = 0.5 h / (2 c)
        updates = cells * 3 * case["span"] * m * 0.8 / 0.25
        return dict(bytes=2 * 4 * size * cells, flops=updates * _flops_per_cell(2))
    if kind == "tube":
        n = case["n"]
        full = {"riemann": 0.2 * 2.2 * n / 0.5, "shu_osher": 1.8 * 4.78 * n / 10.0 / 0.5}[case["problem"]]
        steps = min(full, case["steps"] or full)
        return dict(bytes=2 * 3 * size * n, flops=3 * steps * n * _flops_per_cell(1))
    if kind == "grid":
        cells = case["nx"] * case["ny"]
        return dict(bytes=2 * 4 * size * cells, flops=3 * case["steps"] * cells * _flops_per_cell(2))
    dim = case["dim"]
    cells = case["nx"] * case["ny"] * case["nz"]
    arrays, evals = (2, 1) if kind == "rhs" else (4, 3.5)   # grad: U, w, dU/dt, gradient; reverse ~ 2.5 forward
    return dict(bytes=arrays * (dim + 2) * size * cells, flops=evals * cells * _flops_per_cell(dim))


# ------------------------------------------------------ the same in 64 bits

class _Ref:
    """The scheme in plain float64 tensor operations.  Arrays are [var, ..., along] with the swept direction last."""

    def __init__(self, prob):
        self.p = prob
        self.dim = prob["dim"]
        self.n = prob["n"][:self.dim]
        self.dx = [(prob["hi"][d] - prob["lo"][d]) / self.n[d] for d in range(self.dim)]
        self.bc = [torch.tensor(s[:self.dim + 2], dtype=torch.float64, device="cuda") for s in prob["bc_state"]]

    # boundary conditions of direction d: three ghost cells per side
    def ghosts(self, V, d, t):
        sides = []
        for side, code in ((0, self.p["bc_lo"][d]), (1, self.p["bc_hi"][d])):
            near = V[..., :3] if side == 0 else V[..., -3:]
            far = V[..., -3:] if side == 0 else V[..., :3]
            edge = (V[..., :1] if side == 0 else V[..., -1:]).expand_as(near)
            sign = torch.ones(self.dim + 2, dtype=torch.float64, device="cuda")
            sign[1 + d] = -1.0
            shape = [-1] + [1] * self.dim
            mirror = near.flip(-1) * sign.reshape(shape)
            fixed = [b.reshape(shape).expand_as(near) for b in self.bc]
            if code == P.BC_PERIODIC:
                g = far
            elif code == P.BC_TRANSMISSIVE:
                g = edge
            elif code == P.BC_REFLECT:
                g = mirror
            elif code == P.BC_INFLOW:
                g = fixed[0]
            else:   # double Mach bottom and top: V is [var, x, y]
                x = (self.p["lo"][0] + (torch.arange(self.n[0], dtype=torch.float64, device="cuda") + 0.5)
                     * self.dx[0]).reshape(1, -1, 1)
                if code == P.BC_DMR_BOTTOM:
                    g = torch.where(x < 1.0 / 6.0, fixed[0], mirror)
                else:
                    g = torch.where(x < 1.0 / 6.0 + (1.0 + 20.0 * t) / math.sqrt(3.0), fixed[0], fixed[1])
            sides.append(g)
        return torch.cat([sides[0], V, sides[1]], dim=-1)

    def speeds(self, U, d):
        g, dim = self.p["gamma"], self.dim
        u = [U[1 + k] / U[0] for k in range(dim)]
        p = (g - 1.0) * (U[dim + 1] - 0.5 * U[0] * sum(x * x for x in u))
        return u, p, torch.sqrt(g * p / U[0])

    @staticmethod
    def recon(a, b, c, d, e, lam, eps):
        q = [0.5 * (c + d), 1.5 * c - 0.5 * b, c / 3 + 5 * d / 6 - e / 6, a / 3 - 7 * b / 6 + 11 * c / 6]
        k = 13.0 / 12.0
        beta = [(d - c) ** 2, (c - b) ** 2, k * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2,
                k * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2]
        tau = k * (e - 4 * d + 6 * c - 4 * b + a) ** 2 + 0.25 * (e - 2 * d + 2 * b - a) ** 2
        E = (b - 2 * c + d) ** 2 / 45.0
        al = [w * (1.0 + lam * tau / (lam * bk + (E if i < 2 else 0.0) + eps))
              for i, (w, bk) in enumerate(zip((0.4, 0.2, 0.3, 0.1), beta))]
        return sum(x * y for x, y in zip(al, q)) / sum(al)

    # numerical fluxes of the faces along d of a padded array V[var, lines..., along + 6]
    def fluxes(self, V, d, alpha_g):
        g, dim = self.p["gamma"], self.dim
        nv, last, nf = dim + 2, dim + 1, V.shape[-1] - 5
        u, p, c = self.speeds(V, d)
        H = (V[last] + p) / V[0]
        F = [V[1 + d]] + [V[1 + k] * u[d] + (p if k == d else 0.0) for k in range(dim)] + [(V[last] + p) * u[d]]
        st = lambda x, m: x[..., m:m + nf]   # noqa: E731  stencil cell m of every face
        sq = torch.sqrt(V[0])
        sa, sb = st(sq, 2), st(sq, 3)
        roe = lambda x: (sa * st(x, 2) + sb * st(x, 3)) / (sa + sb)   # noqa: E731
        ru, rH = [roe(x) for x in u], roe(H)
        q2 = sum(x * x for x in ru)
        rc = torch.sqrt((g - 1.0) * (rH - 0.5 * q2))
        b1 = (g - 1.0) / rc ** 2

        def left(x):   # L x, fields u - c, u, shear, u + c
            t1 = b1 * (0.5 * q2 * x[0] - sum(ru[k] * x[1 + k] for k in range(dim)) + x[last])
            a = (ru[d] * x[0] - x[1 + d]) / rc
            shear = [x[1 + k] - ru[k] * x[0] for k in range(dim) if k != d]
            return [0.5 * (t1 + a), x[0] - t1] + shear + [0.5 * (t1 - a)]

        def right(w):   # R w
            out = [w[0] + w[1] + w[last]]
            s, e = 2, 0.0
            for k in range(dim):
                m = ru[k] * out[0]
                if k == d:
                    m = m + rc * (w[last] - w[0])
                else:
                    m = m + w[s]
                    e = e + ru[k] * w[s]
                    s += 1
                out.append(m)
            out.append(rH * (w[0] + w[last]) + ru[d] * rc * (w[last] - w[0]) + 0.5 * q2 * w[1] + e)
            return out

        dU = [st(x, 0) - st(x, 5) + 5 * (st(x, 4) - st(x, 1)) + 10 * (st(x, 2) - st(x, 3)) for x in V]
        dv = [x / 60.0 for x in left(dU)]
        rt2 = sa * sa * sb * sb
        sig = [x * x / rt2 for x in dv]
        eps_h = self.p["C_thr"] * (self.dx[d] / self.p["L_char"]) ** self.p["alpha_thr"]
        smooth = sig[0] < eps_h
        for s in range(1, nv):
            smooth = smooth & (sig[s] < eps_h)
        alpha = []
        for s in range(nv):
            lam = (u[d] - c if s == 0 else u[d] + c if s == last else u[d]).abs()
            if alpha_g is not None:
                alpha.append(alpha_g[0 if s == 0 else 2 if s == last else 1])
                continue
            m = st(lam, 0)
            for k in range(1, 6):
                m = torch.where(st(lam, k) > m, st(lam, k), m)
            alpha.append(m)
        lin = [(st(x, 0) - 8 * st(x, 1) + 37 * st(x, 2) + 37 * st(x, 3) - 8 * st(x, 4) + st(x, 5)) / 60.0 for x in F]
        lin = [x + y for x, y in zip(lin, right([a * x for a, x in zip(alpha, dv)]))]
        vw = [left([st(x, m) for x in V]) for m in range(6)]
        gw = [left([st(x, m) for x in F]) for m in range(6)]
        wch = []
        for s in range(nv):
            fp = [0.5 * (gw[m][s] + alpha[s] * vw[m][s]) for m in range(6)]
            fm = [0.5 * (gw[m][s] - alpha[s] * vw[m][s]) for m in range(6)]
            lam = self.p["c_lambda"] * sig[s]
            wch.append(self.recon(*fp[:5], lam, self.p["eps"]) + self.recon(*fm[:0:-1], lam, self.p["eps"]))
        return [torch.where(smooth, x, y) for x, y in zip(lin, right(wch))]

    def _along(self, U, d):   # direction d last (x is the last axis, y the one before, ...)
        return U.movedim(self.dim - d, -1)

    def _chunks(self, V):   # pieces of whole lines, a few million faces each
        if self.dim == 1:
            return [slice(None)]
        per = max(1, int(2e6 // (V[0, 0].numel())))
        return [slice(i, min(i + per, V.shape[1])) for i in range(0, V.shape[1], per)]

    def alpha_lf(self, U, d):
        if self.p["splitting"] != "lf":
            return None
        u, _, c = self.speeds(U, d)
        return [(u[d] - c).abs().max(), u[d].abs().max(), (u[d] + c).abs().max()]

    def rhs(self, U, t):
        out = torch.zeros_like(U)
        for d in range(self.dim):
            ag = self.alpha_lf(U, d)
            V = self.ghosts(self._along(U, d), d, t)
            o = self._along(out, d)
            for c in self._chunks(V):
                F = torch.stack(self.fluxes(V[:, c] if self.dim > 1 else V, d, ag))
                piece = (F[..., :-1] - F[..., 1:]) / self.dx[d]
                if self.dim > 1:
                    o[:, c] += piece
                else:
                    o += piece
        return out

    def vjp(self, U, w, t):
        grad = torch.zeros_like(U)
        for d in range(self.dim):
            leaf = U.clone().requires_grad_(True)
            V = self.ghosts(self._along(leaf, d), d, t)
            Vd = V.detach()
            G = torch.zeros_like(Vd)
            wd = self._along(w, d)
            for c in self._chunks(Vd):
                x = Vd[:, c].clone().requires_grad_(True)
                F = torch.stack(self.fluxes(x, d, None))
                ((F[..., :-1] - F[..., 1:]) / self.dx[d] * wd[:, c]).sum().backward()
                G[:, c] = x.grad
            V.backward(G)
            grad += leaf.grad
        return grad

    def advance(self, U, t, t_end, steps):
        floor = 0.0
        for d in range(self.dim):
            for side, codes in ((0, (P.BC_INFLOW, P.BC_DMR_BOTTOM, P.BC_DMR_TOP)), (1, (P.BC_DMR_TOP,))):
                if self.p["bc_lo"][d] in codes or self.p["bc_hi"][d] in codes:
                    u, _, c = self.speeds(self.bc[side], 0)
                    floor = max(floor, float(sum((u[e].abs() + c) / self.dx[e] for e in range(self.dim))))
        k = 0
        while k < steps and t < t_end:
            u, _, c = self.speeds(U, 0)
            smax = max(floor, float(sum((u[e].abs() + c) / self.dx[e] for e in range(self.dim)).max()))
            dt, end = self.p["cfl"] / smax, False
            if t + dt >= t_end:
                dt, end = t_end - t, True
            A = U + dt * self.rhs(U, t)
            B = 0.75 * U + 0.25 * (A + dt * self.rhs(A, t + dt))
            U = U / 3.0 + 2.0 / 3.0 * (B + dt * self.rhs(B, t + 0.5 * dt))
            t, k = (t_end if end else t + dt), k + 1
        return U, t, k


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "boxes"):
        return None   # thousands of whole runs
    prob, U, t = _problem(case, seed)
    if case["precision"] != "fp64":
        U = U.float().double()
    ref = _Ref(prob)
    if kind in ("tube", "grid"):
        if case["kind"] == "tube" and case["n"] > 400 and not case["steps"]:
            return None   # thousands of steps
        V, t, k = ref.advance(U, t, prob["t_end"], case["steps"] or 2 ** 31 - 1)
        return dict(U=V, t=t, steps=k)
    if kind == "rhs":
        return ref.rhs(U, t)
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.randn(U.shape, dtype=torch.float64 if case["precision"] == "fp64" else torch.float32, device="cuda",
                    generator=g).double()
    return dict(rhs=ref.rhs(U, t), grad=ref.vjp(U, w, t))
