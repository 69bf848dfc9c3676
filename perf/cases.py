"""Performance cases: the calls a user of this framework makes, over the sizes it is used at.

A case is one pass of one public entry point on one problem.  Sizes and flows are those of
the package's workloads (paper_2410_05489_gb300/problems.py), its benchmark and its tests: the
Sod tube, the isentropic vortex, random Riemann data, Configuration 3, the high-Mach jet, the
mixed batch and the perturbed vortex of the adjoint.  The initial data are rebuilt here on the
device from a seed (centre, strength, states and perturbations drawn), so that a preparation
takes milliseconds and another seed gives other inputs.

exact() evaluates the same scheme in plain torch float64 operations, written from the method
(finite volumes, ASE-DF reconstruction, Lax-Friedrichs or gas-kinetic flux, SSP-RK3; gradients
by torch autograd): none of the package's arithmetic is used there.
"""
from __future__ import annotations

import math
from decimal import Decimal, getcontext
from fractions import Fraction
from functools import lru_cache

import torch

from paper_2410_05489_gb300 import adjoint, ase_df, batch
from paper_2410_05489_gb300.problems import JET_U, Problem

F64 = torch.float64
DEV = "cuda"


# ----------------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: one residual of the 200-cell Sod tube (a 1D solver's inner loop)
        {"name": "residual_sod_200_r5", "kind": "residual", "flow": "sod", "ndim": 1, "nx": 200, "ny": 1, "order": 5},
        # a short 1D run: CFL steps of the Sod tube, each step a chain of small launches
        {"name": "run_sod_200_r5", "kind": "run", "flow": "sod", "ndim": 1, "nx": 200, "ny": 1, "order": 5, "steps": 8},
        # a long 1D line of Riemann data at the highest order, odd size
        {"name": "residual_riemann1d_65537_r9", "kind": "residual", "flow": "riemann", "ndim": 1, "nx": 65537, "ny": 1,
         "order": 9},
        # a small 2D run, the start of a convergence study
        {"name": "run_vortex_64_r7", "kind": "run", "flow": "vortex", "ndim": 2, "nx": 64, "ny": 64, "order": 7,
         "steps": 4},
        # the largest smooth call: one CFL step of the 1024^2 vortex at order 9 (the benchmark's step)
        {"name": "run_vortex_1024_r9", "kind": "run", "flow": "vortex", "ndim": 2, "nx": 1024, "ny": 1024, "order": 9,
         "steps": 1},
        # ragged sizes at order 7 with a wall: one residual of a smooth random field
        {"name": "residual_smooth_701x403_r7", "kind": "residual", "flow": "smooth", "ndim": 2, "nx": 701, "ny": 403,
         "order": 7},
        # shocks: one CFL step of Configuration 3 at order 5
        {"name": "run_config3_512_r5", "kind": "run", "flow": "config3", "ndim": 2, "nx": 512, "ny": 512, "order": 5,
         "steps": 1},
        # the largest grid: one residual of the Mach 20000 jet entering its 1600 x 800 domain
        {"name": "residual_jet_1600x800_r9", "kind": "residual", "flow": "jet", "ndim": 2, "nx": 1600, "ny": 800,
         "order": 9},
        # the gas-kinetic solver on the paper's timing workload
        {"name": "gks_config3_400_r9", "kind": "gks", "flow": "config3", "ndim": 2, "nx": 400, "ny": 400, "order": 9},
        # many independent problems, 1D and 2D, orders 3 to 9 mixed, advanced together
        {"name": "batch_64", "kind": "batch", "problems": 64, "n1_hi": 16384, "n2_hi": 512, "mix": 20241008},
        # a gradient of one residual on the adjoint workload's grid (backward pass)
        {"name": "adjoint_vortex_256_r7", "kind": "adjoint", "flow": "perturbed", "ndim": 2, "nx": 256, "ny": 256,
         "order": 7},
        # a training-style pass: a short checkpointed rollout and its gradient
        {"name": "rollout_vortex_96_r7", "kind": "rollout", "flow": "perturbed", "ndim": 2, "nx": 96, "ny": 96,
         "order": 7, "steps": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["residual", "residual", "residual", "run", "run", "gks", "batch", "adjoint", "rollout"])
    if kind == "batch":
        return {"kind": "batch", "problems": _log_int(rng, 8, 64), "n1_hi": 16384, "n2_hi": _log_int(rng, 96, 512),
                "mix": rng.randrange(1 << 30)}
    order = rng.choice([3, 5, 7, 9])
    case = {"kind": kind, "order": order, "ndim": 2}
    if kind in ("adjoint", "rollout"):
        case["order"] = rng.choice([5, 7, 9])
        case["flow"] = "perturbed"
        hi = 512 if kind == "adjoint" else 128
        case["nx"], case["ny"] = _log_int(rng, 48, hi), _log_int(rng, 48, hi)
        if kind == "rollout":
            case["steps"] = rng.randint(2, 5)
        return case
    if kind == "gks":
        case["flow"] = rng.choice(["config3", "vortex"])
        case["nx"], case["ny"] = _log_int(rng, 64, 400), _log_int(rng, 64, 400)
        return case
    if rng.random() < 0.25:
        case["ndim"], case["ny"] = 1, 1
        case["flow"] = rng.choice(["sod", "riemann"])
        case["nx"] = _log_int(rng, 128, 131072)
    else:
        case["flow"] = rng.choice(["vortex", "smooth", "config3", "riemann"] + (["jet"] if kind == "residual" else []))
        case["nx"], case["ny"] = _log_int(rng, 48, 1024), _log_int(rng, 48, 1024)
        if case["flow"] == "jet":
            case["nx"] = max(case["nx"], 200)
            case["ny"] = max(case["ny"], 100)
    if kind == "run":
        case["steps"] = 1 if case["nx"] * case["ny"] > 40000 else rng.randint(1, 4)
    return case


# ----------------------------------------------------------------------------------
# problems and their initial data
# ----------------------------------------------------------------------------------
def _problem(case) -> Problem:
    flow, nx, ny, r = case["flow"], case["nx"], case["ny"], case["order"]
    if flow in ("vortex", "perturbed"):
        return Problem(ndim=2, nx=nx, ny=ny, x1=10.0, y1=10.0, order=r, bc=("periodic",) * 4)
    if flow == "smooth":  # periodic in x, a wall below, outflow above
        return Problem(ndim=2, nx=nx, ny=ny, order=r, bc=("periodic", "periodic", "reflect", "outflow"))
    if flow == "jet":
        return Problem(ndim=2, nx=nx, ny=ny, y0=-0.25, y1=0.25, order=r, gamma=5.0 / 3.0,
                       bc=("inflow", "outflow", "outflow", "outflow"), inflow=(5.0, JET_U, 0.0, 0.4127),
                       inflow_lo=-0.05, inflow_hi=0.05)
    return Problem(ndim=case["ndim"], nx=nx, ny=ny, order=r)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _rand(g, *shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, dtype=F64, device=DEV)


def _cons(prim, gamma):
    rho, p = prim[0], prim[-1]
    vel = prim[1:-1]
    kin = sum(0.5 * rho * v * v for v in vel)
    return torch.stack([rho] + [rho * v for v in vel] + [p / (gamma - 1.0) + kin])


def _average(pb, fn):
    """Cell averages of the conservative variables of fn(x[, y]) by 4-point Gauss quadrature."""
    nodes, weights = _gauss(4)
    nx, ny = pb.nx, pb.nyc
    cx = torch.arange(nx, dtype=F64, device=DEV)
    cy = torch.arange(ny, dtype=F64, device=DEV)
    out = 0.0
    for tx, wx in zip(nodes, weights):
        x = pb.x0 + (cx + float(tx)) * pb.dx
        if pb.ndim == 1:
            out = out + float(wx) * _cons(fn(x[None, :]), pb.gamma)
            continue
        for ty, wy in zip(nodes, weights):
            y = pb.y0 + (cy + float(ty)) * pb.dy
            out = out + float(wx) * float(wy) * _cons(fn(*torch.broadcast_tensors(x[None, :], y[:, None])), pb.gamma)
    return out.contiguous()


def _state(case, pb, g):
    flow = case["flow"]
    if flow == "sod":  # the tube, its diaphragm and right state drawn near the textbook's
        u = _rand(g, 3).tolist()
        xd, rr, pr = 0.45 + 0.1 * u[0], 0.115 + 0.02 * u[1], 0.09 + 0.02 * u[2]
        return _average(pb, lambda x: (torch.where(x < xd, 1.0, rr), torch.zeros_like(x), torch.where(x < xd, 1.0, pr)))
    if flow in ("vortex", "perturbed"):
        u = _rand(g, 3).tolist()
        xc, yc, eps = 4.0 + 2.0 * u[0], 4.0 + 2.0 * u[1], 4.5 + u[2]
        gam = pb.gamma

        def prim(x, y):
            dx = torch.remainder(x - xc + 5.0, 10.0) - 5.0
            dy = torch.remainder(y - yc + 5.0, 10.0) - 5.0
            e = torch.exp(0.5 * (1.0 - dx * dx - dy * dy))
            T = 1.0 - (gam - 1.0) * eps * eps / (8.0 * gam * math.pi ** 2) * e * e
            rho = T ** (1.0 / (gam - 1.0))
            return rho, 1.0 - eps / (2.0 * math.pi) * e * dy, 1.0 + eps / (2.0 * math.pi) * e * dx, rho * T

        W = _average(pb, prim)
        if flow == "perturbed":  # 1 % random density, velocity and pressure held
            f = 1.0 + 0.01 * _rand(g, pb.nyc, pb.nx, lo=-1.0)
            p = W[3] - 0.5 * (W[1] ** 2 + W[2] ** 2) / W[0]
            W = torch.stack([W[0] * f, W[1] * f, W[2] * f, p + 0.5 * (W[1] ** 2 + W[2] ** 2) / W[0] * f])
        return W
    if flow == "smooth":  # random Fourier modes of O(1) relative variation
        k = (1.0 + torch.floor(_rand(g, 4, 3, 2, hi=12.0))).tolist()
        ph = _rand(g, 4, 3, 2, hi=2.0 * math.pi).tolist()
        amp = _rand(g, 4, 3, lo=-1.0).tolist()
        base, rng = (1.0, 0.5, -0.3, 1.0), (0.15, 0.3, 0.3, 0.15)

        def prim(x, y):
            out = []
            for c in range(4):
                f = torch.full_like(x, base[c])
                for m in range(3):
                    f = f + rng[c] * amp[c][m] * torch.sin(2 * math.pi * k[c][m][0] * x + ph[c][m][0]) * torch.sin(
                        2 * math.pi * k[c][m][1] * y + ph[c][m][1])
                out.append(f)
            return out

        return _average(pb, prim)
    X = pb.x0 + (torch.arange(pb.nx, dtype=F64, device=DEV) + 0.5) * pb.dx
    if pb.ndim == 1:  # riemann: two random states
        rho, p = torch.exp(_rand(g, 2, lo=math.log(0.1), hi=math.log(10.0))), torch.exp(
            _rand(g, 2, lo=math.log(0.1), hi=math.log(10.0)))
        u = _rand(g, 2, lo=-2.0, hi=2.0)
        s = (X >= float(_rand(g, 1, lo=0.3, hi=0.7))).long()[None, :]
        return _cons((rho[s], u[s], p[s]), pb.gamma).contiguous()
    Y = pb.y0 + (torch.arange(pb.ny, dtype=F64, device=DEV) + 0.5) * pb.dy
    X, Y = X[None, :].expand(pb.ny, pb.nx), Y[:, None].expand(pb.ny, pb.nx)
    if flow == "riemann":  # four random quadrants
        rho, p = torch.exp(_rand(g, 4, lo=math.log(0.1), hi=math.log(10.0))), torch.exp(
            _rand(g, 4, lo=math.log(0.1), hi=math.log(10.0)))
        u, v = _rand(g, 4, lo=-2.0, hi=2.0), _rand(g, 4, lo=-2.0, hi=2.0)
        q = (X >= 0.5).long() + 2 * (Y >= 0.5).long()
        return _cons((rho[q], u[q], v[q], p[q]), pb.gamma).contiguous()
    if flow == "config3":  # the four states of Configuration 3, the corner drawn near (0.7, 0.7)
        xs, ys = _rand(g, 2, lo=0.65, hi=0.75).tolist()
        q = (X >= xs).long() + 2 * (Y >= ys).long()
        tab = torch.tensor([[0.138, 0.5323, 0.5323, 1.5], [1.206, 0.0, 1.206, 0.0], [1.206, 1.206, 0.0, 0.0],
                            [0.129, 0.3, 0.3, 1.5]], dtype=F64, device=DEV)
        tab[0] = tab[0] * (1.0 + 0.01 * _rand(g, 4))
        return _cons(tuple(tab[c][q] for c in range(4)), pb.gamma).contiguous()
    # jet: the beam has entered to a drawn depth, with a smooth rim of a few cells
    depth, amb = 0.1 + 0.3 * float(_rand(g, 1)), 1.0 + 0.05 * _rand(g, pb.ny, pb.nx)
    w = 3.0 * max(pb.dx, pb.dy)
    f = 0.25 * (1.0 - torch.tanh((X - depth) / w)) * (1.0 - torch.tanh((Y.abs() - 0.05) / w))
    rho = 0.5 + 4.5 * f
    return _cons((rho, JET_U * f, torch.zeros_like(f), 0.4127 * amb * (1.0 + 1e3 * f * (1.0 - f))), pb.gamma).contiguous()


def _mix(case):
    """Problems of a batch: half 1D, half 2D, sizes log-uniform, orders 3 to 9."""
    g = torch.Generator()
    g.manual_seed(case["mix"])
    n = case["problems"]
    u = torch.rand(n, 3, generator=g, dtype=F64).tolist()
    sub = []
    for i in range(n):
        r = 3 + 2 * int(4 * u[i][1])
        lo, hi = (128, case["n1_hi"]) if i < n // 2 else (64, case["n2_hi"])
        m = int(round(math.exp(math.log(lo) + u[i][0] * (math.log(hi) - math.log(lo)))))
        sub.append({"flow": "riemann", "ndim": 1 if i < n // 2 else 2, "nx": m, "ny": 1 if i < n // 2 else m, "order": r})
    return sub


def _inputs(case, seed):
    """-> (problem, W, sx, sy): the state and the face strengths a residual of it has produced."""
    pb = _problem(case)
    W = _state(case, pb, _gen(seed))
    _, sx, sy = _residual(pb, W, *_zero_sigma(pb))
    return pb, W, sx.contiguous(), sy.contiguous()


def _zero_sigma(pb):
    return torch.zeros(pb.sx_shape, dtype=F64, device=DEV), torch.zeros(pb.sy_shape, dtype=F64, device=DEV)


def _cotangents(pb, seed):
    g = _gen(seed + 7919)
    return torch.randn(*pb.state_shape, generator=g, dtype=F64, device=DEV)


# ----------------------------------------------------------------------------------
# what is measured
# ----------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        sub = _mix(case)
        pbs = [_problem(s) for s in sub]
        W = [_state(s, p, _gen(seed + 101 * i)) for i, (s, p) in enumerate(zip(sub, pbs))]
        sig = [_residual(p, w, *_zero_sigma(p))[1:] for p, w in zip(pbs, W)]
        return {"kind": kind, "batch": batch.Batch(pbs), "W": torch.cat([w.reshape(-1) for w in W]),
                "sx": torch.cat([x.reshape(-1) for x, _ in sig]),
                "sy": torch.cat([y.reshape(-1) for p, (_, y) in zip(pbs, sig) if p.ndim == 2])}
    pb, W, sx, sy = _inputs(case, seed)
    st = {"kind": kind, "pb": pb, "W": W, "sx": sx, "sy": sy, "solver": ase_df.Solver(pb), "steps": case.get("steps")}
    if kind == "adjoint":
        st["Lbar"] = _cotangents(pb, seed)
    if kind in ("gks", "rollout"):
        st["dt"] = 0.4 / _max_speed(pb, W)
    if kind == "rollout":
        st["Wbar"] = _cotangents(pb, seed)
    return st


def run(state):
    kind = state["kind"]
    if kind == "batch":  # one CFL step of every problem from the given state
        b = state["batch"]
        b.W.copy_(state["W"])
        b.sx.copy_(state["sx"])
        b.sy.copy_(state["sy"])
        b.run(1)
        return {"W": b.W, "sx": b.sx, "sy": b.sy}
    s, W, sx, sy = state["solver"], state["W"], state["sx"], state["sy"]
    if kind == "residual":
        L, sxo, syo = s.residual(W, sx, sy)
        return {"L": L, "sx": sxo, "sy": syo} if s.pb.ndim == 2 else {"L": L, "sx": sxo}
    if kind == "run":  # CFL steps from the given state, as graph replays
        s.W.copy_(W)
        s.sx.copy_(sx)
        s.sy.copy_(sy)
        s.run(state["steps"])
        return {"W": s.W, "sx": s.sx, "sy": s.sy} if s.pb.ndim == 2 else {"W": s.W, "sx": s.sx}
    if kind == "gks":
        L, Lt, sxo, syo = s.gks_residual(state["dt"], W, sx, sy)
        return {"L": L, "Lt": Lt, "sx": sxo, "sy": syo}
    if kind == "adjoint":
        Wb, sxb, syb = s.residual_adjoint(W, sx, sy, Lbar=state["Lbar"])
        return {"Wbar": Wb, "sxbar": sxb, "sybar": syb}
    W0 = W.detach().requires_grad_(True)  # rollout and its gradient
    WT = adjoint.rollout(s, W0, state["steps"], state["dt"], every=2)
    (grad,) = torch.autograd.grad(WT, W0, state["Wbar"])
    return {"W": WT.detach(), "grad": grad}


def _cells_flops(ndim, r, nx, ny):
    """Algorithmic operations of one Lax-Friedrichs residual (both sweeps): per face 2C(2r-1)
    for the normal reconstruction, 2CG(2r-1) for the tangential one, and the Gauss points."""
    C, G = (4, 1 if r == 3 else (r - 1) // 2) if ndim == 2 else (3, 1)
    phi = 70 if ndim == 2 else 56
    face = 2 * C * (2 * r - 1) + (2 * C * G * (2 * r - 1) if ndim == 2 else 0) + G * (phi + 2 * C + 1) + 1
    faces = (nx + 1) * ny + ((ny + 1) * nx if ndim == 2 else 0)
    return face * faces


def _gks_flops(r, nx, ny):
    G = 1 if r == 3 else (r - 1) // 2
    face = 16 * (2 * r - 1) + 8 + 8 * G * (3 * (2 * r - 1) + 1) + G * (1365 + 43 + 17) + 1
    return face * ((nx + 1) * ny + (ny + 1) * nx)


def work(case):
    if case["kind"] == "batch":
        sub = _mix(case)
        cells = sum((3 if s["ndim"] == 1 else 4) * s["nx"] * s["ny"] for s in sub)
        sig = sum((s["nx"] + 1) * s["ny"] + ((s["ny"] + 1) * s["nx"] if s["ndim"] == 2 else 0) for s in sub)
        return {"bytes": 16 * (cells + sig), "flops": 3 * sum(_cells_flops(s["ndim"], s["order"], s["nx"], s["ny"])
                                                               for s in sub)}
    nd, r, nx, ny = case["ndim"], case["order"], case["nx"], case["ny"]
    w = (3 if nd == 1 else 4) * nx * ny
    sig = (nx + 1) * ny + ((ny + 1) * nx if nd == 2 else 0)
    res = _cells_flops(nd, r, nx, ny)
    kind = case["kind"]
    if kind == "residual":
        return {"bytes": 16 * (w + sig), "flops": res}
    if kind == "run":
        return {"bytes": 16 * (w + sig), "flops": 3 * case["steps"] * res}
    if kind == "gks":
        return {"bytes": 8 * (3 * w + 2 * sig), "flops": _gks_flops(r, nx, ny)}
    grad = {5: 1.4197, 7: 1.4451, 9: 1.4552}[r]  # edges per operation of the reverse-mode graph
    if kind == "adjoint":
        return {"bytes": 8 * (3 * w + 2 * sig), "flops": int(res * (1 + 2 * grad))}
    return {"bytes": 8 * 4 * w, "flops": int(3 * case["steps"] * res * (2 + 2 * grad))}


# ----------------------------------------------------------------------------------
# the scheme in plain float64 torch operations
# ----------------------------------------------------------------------------------
@lru_cache(maxsize=None)
def _gauss(n):
    """Gauss-Legendre nodes and weights on [0, 1], ascending (40-digit decimals)."""
    getcontext().prec = 45
    nodes, weights = [], []
    for i in range(n):
        x = Decimal(repr(math.cos(math.pi * (n - i - 0.25) / (n + 0.5))))
        for _ in range(8):
            p0, p1 = Decimal(1), x
            for k in range(2, n + 1):
                p0, p1 = p1, ((2 * k - 1) * x * p1 - (k - 1) * p0) / k
            d = n * (x * p1 - p0) / (x * x - 1)
            x -= p1 / d
        nodes.append(Fraction((x + 1) / 2))
        weights.append(Fraction(1 / ((1 - x * x) * d * d)))
    return nodes, weights


@lru_cache(maxsize=None)
def _poly(offsets):
    """Rows q: weights of the cell averages in the coefficient of xi^q of the polynomial on
    cells [t-1, t], t in offsets (exact rationals)."""
    n = len(offsets)
    A = [[(Fraction(t) ** (q + 1) - Fraction(t - 1) ** (q + 1)) / (q + 1) for q in range(n)] +
         [Fraction(int(i == j)) for j in range(n)] for i, t in enumerate(offsets)]
    for c in range(n):
        piv = next(i for i in range(c, n) if A[i][c] != 0)
        A[c], A[piv] = A[piv], A[c]
        A[c] = [v / A[c][c] for v in A[c]]
        for i in range(n):
            if i != c and A[i][c] != 0:
                A[i] = [u - A[i][c] * v for u, v in zip(A[i], A[c])]
    return [row[n:] for row in A]


@lru_cache(maxsize=None)
def _weights(offsets, xi, deriv):
    P = _poly(offsets)
    n = len(offsets)
    if deriv:
        return [float(sum(q * xi ** (q - 1) * P[q][i] for q in range(1, n))) for i in range(n)]
    return [float(sum(xi ** q * P[q][i] for q in range(n))) for i in range(n)]


def _dot(w, v):
    acc = w[0] * v[0]
    for a, b in zip(w[1:], v[1:]):
        acc = acc + a * b
    return acc


def _reconstruct(v, s, r, thres, points, deriv=False):
    """v: the r stencil arrays [C, ...]; s: the r - 1 face-strength arrays.  Values (and
    derivatives) of the polynomial of Algorithm 1 at the points xi."""
    K = (r - 1) // 2
    A = {3: s[K - 1] + s[K]}
    if r >= 5:
        A[5] = (s[K - 2] + s[K - 1]) + (s[K] + s[K + 1])
    if r >= 7:
        A[7] = A[5] + (s[K - 3] + s[K + 2])
    if r >= 9:
        A[9] = A[7] + (s[K - 4] + s[K + 3])
    alpha = lambda a: thres / torch.clamp(a, min=thres)  # noqa: E731
    c = v[K]
    cells = lambda h: (tuple(range(-h, h + 1)), v[K - h:K + h + 1])  # noqa: E731
    outs = []
    if r >= 5:
        subs = [tuple(range(k - 2, k + 1)) for k in range(3)]
        beta = []
        for k, off in enumerate(subs):
            u, P = v[K + k - 2:K + k + 1], _poly(off)
            c1, c2 = (_dot([float(x) for x in P[q]], u) for q in (1, 2))
            beta.append(c1 * (c1 - 2.0 * c2) + (16.0 / 3.0) * c2 * c2)
        b5 = (beta[0] + 4.0 * beta[1] + beta[2]) / 6.0 + (beta[0] - beta[2]).abs()
        tau = ((b5 - beta[0]).abs() + (b5 - beta[1]).abs() + (b5 - beta[2]).abs()) / 3.0
        d5, d3 = 0.85, (0.01125, 0.1275, 0.01125)
        w5 = d5 * (1.0 + tau ** 2 / (b5 + 1e-6) ** 2)
        w3 = [d * (1.0 + tau ** 2 / (b + 1e-6) ** 2) for d, b in zip(d3, beta)]
        tot = w5 + w3[0] + w3[1] + w3[2]
        g5 = w5 / tot / d5
        g3 = [w / tot - g5 * d for w, d in zip(w3, d3)]
        a5 = alpha(A[5])
        a3 = [alpha(s[K - 2] + s[K - 1]), alpha(A[3]), alpha(s[K] + s[K + 1])]
    for xi in points:
        for der in ((False, True) if deriv else (False,)):
            base = 0.0 if der else c
            if r == 3:
                off, u = cells(1)
                out = base + alpha(A[3]) * (_dot(_weights(off, xi, der), u) - base)
                lin = _dot(_weights(off, xi, der), u)
                outs.append(torch.where(A[3] < thres, lin, out))
                continue
            off, u = cells(2)
            out = g5 * (base + a5 * (_dot(_weights(off, xi, der), u) - base))
            for k in range(3):
                out = out + g3[k] * (base + a3[k] * (_dot(_weights(subs[k], xi, der), v[K + k - 2:K + k + 1]) - base))
            for m in range(5, r + 1, 2):
                off, u = cells((m - 1) // 2)
                out = torch.where(A[m] < thres, _dot(_weights(off, xi, der), u), out)
            outs.append(out)
    return outs


def _map_cells(n, lo, hi, g):
    """Interior index of ghost-extended cells -g .. n-1+g, and where a wall mirrors them."""
    i = torch.arange(-g, n + g, device=DEV)
    below, above = i < 0, i >= n
    j = i.clamp(0, n - 1)
    if lo == "periodic":
        return torch.remainder(i, n), torch.zeros_like(below)
    if lo == "reflect":
        j = torch.where(below, -1 - i, j)
    if hi == "reflect":
        j = torch.where(above, 2 * n - 1 - i, j)
    return j, (below & (lo == "reflect")) | (above & (hi == "reflect"))


def _map_faces(n, lo, hi, g):
    f = torch.arange(-g, n + 1 + g, device=DEV)
    if lo == "periodic":
        return torch.where((f >= 0) & (f <= n), f, torch.remainder(f, n))
    j = f.clamp(0, n)
    if lo == "reflect":
        j = torch.where(f < 0, -f, j)
    if hi == "reflect":
        j = torch.where(f > n, 2 * n - f, j)
    return j


def _extend(pb, W, sx, sy):
    """State and face strengths with K + 1 ghost layers."""
    g = (pb.order - 1) // 2 + 1
    bc = pb.bc
    ix, mx = _map_cells(pb.nx, bc[0], bc[1], g)
    We = W[:, :, ix]
    We = torch.cat([We[:1], torch.where(mx, -We[1:2], We[1:2]), We[2:]])
    fx = _map_faces(pb.nx, bc[0], bc[1], g)
    if pb.ndim == 1:
        return We, sx[:, fx], None
    iy, my = _map_cells(pb.ny, bc[2], bc[3], g)
    We = We[:, iy, :]
    We = torch.cat([We[:2], torch.where(my[:, None], -We[2:3], We[2:3]), We[3:]])
    if bc[0] == "inflow":
        yc = pb.y0 + (torch.arange(-g, pb.ny + g, dtype=F64, device=DEV) + 0.5) * pb.dy
        band = (yc > pb.inflow_lo) & (yc < pb.inflow_hi)
        q = _cons([torch.tensor(v, dtype=F64, device=DEV) for v in pb.inflow], pb.gamma)
        ghost = torch.arange(pb.nx + 2 * g, device=DEV) < g
        We = torch.where((band[:, None] & ghost[None, :])[None], q[:, None, None], We)
    fy = _map_faces(pb.ny, bc[2], bc[3], g)
    return We, sx[iy][:, fx], sy[fy][:, ix]


def _lf(a, b, ca, cb, gamma):
    """Lax-Friedrichs flux and face strength of states in (rho, m_n[, m_t], E) order."""
    def prim(q):
        vel = [q[k] / q[0] for k in range(1, len(q) - 1)]
        return vel, (gamma - 1.0) * (q[-1] - 0.5 * q[0] * sum(v * v for v in vel))

    (_, pa), (_, pb_) = prim(a), prim(b)
    ok = (a[0] > 0) & (b[0] > 0) & (pa > 0) & (pb_ > 0)
    a = [torch.where(ok, x, y) for x, y in zip(a, ca)]
    b = [torch.where(ok, x, y) for x, y in zip(b, cb)]
    (va, pa), (vb, pr) = prim(a), prim(b)
    ca_, cb_ = torch.sqrt(gamma * pa / a[0]), torch.sqrt(gamma * pr / b[0])
    lam = torch.maximum(va[0].abs() + ca_, vb[0].abs() + cb_)
    flux = []
    for c in range(len(a)):
        fa, fb = a[c] * va[0], b[c] * vb[0]
        if c == 1:
            fa, fb = fa + pa, fb + pr
        if c == len(a) - 1:
            fa, fb = fa + pa * va[0], fb + pr * vb[0]
        flux.append(0.5 * (fa + fb - lam * (b[c] - a[c])))
    sig = (pa - pr).abs() * (1.0 / pa + 1.0 / pr)
    for k in range(len(va)):
        sig = sig + (va[k] / ca_ - vb[k] / cb_) ** 2
    return flux, torch.where(ok, sig, torch.full_like(sig, 1e30))


def _sweep(pb, We, sn, st, n, m, point_flux, deriv=None):
    """Faces normal to the last axis of We [C][lines + 2g][n + 2g]: Gauss sums of point_flux and
    the face strengths.  deriv = (1/h_n, 1/h_t) adds the slopes of the two states."""
    r = pb.order
    K, g, thres = (r - 1) // 2, (r - 1) // 2 + 1, pb.sigma_thres
    two = pb.ndim == 2
    lo = g - K if two else 0
    L = slice(lo, lo + m + 2 * K) if two else slice(0, 1)
    cut = lambda A, t: A[..., L, g - 1 + t:g - 1 + t + n + 2]  # noqa: E731  cells -1 .. n, shifted by t
    v = [cut(We, t) for t in range(-K, K + 1)]
    s = [cut(sn, t) for t in range(-K + 1, K + 1)]
    both = _reconstruct(v, s, r, thres, (Fraction(0), Fraction(-1)), deriv is not None)
    if deriv is None:
        sides = [(both[0], None), (both[1], None)]
    else:
        sides = [(both[0], both[1] * deriv[0]), (both[2], both[3] * deriv[0])]
    G = (1 if r == 3 else K) if two else 1
    nodes, weights = _gauss(G)
    states = []
    for side, (Q, D) in enumerate(sides):
        cols = slice(side, side + n + 1)
        if not two:
            states.append([(Q[..., cols], None if D is None else D[..., cols], None)])
            continue
        sl = [st[g - K + 1 + k:g - K + 1 + k + m, g - 1 + side:g + side + n] for k in range(2 * K)]
        pts = [x - 1 for x in nodes]
        q = [Q[:, k:k + m, cols] for k in range(2 * K + 1)]
        val = _reconstruct(q, sl, r, thres, pts, deriv is not None)
        if deriv is None:
            states.append([(x, None, None) for x in val])
        else:
            d = [D[:, k:k + m, cols] for k in range(2 * K + 1)]
            # the slopes take the weights of the values' polynomial of their own data
            nd = _reconstruct(d, sl, r, thres, pts)
            states.append([(val[2 * i], nd[i], val[2 * i + 1] * deriv[1]) for i in range(G)])
    mid = slice(g, g + m) if two else slice(0, 1)
    ca, cb = We[:, mid, g - 1:g + n], We[:, mid, g:g + n + 1]
    total, sig = None, 0.0
    for w, a, b in zip(weights, states[0], states[1]):
        out, sg = point_flux(a, b, ca, cb)
        out = [float(w) * x for x in out]
        total = out if total is None else [x + y for x, y in zip(total, out)]
        sig = sig + sg
    return torch.stack(total), sig / G


def _directions(pb, W, sx, sy):
    We, sxe, sye = _extend(pb, W, sx, sy)
    yield We, sxe, sye, pb.nx, pb.nyc
    if pb.ndim == 2:  # rows as sweep lines, the two momenta exchanged
        yield We[[0, 2, 1, 3]].transpose(1, 2), sye.T, sxe.T, pb.ny, pb.nx


def _residual(pb, W, sx, sy):
    flux, sig = [], []
    for We, sn, st, n, m in _directions(pb, W, sx, sy):
        F, s = _sweep(pb, We, sn, st, n, m, lambda a, b, ca, cb: _lf(a[0], b[0], ca, cb, pb.gamma))
        flux.append(F)
        sig.append(s)
    L = -(flux[0][..., 1:] - flux[0][..., :-1]) / pb.dx
    if pb.ndim == 1:
        return L, sig[0], torch.zeros(1, 1, dtype=F64, device=DEV)
    Fy = flux[1][[0, 2, 1, 3]].transpose(1, 2)
    return L - (Fy[:, 1:] - Fy[:, :-1]) / pb.dy, sig[0], sig[1].T


def _max_speed(pb, W):
    vel = [W[k] / W[0] for k in range(1, W.shape[0] - 1)]
    p = (pb.gamma - 1.0) * (W[-1] - 0.5 * W[0] * sum(v * v for v in vel))
    c = torch.sqrt(pb.gamma * p / W[0])
    s = sum((v.abs() + c) / h for v, h in zip(vel, (pb.dx, pb.dy)))
    return float(s.max())


def _step(pb, W, sx, sy, dt):
    L, x1, y1 = _residual(pb, W, sx, sy)
    W1 = W + dt * L
    L, x2, y2 = _residual(pb, W1, x1, y1)
    W2 = 0.75 * W + 0.25 * (W1 + dt * L)
    L, x3, y3 = _residual(pb, W2, x2, y2)
    return W / 3.0 + (2.0 / 3.0) * (W2 + dt * L), x3, y3


def _physical(pb, W):
    kin = sum(W[k] ** 2 for k in range(1, W.shape[0] - 1))
    return bool(((W[0] > 0) & (W[-1] * W[0] - 0.5 * kin > 0)).all())


def _cfl_steps(pb, W, sx, sy, steps):
    for _ in range(steps):
        W, sx, sy = _step(pb, W, sx, sy, pb.cfl / _max_speed(pb, W))
        if not _physical(pb, W):
            return None  # the solver repairs such cells; that path has no closed reference here
    return W, sx, sy


# -- gas-kinetic flux (Sec. 2.2 and Appendix A of the paper) -------------------------
def _moments(U, h, n, half=None):
    """<u^k>, k <= n, of a Maxwellian of mean U and variance h: full line, or u > 0 / u < 0."""
    if half is None:
        m = [torch.ones_like(U), U]
    else:
        z = U / torch.sqrt(2.0 * h)
        e = half * torch.sqrt(h / (2.0 * math.pi)) * torch.exp(-z * z)
        m = [0.5 * torch.erfc(-half * z)]
        m.append(U * m[0] + e)
    for k in range(n - 1):
        m.append(U * m[k + 1] + (k + 1) * h * m[k])
    return m


class _Gas:
    def __init__(self, W, gamma):
        self.rho = W[0]
        self.U, self.V = W[1] / W[0], W[2] / W[0]
        self.p = (gamma - 1.0) * (W[3] - 0.5 * W[0] * (self.U ** 2 + self.V ** 2))
        self.h = self.p / self.rho
        self.K = (4.0 - 2.0 * gamma) / (gamma - 1.0)
        self.mu = _moments(self.U, self.h, 6)
        self.mv = _moments(self.V, self.h, 6)
        self.mx = [torch.ones_like(self.U), self.K * self.h, self.K * (self.K + 2.0) * self.h ** 2]

    def m(self, mu, a, b, c):
        return mu[a] * self.mv[b] * self.mx[c]

    def psi(self, mu, a, b, c=0):
        """<u^a v^b xi^2c psi>, psi = (1, u, v, (u^2 + v^2 + xi^2) / 2)."""
        return [self.m(mu, a, b, c), self.m(mu, a + 1, b, c), self.m(mu, a, b + 1, c),
                0.5 * (self.m(mu, a + 2, b, c) + self.m(mu, a, b + 2, c) + self.m(mu, a, b, c + 1))]

    def poly(self, mu, s, a, b):
        """<u^a v^b (s . psi) psi>."""
        terms = ((s[0], 0, 0, 0), (s[1], 1, 0, 0), (s[2], 0, 1, 0), (0.5 * s[3], 2, 0, 0), (0.5 * s[3], 0, 2, 0),
                 (0.5 * s[3], 0, 0, 1))
        out = [0.0] * 4
        for w, i, j, k in terms:
            out = [o + w * x for o, x in zip(out, self.psi(mu, a + i, b + j, k))]
        return out

    def slope(self, b):
        """a with <psi psi^T> a = b."""
        D, U, V, h = self.K + 2.0, self.U, self.V, self.h
        q = U * U + V * V + D * h
        r2, r3, r4 = b[1] - U * b[0], b[2] - V * b[0], 2.0 * b[3] - q * b[0]
        a3 = (r4 - 2.0 * U * r2 - 2.0 * V * r3) / (D * h * h)
        a2, a1 = r3 / h - V * a3, r2 / h - U * a3
        return [b[0] - U * a1 - V * a2 - 0.5 * a3 * q, a1, a2, a3]


def _gks(pb, dt, a, b, ca, cb):
    gam = pb.gamma
    sig = _lf(a[0], b[0], ca, cb, gam)[1]
    ok = sig < 1e30
    q = [torch.where(ok, a[0], ca), torch.where(ok, b[0], cb)]
    dx = [torch.where(ok, x[1], torch.zeros_like(x[1])) for x in (a, b)]
    dy = [torch.where(ok, x[2], torch.zeros_like(x[2])) for x in (a, b)]
    add = lambda x, y: [i + j for i, j in zip(x, y)]  # noqa: E731
    mul = lambda k, x: [k * i for i in x]  # noqa: E731
    gas = [_Gas(w, gam) for w in q]
    half = [_moments(s.U, s.h, 6, sgn) for s, sgn in zip(gas, (1.0, -1.0))]
    ax = [s.slope([x / s.rho for x in d]) for s, d in zip(gas, dx)]
    ay = [s.slope([x / s.rho for x in d]) for s, d in zip(gas, dy)]

    def both(f):
        return add(*[mul(s.rho, f(s, mu, i)) for i, (s, mu) in enumerate(zip(gas, half))])

    Wc = both(lambda s, mu, i: s.psi(mu, 0, 0))
    gc = _Gas(Wc, gam)
    cx = gc.slope([x / gc.rho for x in both(lambda s, mu, i: s.poly(mu, ax[i], 0, 0))])
    cy = gc.slope([x / gc.rho for x in both(lambda s, mu, i: s.poly(mu, ay[i], 0, 0))])
    A = gc.slope([-x for x in add(gc.poly(gc.mu, cx, 1, 0), gc.poly(gc.mu, cy, 0, 1))])
    T0 = mul(gc.rho, gc.psi(gc.mu, 1, 0))
    T1 = mul(gc.rho, add(gc.poly(gc.mu, cx, 2, 0), gc.poly(gc.mu, cy, 1, 1)))
    T2 = mul(gc.rho, gc.poly(gc.mu, A, 1, 0))
    T3 = both(lambda s, mu, i: s.psi(mu, 1, 0))
    T4 = both(lambda s, mu, i: add(s.poly(mu, ax[i], 2, 0), s.poly(mu, ay[i], 1, 1)))
    pl, pr = gas[0].p, gas[1].p
    tn = pb.gks_c1 * dt + pb.gks_c2 * (pl - pr).abs() / (pl + pr) * dt
    Fd = []
    for d in (dt, 0.5 * dt):
        e = torch.exp(-d / tn)
        c1, c2, c3, c4 = d - tn * (1 - e), tn * tn * (1 - e) - tn * d * e, 0.5 * d * d, tn * (1 - e)
        Fd.append([c1 * t0 + c2 * (t1 - t4) + c3 * t2 + c4 * t3 for t0, t1, t2, t3, t4 in zip(T0, T1, T2, T3, T4)])
    F = [(4.0 * y - x) / dt for x, y in zip(*Fd)]
    Ft = [4.0 * (x - 2.0 * y) / dt ** 2 for x, y in zip(*Fd)]
    return F + Ft, sig


def _gks_residual(pb, W, sx, sy, dt):
    flux, sig = [], []
    h = (pb.dx, pb.dy)
    for d, (We, sn, st, n, m) in enumerate(_directions(pb, W, sx, sy)):
        F, s = _sweep(pb, We, sn, st, n, m, lambda a, b, ca, cb: _gks(pb, dt, a, b, ca, cb),
                      (1.0 / h[d], 1.0 / h[1 - d]))
        flux.append(F)
        sig.append(s)
    out = []
    for k in (0, 4):
        Fx, Fy = flux[0][k:k + 4], flux[1][k:k + 4][[0, 2, 1, 3]].transpose(1, 2)
        out.append(-(Fx[..., 1:] - Fx[..., :-1]) / pb.dx - (Fy[:, 1:] - Fy[:, :-1]) / pb.dy)
    return out[0], out[1], sig[0], sig[1].T


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        W, sx, sy = [], [], []
        for i, s in enumerate(_mix(case)):
            pb = _problem(s)
            w = _state(s, pb, _gen(seed + 101 * i))
            _, x, y = _residual(pb, w, *_zero_sigma(pb))
            out = _cfl_steps(pb, w, x, y, 1)
            if out is None:
                return {"W": None, "sx": None, "sy": None}
            W.append(out[0].reshape(-1))
            sx.append(out[1].reshape(-1))
            if pb.ndim == 2:
                sy.append(out[2].reshape(-1))
        return {"W": torch.cat(W), "sx": torch.cat(sx), "sy": torch.cat(sy)}
    pb, W, sx, sy = _inputs(case, seed)
    if kind == "residual":
        L, x, y = _residual(pb, W, sx, sy)
        return {"L": L, "sx": x, "sy": y} if pb.ndim == 2 else {"L": L, "sx": x}
    if kind == "run":
        out = _cfl_steps(pb, W, sx, sy, case["steps"])
        out = (None, None, None) if out is None else out
        return dict(zip(("W", "sx", "sy"), out)) if pb.ndim == 2 else dict(zip(("W", "sx"), out))
    if kind == "gks":
        L, Lt, x, y = _gks_residual(pb, W, sx, sy, 0.4 / _max_speed(pb, W))
        return {"L": L, "Lt": Lt, "sx": x, "sy": y}
    if kind == "adjoint":
        ins = [t.clone().requires_grad_(True) for t in (W, sx, sy)]
        L, _, _ = _residual(pb, *ins)
        g = torch.autograd.grad(L, ins, _cotangents(pb, seed), allow_unused=True)
        g = [torch.zeros_like(t) if x is None else x for x, t in zip(g, ins)]
        return {"Wbar": g[0], "sxbar": g[1], "sybar": g[2]}
    dt = 0.4 / _max_speed(pb, W)
    W0 = W.clone().requires_grad_(True)
    _, x, y = _residual(pb, W0, *_zero_sigma(pb))
    WT = W0
    for _ in range(case["steps"]):
        WT, x, y = _step(pb, WT, x, y, dt)
    (grad,) = torch.autograd.grad(WT, W0, _cotangents(pb, seed))
    return {"W": WT.detach(), "grad": grad}
