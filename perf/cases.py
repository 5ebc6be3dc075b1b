"""Workloads of the WENO-theta library for timing, through its public entry points.

A case is a dict of plain values; ``prepare`` makes what a program holds before the call (the
initial state on the device, the problem and grid records, the workspace), ``run`` is one call,
``exact`` is the same computation in plain torch binary64, and ``work`` the bytes and flops the
call cannot do without (the state read once and written once; the method's literal operation
count).  Initial data come from ``paper_1504_00731_gb300.workloads`` (grids and seeded initial
states only); every integration starts from the initial state, so passes repeat.
"""
import math

import numpy as np
import torch

from paper_1504_00731_gb300 import binding as B
from paper_1504_00731_gb300 import workloads as W
from paper_1504_00731_gb300.autograd import WenoThetaEuler1D

PERIODIC, OUTFLOW, REFLECTIVE = B.WT_BC_PERIODIC, B.WT_BC_OUTFLOW, B.WT_BC_REFLECTIVE
FLUX = {"euler": B.WT_FLUX_EULER1D, "advection": B.WT_FLUX_ADVECTION, "burgers": B.WT_FLUX_BURGERS}
# literal operations of one cell-update (one cell, one RK3 step)
FLOPS = {"euler": 3696.0, "advection": 938.0, "burgers": 938.0, "euler2d": 10449.0}


def listed():
    return [
        # method-of-lines use: L(u) of a small grid inside the caller's own time integrator
        {"name": "rhs_200", "kind": "rhs", "flux": "euler", "data": "riemann", "n": 200, "strict": False},
        # the paper's scalar test: linear advection of a sine, 200 cells, CFL 0.4 to t = 2 (500 steps)
        {"name": "advection_200", "kind": "step", "flux": "advection", "data": "sine", "n": 200, "cfl": 0.4,
         "steps": 100000, "t_final": 2.0, "strict": False, "host": False},
        # the paper's shock-tube size: Lax's problem on 300 cells to t = 1.3
        {"name": "lax_300", "kind": "step", "flux": "euler", "data": "lax", "n": 300, "cfl": 0.5, "steps": 100000,
         "t_final": 1.3, "strict": False, "host": False},
        # the single-problem workload: 4096 cells, Riemann data with an entropy wave
        {"name": "euler_4096", "kind": "step", "flux": "euler", "data": "riemann", "n": 4096, "cfl": 0.5, "steps": 200,
         "t_final": 0.0, "strict": False, "host": False},
        # a ragged mid-size run: blast waves between walls, more cells than one tile per SM
        {"name": "blast_20001", "kind": "step", "flux": "euler", "data": "blast", "n": 20001, "cfl": 0.5, "steps": 40,
         "t_final": 0.0, "strict": False, "host": False},
        # a high-resolution 1D run that fills the GPU, odd length
        {"name": "euler_999983", "kind": "step", "flux": "euler", "data": "riemann", "n": 999983, "cfl": 0.5, "steps": 8,
         "t_final": 0.0, "strict": False, "host": False},
        # a large scalar run: Burgers with a steepening sine
        {"name": "burgers_1048583", "kind": "step", "flux": "burgers", "data": "sine", "n": 1048583, "cfl": 0.4,
         "steps": 10, "t_final": 0.0, "strict": False, "host": False},
        # a parameter sweep: many small problems of uneven length, 20 steps, a status for each
        {"name": "batch_600_small", "kind": "batch", "nprob": 600, "nmin": 64, "nmax": 1024, "mix": 3, "steps": 20,
         "strict": False, "host": False},
        # the batched workload's length mix (256 .. 65536 cells), a quarter of its problems
        {"name": "batch_1024_mixed", "kind": "batch", "nprob": 1024, "nmin": 256, "nmax": 65536, "mix": 0, "steps": 4,
         "strict": False, "host": False},
        # the paper's Rayleigh-Taylor grid: 120 x 360, gravity, walls in y
        {"name": "rayleigh_taylor_120x360", "kind": "step2d", "data": "rt", "nx": 120, "ny": 360, "cfl": 0.4, "steps": 40,
         "strict": False},
        # a large periodic 2D run: four states and vortices
        {"name": "vortices_2048", "kind": "step2d", "data": "vortices", "nx": 2048, "ny": 2048, "cfl": 0.4, "steps": 2,
         "strict": False},
        # gradients of a loss on the final density of a batch, through torch's autograd
        {"name": "adjoint_48x4096", "kind": "adjoint", "data": "riemann", "nprob": 48, "n": 4096, "steps": 16, "every": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rhs", "step", "step", "step", "batch", "batch", "rhs2d", "step2d", "step2d", "adjoint"])
    strict = rng.random() < 0.08
    if kind == "rhs":
        flux = rng.choice(["euler", "euler", "advection", "burgers"])
        data = rng.choice(["riemann", "smooth", "blast"]) if flux == "euler" else "sine"
        return {"kind": kind, "flux": flux, "data": data, "n": _log(rng, 100, 2000000), "strict": strict}
    if kind == "step":
        flux = rng.choice(["euler", "euler", "euler", "advection", "burgers"])
        data = rng.choice(["riemann", "smooth", "blast", "lax"]) if flux == "euler" else "sine"
        n = _log(rng, 100, 1000000)
        return {"kind": kind, "flux": flux, "data": data, "n": n, "cfl": 0.5 if flux == "euler" else 0.4,
                "steps": max(4, min(200, 8000000 // n)), "t_final": 0.0, "strict": strict, "host": rng.random() < 0.15}
    if kind == "batch":
        nmin = rng.choice([64, 256])
        nmax = _log(rng, 512, 65536)
        nprob = _log(rng, 16, max(17, min(2048, 12000000 // nmax * 2)))
        return {"kind": kind, "nprob": nprob, "nmin": nmin, "nmax": nmax, "mix": rng.randrange(1000),
                "steps": rng.randint(2, 6), "strict": strict, "host": rng.random() < 0.2}
    if kind in ("rhs2d", "step2d"):
        data = rng.choice(["rt", "vortices", "implosion"])
        nx = _log(rng, 40, 1500)
        ny = _log(rng, 40, 1500)
        if data == "implosion":
            ny = nx
        case = {"kind": kind, "data": data, "nx": nx, "ny": ny, "strict": strict}
        if kind == "step2d":
            case.update(cfl=0.4, steps=max(2, min(40, 4000000 // (nx * ny))))
        return case
    n = _log(rng, 200, 8192)
    return {"kind": "adjoint", "data": rng.choice(["riemann", "smooth"]), "nprob": _log(rng, 2, max(3, 200000 // n)),
            "n": n, "steps": rng.randint(6, 16), "every": rng.choice([2, 4, 8, 32])}


# --------------------------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------------------------

def _rng(seed):
    return np.random.default_rng([int(seed), 20150400731 % 2 ** 31])


def _smooth(n, rng):
    """Smooth periodic data on [-1, 1] in which every characteristic field carries a wave."""
    x, dx = W.grid_1d(n, -1.0, 1.0, periodic=True)
    a, ph = rng.uniform(0.05, 0.2, 3), rng.uniform(0, 2 * np.pi, 3)
    return W.cons_1d(1.0 + a[0] * np.sin(np.pi * x + ph[0]), 0.3 + a[1] * np.sin(np.pi * x + ph[1]),
                     1.0 + a[2] * np.cos(np.pi * x + ph[2]))


def _state_1d(case, seed):
    """(u [m][n], lo, hi, boundary, alpha_R) of a single 1D problem."""
    n, data, rng = case["n"], case["data"], _rng(seed)
    if data == "riemann":
        return W.euler_riemann(n, W.riemann_params(int(seed) % 2 ** 31))[0], -5.0, 5.0, OUTFLOW, W.ALPHA_R_SEEDED
    if data == "smooth":
        return _smooth(n, rng), -1.0, 1.0, PERIODIC, 50.0
    if data == "blast":  # the blast waves with their high pressures varied by 5%
        U, _, _ = W.blast_waves(n)
        x = (np.arange(n) + 0.5) / n
        f = 1.0 + 0.05 * rng.uniform(-1.0, 1.0, 2)
        U[2] = U[2] * np.where(x < 0.1, f[0], np.where(x < 0.9, 1.0, f[1]))
        return U, 0.0, 1.0, REFLECTIVE, 10.0
    if data == "lax":  # Lax's data with the pressures and densities varied by 5%
        U, _, _ = W.lax(n)
        f = 1.0 + 0.05 * rng.uniform(-1.0, 1.0, 2)
        left = np.arange(n) < n // 2
        return U * np.where(left, f[0], f[1]), -5.0, 5.0, OUTFLOW, 10.0
    x, _ = W.grid_1d(n, -1.0, 1.0, periodic=True)  # a sine with a random offset, amplitude and phase
    a, b, ph = rng.uniform(0.5, 1.0), rng.uniform(0.0, 0.5), rng.uniform(0.0, 2.0 * np.pi)
    return (b + a * np.sin(np.pi * x + ph))[None, :], -1.0, 1.0, PERIODIC, 50.0


def _state_2d(case, seed):
    """(u [4][ny][nx], lo, hi, boundary x, boundary y, alpha_R, gravity)."""
    nx, ny, data, rng = case["nx"], case["ny"], case["data"], _rng(seed)
    if data == "vortices":
        return (W.euler2d_vortices(nx, ny, int(seed) % 2 ** 31)[0], (0.0, 0.0), (1.0, 1.0), PERIODIC, PERIODIC,
                W.ALPHA_R_SEEDED, 0.0)
    f = 1.0 + 0.1 * rng.uniform(-1.0, 1.0)
    if data == "rt":  # the perturbation's amplitude varied by 10%
        U, _, _ = W.rayleigh_taylor(nx, ny)
        U[3] += 0.5 * (f * f - 1.0) * U[2] * U[2] / U[0]
        U[2] *= f
        return U, (-0.25, -0.75), (0.25, 0.75), PERIODIC, REFLECTIVE, 50.0, W.RT_GRAVITY
    U, _, _ = W.implosion(nx)
    return U * f, (0.0, 0.0), (1.0, 1.0), REFLECTIVE, REFLECTIVE, 1.0, 0.0


def _batch(case, seed):
    lengths = W.batch_lengths(case["nprob"], case["mix"], case["nmin"], case["nmax"])
    return W.euler_batch(case["nprob"], int(seed) % 2 ** 20, lengths=lengths)


def _adjoint_states(case, seed):
    """(u0, target density, lo, hi, boundary, alpha_R): initial states and the density to match."""
    nprob, n, rng = case["nprob"], case["n"], _rng(seed)
    if case["data"] == "riemann":
        s = int(seed) % 2 ** 20
        U = W.adjoint_batch(nprob, n, s)[0]
        return U, W.adjoint_batch(nprob, n, s, perturbed=True)[0][:, 0], -5.0, 5.0, OUTFLOW, W.ALPHA_R_SEEDED
    U = np.stack([_smooth(n, rng) for _ in range(nprob)])
    x = np.arange(n) / n
    target = U[:, 0] * (1.0 + 0.01 * np.sin(2.0 * np.pi * (x[None] + rng.uniform(0, 1, (nprob, 1)))))
    return U, target, -1.0, 1.0, PERIODIC, 50.0


def _mode(case):
    return B.WT_MODE_STRICT if case["strict"] else B.WT_MODE_FAST


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("rhs", "step"):
        U, lo, hi, bc, aR = _state_1d(case, seed)
        prob = B.problem(FLUX[case["flux"]], bc=bc, alpha_R=aR, mode=_mode(case))
        grid = B.grid_1d(case["n"], lo, hi)
    elif kind in ("rhs2d", "step2d"):
        U, lo, hi, bx, by, aR, g = _state_2d(case, seed)
        prob = B.problem(B.WT_FLUX_EULER2D, bc=bx, bc_y=by, alpha_R=aR, mode=_mode(case), gravity=g)
        grid = B.grid_2d(case["nx"], case["ny"], lo, hi)
    elif kind == "batch":
        b = _batch(case, seed)
        prob = B.problem(B.WT_FLUX_EULER1D, alpha_R=W.ALPHA_R_SEEDED, mode=_mode(case))
        segs = []
        for p in range(case["nprob"]):
            s = B.WtSegment()
            s.offset, s.n, s.lo, s.hi = int(b.offsets[p]), int(b.lengths[p]), float(b.lo[p]), float(b.hi[p])
            s.bc_lo = s.bc_hi = int(b.bc[p])
            segs.append(s)
        total = int(b.u.shape[1])
        ws = B.alloc_workspace(B.workspace_bytes(prob, None, total, len(segs)))
        if case["host"]:
            u0 = torch.from_numpy(b.u)
            u = torch.empty(u0.shape, dtype=torch.float64, pin_memory=True)
            t, status = torch.zeros(len(segs), dtype=torch.float64), torch.zeros(len(segs), dtype=torch.int32)
        else:
            u0 = _dev(b.u)
            u = torch.empty_like(u0)
            t = torch.zeros(len(segs), dtype=torch.float64, device="cuda")
            status = torch.zeros(len(segs), dtype=torch.int32, device="cuda")
        return {"case": case, "prob": prob, "segs": segs, "total": total, "ws": ws, "u0": u0, "u": u, "t": t,
                "status": status}
    else:
        U, target, lo, hi, bc, aR = _adjoint_states(case, seed)
        return {"case": case, "u0": _dev(U).requires_grad_(True), "target": _dev(target), "lo": lo, "hi": hi, "bc": bc,
                "alpha_R": aR}
    ws = B.alloc_workspace(B.workspace_bytes(prob, grid))
    if case.get("host"):
        u0 = torch.from_numpy(np.ascontiguousarray(U))
        u = torch.empty(u0.shape, dtype=torch.float64, pin_memory=True)
    else:
        u0 = _dev(U)
        u = torch.empty_like(u0)
    return {"case": case, "prob": prob, "grid": grid, "ws": ws, "u0": u0, "u": u}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("rhs", "rhs2d"):
        B.weno_theta_rhs(state["prob"], state["grid"], state["u0"], state["u"], state["ws"])
        return state["u"]
    if kind in ("step", "step2d"):
        u = state["u"]
        u.copy_(state["u0"])
        t_final = case.get("t_final") or math.inf
        t, steps = B.weno_theta_step(state["prob"], state["grid"], u, case["cfl"], state["ws"], t_final=t_final,
                                     max_steps=case["steps"])
        return {"u": u, "t": t, "steps": steps}
    if kind == "batch":
        u = state["u"]
        u.copy_(state["u0"])
        B.weno_theta_step_batched(state["prob"], state["segs"], u, state["total"], 0.5, case["steps"], state["ws"],
                                  t_per_problem=state["t"], status_per_problem=state["status"])
        return {"u": u, "t": state["t"], "status": state["status"]}
    u0 = state["u0"]
    dx = (state["hi"] - state["lo"]) / case["n"]
    uT = WenoThetaEuler1D.apply(u0, state["lo"], state["hi"], 0.5, case["steps"], case["every"], state["bc"],
                                state["alpha_R"])
    loss = 0.5 * dx * ((uT[:, 0] - state["target"]) ** 2).sum()
    (grad,) = torch.autograd.grad(loss, u0)
    return {"uT": uT.detach(), "loss": loss.detach(), "grad": grad}


def work(case):
    kind = case["kind"]
    if kind in ("rhs", "step"):
        m = 3 if case["flux"] == "euler" else 1
        steps = 1.0 / 3.0
        if kind == "step":
            # a run to a final time: about t_final max|lambda| / (CFL dx) steps
            steps = case["steps"] if not case["t_final"] else case["t_final"] * case["n"] / (
                case["cfl"] * (2.0 if case["flux"] == "advection" else 10.0 / 4.7))
        return {"bytes": 16.0 * m * case["n"], "flops": FLOPS[case["flux"]] * case["n"] * steps}
    if kind in ("rhs2d", "step2d"):
        cells = case["nx"] * case["ny"]
        return {"bytes": 64.0 * cells, "flops": FLOPS["euler2d"] * cells * case.get("steps", 1.0 / 3.0)}
    if kind == "batch":
        cells = int(W.batch_lengths(case["nprob"], case["mix"], case["nmin"], case["nmax"]).sum())
        return {"bytes": 48.0 * cells, "flops": FLOPS["euler"] * cells * case["steps"]}
    # the forward run, and a reverse sweep of about twice its arithmetic; state in, state and gradient out
    cells = case["nprob"] * case["n"]
    return {"bytes": 80.0 * cells, "flops": 3.0 * FLOPS["euler"] * cells * case["steps"]}


# --------------------------------------------------------------------------------------------
# The method in plain torch binary64 (arXiv 1504.00731: Eqs. (fh0)-(fh3), (be0_cen)-(be3_cen),
# (be_res), (tau_5), (tau_6), (tau_we6), (gam_we6), (om), (fh_nonlinear), (flux_split_lf), (3rd_RK))
# --------------------------------------------------------------------------------------------

GAMMA, EPS = 1.4, 1e-10


def _weno(q, aR):
    fh = [(2 * q[0] - 7 * q[1] + 11 * q[2]) / 6, (-q[1] + 5 * q[2] + 2 * q[3]) / 6, (2 * q[2] + 5 * q[3] - q[4]) / 6,
          (11 * q[3] - 7 * q[4] + 2 * q[5]) / 6]
    b = [13 / 12 * (q[0] - 2 * q[1] + q[2]) ** 2 + (q[0] - 3 * q[1] + 2 * q[2]) ** 2,
         13 / 12 * (q[1] - 2 * q[2] + q[3]) ** 2 + (q[3] - q[2]) ** 2,
         13 / 12 * (q[2] - 2 * q[3] + q[4]) ** 2 + (q[2] - q[3]) ** 2,
         13 / 48 * (3 * q[2] - 7 * q[3] + 5 * q[4] - q[5]) ** 2 + (2 * q[3] - 3 * q[4] + q[5]) ** 2]
    t5 = (13 / 12 * (q[0] - 4 * q[1] + 6 * q[2] - 4 * q[3] + q[4]) ** 2 + (-q[1] + 3 * q[2] - 3 * q[3] + q[4]) ** 2)
    t6 = (13 / 12 * (-q[0] + 5 * q[1] - 10 * q[2] + 10 * q[3] - 5 * q[4] + q[5]) ** 2
          + 0.25 * (q[0] - 3 * q[1] + 2 * q[2] + 2 * q[3] - 3 * q[4] + q[5]) ** 2)
    big = torch.maximum(torch.maximum(b[0], b[1]), torch.maximum(b[2], b[3]))
    small = torch.minimum(torch.minimum(b[0], b[1]), torch.minimum(b[2], b[3]))
    free = (big / (EPS + small) > aR).to(q[0].dtype)
    th = (~(t6 < t5)).to(q[0].dtype)
    tau = torch.where(t6 < t5, t6, t5)
    g = [(1 + th) / 20, 3 * (3 + th) / 20, 3 * (3 - th) / 20, (1 - th) / 20]
    a = [g[k] * (1 + tau / (EPS + free * b[k])) for k in range(4)]
    s = a[0] + a[1] + a[2] + a[3]
    return sum((a[k] / s) * fh[k] for k in range(4))


def _reconstruct(v, w, alpha, aR):
    """F+ + F- of one field from its projected flux v and state w on the six stencil cells."""
    p = [0.5 * (v[k] + alpha * w[k]) for k in range(6)]
    m = [0.5 * (v[k] - alpha * w[k]) for k in range(6)][::-1]
    return _weno(p, aR) + _weno(m, aR)


class _Lines:
    """Index maps of 1D problems packed one after another: ghost-padded cells and interfaces."""

    def __init__(self, lengths, bcs, device):
        n = np.asarray(lengths, dtype=np.int64)
        src, flip, left, cell0 = [], [], [], 0
        pad0 = 0
        for k, bc in zip(n, bcs):
            j = np.arange(-3, k + 3)
            if bc == PERIODIC:
                s, f = j % k, np.ones(k + 6)
            elif bc == OUTFLOW:
                s, f = np.clip(j, 0, k - 1), np.ones(k + 6)
            else:
                s = np.where(j < 0, -1 - j, np.where(j >= k, 2 * k - 1 - j, j))
                f = np.where((j < 0) | (j >= k), -1.0, 1.0)
            src.append(cell0 + s)
            flip.append(f)
            left.append(pad0 + 2 + np.arange(k + 1))
            cell0 += k
            pad0 += k + 6
        iface0 = np.concatenate([[0], np.cumsum(n + 1)[:-1]])
        to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(device)  # noqa: E731
        self.n = to(n)
        self.src, self.flip, self.left = to(np.concatenate(src)), to(np.concatenate(flip)), to(np.concatenate(left))
        self.problem = torch.repeat_interleave(torch.arange(len(n), device=device), self.n)
        self.iproblem = torch.repeat_interleave(torch.arange(len(n), device=device), self.n + 1)
        self.right = to(np.concatenate([o + 1 + np.arange(k) for o, k in zip(iface0, n)]))  # interface right of a cell
        self.nprob, self.one = len(n), len(n) == 1

    def max(self, v):
        """The maximum of a cell array per problem, taken at the first cell that attains it."""
        top = torch.full((self.nprob,), -math.inf, dtype=v.dtype, device=v.device)
        top = top.scatter_reduce(0, self.problem, v.detach(), "amax")
        if not v.requires_grad:
            return top
        at = torch.where(v.detach() == top[self.problem], torch.arange(v.numel(), device=v.device), v.numel())
        first = torch.full((self.nprob,), v.numel(), dtype=torch.int64, device=v.device)
        return v[first.scatter_reduce(0, self.problem, at, "amin")]


def _speeds_1d(flux, U):
    if flux == "advection":
        return [torch.ones_like(U[0])]
    if flux == "burgers":
        return [U[0].abs()]
    u = U[1] / U[0]
    p = (GAMMA - 1) * (U[2] - 0.5 * U[0] * u * u)
    c = torch.sqrt(GAMMA * p / U[0])
    return [torch.nan_to_num((u - c).abs(), nan=0.0), u.abs(), torch.nan_to_num((u + c).abs(), nan=0.0)]


def _rhs_1d(flux, lines, dx, aR, U, alpha):
    """L(U) of packed 1D problems: U a list of components over cells, dx per problem."""
    X = [c[lines.src] for c in U]
    k0 = [lines.left - 2 + k for k in range(6)]
    al = [a[lines.iproblem] for a in alpha]
    if flux != "euler":
        f = X[0] if flux == "advection" else 0.5 * X[0] * X[0]
        h = [_reconstruct([f[k] for k in k0], [X[0][k] for k in k0], al[0], aR)]
    else:
        X[1] = X[1] * lines.flip
        u = X[1] / X[0]
        p = (GAMMA - 1) * (X[2] - 0.5 * X[0] * u * u)
        f = [X[1], p + X[1] * u, (X[2] + p) * u]
        H, s = (X[2] + p) / X[0], torch.sqrt(X[0])
        a, b = lines.left, lines.left + 1
        um, Hm = (s[a] * u[a] + s[b] * u[b]) / (s[a] + s[b]), (s[a] * H[a] + s[b] * H[b]) / (s[a] + s[b])
        c = torch.sqrt((GAMMA - 1) * (Hm - 0.5 * um * um))
        b1 = (GAMMA - 1) / (c * c)
        b2 = 0.5 * um * um * b1
        L = [[0.5 * (b2 + um / c), -0.5 * (b1 * um + 1 / c), 0.5 * b1], [1 - b2, b1 * um, -b1],
             [0.5 * (b2 - um / c), -0.5 * (b1 * um - 1 / c), 0.5 * b1]]
        F = []
        for q in range(3):
            v = [sum(L[q][e] * f[e][k] for e in range(3)) for k in k0]
            w = [sum(L[q][e] * X[e][k] for e in range(3)) for k in k0]
            F.append(_reconstruct(v, w, al[q], aR))
        h = [F[0] + F[1] + F[2], (um - c) * F[0] + um * F[1] + (um + c) * F[2],
             (Hm - um * c) * F[0] + 0.5 * um * um * F[1] + (Hm + um * c) * F[2]]
    d = dx[lines.problem]
    return [-(x[lines.right] - x[lines.right - 1]) / d for x in h]


def _run_1d(flux, lines, dx, aR, U, cfl, steps, t_final):
    t, done = torch.zeros_like(dx), 0
    bounded = math.isfinite(t_final)
    while done < steps and not (bounded and not float(t[0]) < t_final):
        alpha = [lines.max(v) for v in _speeds_1d(flux, U)]
        dt = cfl * dx / torch.maximum(alpha[0], alpha[-1])
        if bounded:
            dt = torch.minimum(dt, t_final - t)
        d = dt[lines.problem]
        L = _rhs_1d(flux, lines, dx, aR, U, alpha)
        U1 = [u + d * x for u, x in zip(U, L)]
        L = _rhs_1d(flux, lines, dx, aR, U1, [lines.max(v) for v in _speeds_1d(flux, U1)])
        U2 = [0.75 * u + 0.25 * (v + d * x) for u, v, x in zip(U, U1, L)]
        L = _rhs_1d(flux, lines, dx, aR, U2, [lines.max(v) for v in _speeds_1d(flux, U2)])
        U = [u / 3.0 + (v + d * x) * (2.0 / 3.0) for u, v, x in zip(U, U2, L)]
        t = t + dt.detach()
        done += 1
    return U, t, done


def _speeds_2d(U):
    u, v = U[1] / U[0], U[2] / U[0]
    p = (GAMMA - 1) * (U[3] - 0.5 * U[0] * (u * u + v * v))
    return u, v, torch.sqrt(GAMMA * p / U[0])


def _sweep(U, bc, h, aR):
    """-(flux difference) / h along the last axis; U = (rho, normal momentum, tangential, E)."""
    n = U[0].shape[-1]
    j = torch.arange(-3, n + 3, device=U[0].device)
    if bc == PERIODIC:
        s = j % n
    elif bc == OUTFLOW:
        s = j.clamp(0, n - 1)
    else:
        s = torch.where(j < 0, -1 - j, torch.where(j >= n, 2 * n - 1 - j, j))
    u, v, c = _speeds_2d(U)
    alpha = [(u - c).abs().max(), u.abs().max(), u.abs().max(), (u + c).abs().max()]
    X = [x[..., s] for x in U]
    if bc == REFLECTIVE:
        X[1] = X[1] * torch.where((j < 0) | (j >= n), -1.0, 1.0)
    u, v = X[1] / X[0], X[2] / X[0]
    p = (GAMMA - 1) * (X[3] - 0.5 * X[0] * (u * u + v * v))
    f = [X[1], p + X[1] * u, X[1] * v, (X[3] + p) * u]
    H, r = (X[3] + p) / X[0], torch.sqrt(X[0])
    A, Bc = slice(2, n + 3), slice(3, n + 4)
    mean = lambda y: (r[..., A] * y[..., A] + r[..., Bc] * y[..., Bc]) / (r[..., A] + r[..., Bc])  # noqa: E731
    um, vm, Hm = mean(u), mean(v), mean(H)
    k2 = um * um + vm * vm
    c = torch.sqrt((GAMMA - 1) * (Hm - 0.5 * k2))
    b1 = (GAMMA - 1) / (c * c)
    b2 = 0.5 * k2 * b1
    zero, one = torch.zeros_like(c), torch.ones_like(c)
    L = [[0.5 * (b2 + um / c), -0.5 * (b1 * um + 1 / c), -0.5 * b1 * vm, 0.5 * b1], [1 - b2, b1 * um, b1 * vm, -b1],
         [-vm, zero, one, zero], [0.5 * (b2 - um / c), -0.5 * (b1 * um - 1 / c), -0.5 * b1 * vm, 0.5 * b1]]
    F = []
    for q in range(4):
        a = [sum(L[q][e] * f[e][..., k:k + n + 1] for e in range(4)) for k in range(6)]
        b = [sum(L[q][e] * X[e][..., k:k + n + 1] for e in range(4)) for k in range(6)]
        F.append(_reconstruct(a, b, alpha[q], aR))
    out = [F[0] + F[1] + F[3], (um - c) * F[0] + um * F[1] + (um + c) * F[3], vm * (F[0] + F[1] + F[3]) + F[2],
           (Hm - um * c) * F[0] + 0.5 * k2 * F[1] + vm * F[2] + (Hm + um * c) * F[3]]
    return [-(x[..., 1:] - x[..., :-1]) / h for x in out]


def _rhs_2d(U, dx, dy, bx, by, aR, g):
    Lx = _sweep(U, bx, dx, aR)
    T = [U[0].T, U[2].T, U[1].T, U[3].T]
    Ly = [x.T for x in _sweep(T, by, dy, aR)]
    L = [Lx[0] + Ly[0], Lx[1] + Ly[2], Lx[2] + Ly[1], Lx[3] + Ly[3]]
    return [L[0], L[1], L[2] - g * U[0], L[3] - g * U[2]]


def exact(case, seed):
    kind = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    to = lambda a: [x for x in torch.from_numpy(np.ascontiguousarray(a)).to(dev)]  # noqa: E731
    if kind in ("rhs", "step"):
        U, lo, hi, bc, aR = _state_1d(case, seed)
        lines = _Lines([case["n"]], [bc], dev)
        dx = torch.tensor([(hi - lo) / case["n"]], dtype=torch.float64, device=dev)
        U, flux = to(U), case["flux"]
        if kind == "rhs":
            return torch.stack(_rhs_1d(flux, lines, dx, aR, U, [lines.max(v) for v in _speeds_1d(flux, U)]))
        U, t, steps = _run_1d(flux, lines, dx, aR, U, case["cfl"], case["steps"], case["t_final"] or math.inf)
        return {"u": torch.stack(U), "t": float(t[0]), "steps": steps}
    if kind == "batch":
        b = _batch(case, seed)
        lines = _Lines(b.lengths, b.bc, dev)
        dx = torch.from_numpy(b.dx).to(dev)
        U, t, _ = _run_1d("euler", lines, dx, W.ALPHA_R_SEEDED, to(b.u), 0.5, case["steps"], math.inf)
        return {"u": torch.stack(U), "t": t, "status": None}
    if kind in ("rhs2d", "step2d"):
        U, lo, hi, bx, by, aR, g = _state_2d(case, seed)
        dx, dy = (hi[0] - lo[0]) / case["nx"], (hi[1] - lo[1]) / case["ny"]
        U = to(U)
        if kind == "rhs2d":
            return torch.stack(_rhs_2d(U, dx, dy, bx, by, aR, g))
        t = 0.0
        for _ in range(case["steps"]):
            u, v, c = _speeds_2d(U)
            dt = case["cfl"] / float(((u.abs() + c) / dx + (v.abs() + c) / dy).max())
            L = _rhs_2d(U, dx, dy, bx, by, aR, g)
            U1 = [a + dt * x for a, x in zip(U, L)]
            L = _rhs_2d(U1, dx, dy, bx, by, aR, g)
            U2 = [0.75 * a + 0.25 * (b + dt * x) for a, b, x in zip(U, U1, L)]
            L = _rhs_2d(U2, dx, dy, bx, by, aR, g)
            U = [a / 3.0 + (b + dt * x) * (2.0 / 3.0) for a, b, x in zip(U, U2, L)]
            t += dt
        return {"u": torch.stack(U), "t": t, "steps": case["steps"]}
    # the adjoint: reverse mode through the plain forward.  On the Riemann data the gradient has no one
    # value: its acoustic fields carry rounding noise alone, on which theta's branch is taken
    U, target, lo, hi, bc, aR = _adjoint_states(case, seed)
    smooth = case["data"] == "smooth"
    nprob, n = case["nprob"], case["n"]
    lines = _Lines([n] * nprob, [bc] * nprob, dev)
    dx = torch.full((nprob,), (hi - lo) / n, dtype=torch.float64, device=dev)
    u0 = torch.from_numpy(np.ascontiguousarray(U)).to(dev).requires_grad_(smooth)
    V, _, _ = _run_1d("euler", lines, dx, aR, [u0[:, e].reshape(-1) for e in range(3)], 0.5, case["steps"], math.inf)
    uT = torch.stack([v.reshape(nprob, n) for v in V], dim=1)
    loss = 0.5 * (hi - lo) / n * ((uT[:, 0] - torch.from_numpy(np.ascontiguousarray(target)).to(dev)) ** 2).sum()
    grad = torch.autograd.grad(loss, u0)[0] if smooth else None
    return {"uT": uT.detach(), "loss": loss.detach(), "grad": grad}
