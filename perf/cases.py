"""Timed workloads of the WENO-ZN solver, each run through the package's public entry points.

A case is a dict of plain values.  `prepare` builds what a user's program holds before the
call (initial state, problem, workspace), `run` makes one pass through the public API and
returns its whole outputs, `work` gives the bytes and flops the path cannot do without and
`exact` evaluates the same pass in plain 64-bit torch, in the paper's order, without the
package's kernels.

Kinds:
  advection   linear advection, chained SSP-RK3 steps of the convergence study's fixed step
  euler1d     1D Euler (Shu-Osher family), chained CFL steps
  euler2d     2D Euler, four-quadrant Riemann data with smooth waves on top (a developed flow
              has structure in every cell, the bare initial data almost none), chained CFL
              steps; any weight function, splitting and boundary condition
  batch       ragged batch of independent 1D Euler problems, set up and stepped
  reconstruct the reconstruction entry point, both sides of one line
  rollout     fixed-step rollout under autograd: forward, loss and gradient of the initial state
"""
import math

import numpy as np
import torch

from paper_2004_07954_gb300 import inputs, rollout, wenozn as W

GAMMA, EPS, A_ZN, CFL = 1.4, 1e-40, 10.0, 0.5


# ------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the convergence study's grids hold 40 to 320 cells: launches and latency are all there is
        {"name": "advection_160", "kind": "advection", "n": 160, "steps": 50},
        # the smallest 1D Euler grid in use (shock-tube resolution)
        {"name": "euler1d_200", "kind": "euler1d", "n": 200, "steps": 20},
        # the largest 1D Euler grid
        {"name": "euler1d_1048576", "kind": "euler1d", "n": 1048576, "steps": 2},
        # a 2D grid used for quick looks and tests: a few blocks per SM
        {"name": "euler2d_256", "kind": "euler2d", "nx": 256, "ny": 256, "steps": 5, "split": 0, "weights": 0, "bc": 1},
        # the two grids of the 2D configuration
        {"name": "euler2d_1024", "kind": "euler2d", "nx": 1024, "ny": 1024, "steps": 2, "split": 0, "weights": 0, "bc": 1},
        {"name": "euler2d_4096", "kind": "euler2d", "nx": 4096, "ny": 4096, "steps": 1, "split": 0, "weights": 0, "bc": 1},
        # the paper's own 2D splitting (Steger-Warming), a ragged grid between walls
        {"name": "euler2d_sw_walls", "kind": "euler2d", "nx": 1501, "ny": 999, "steps": 1, "split": 3, "weights": 0, "bc": 2},
        # a comparison run: WENO-Z weights with local Lax-Friedrichs on a periodic box
        {"name": "euler2d_llf_wenoz", "kind": "euler2d", "nx": 640, "ny": 777, "steps": 1, "split": 2, "weights": 1, "bc": 0},
        # a parameter study: many 1D problems of uneven size advanced together
        {"name": "batch_512", "kind": "batch", "instances": 512, "n_min": 128, "n_max": 16384, "steps": 4},
        # the reconstruction by itself, as post-processing or another solver calls it
        {"name": "reconstruct_16m", "kind": "reconstruct", "n": 16777221},
        # gradient of an initial state through a checkpointed rollout
        {"name": "rollout_8192", "kind": "rollout", "n": 8192, "steps": 40, "every": 20},
        # the same on a long line, every step's stages kept
        {"name": "rollout_131071", "kind": "rollout", "n": 131071, "steps": 3, "every": 1},
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["advection", "euler1d", "euler2d", "euler2d", "euler2d", "batch", "reconstruct", "rollout"])
    if kind == "advection":
        return {"kind": kind, "n": _log_size(rng, 40, 4000), "steps": rng.randint(10, 60)}
    if kind == "euler1d":
        n = _log_size(rng, 200, 1048576)
        return {"kind": kind, "n": n, "steps": rng.randint(1, 20) if n < 50000 else rng.randint(1, 2)}
    if kind == "euler2d":
        nx, ny = _log_size(rng, 64, 2600), _log_size(rng, 64, 2600)
        split = rng.choice([0, 0, 0, 1, 2, 3])
        return {"kind": kind, "nx": nx, "ny": ny, "steps": rng.randint(1, 4) if nx * ny < 400000 else 1, "split": split,
                "weights": rng.choice([0, 0, 0, 1, 3]), "bc": rng.choice([0, 1, 1, 2])}
    if kind == "batch":
        return {"kind": kind, "instances": rng.randint(3, 500), "n_min": 128, "n_max": _log_size(rng, 400, 16384),
                "steps": rng.randint(2, 5)}
    if kind == "reconstruct":
        return {"kind": kind, "n": _log_size(rng, 1000, 16777216)}
    n = _log_size(rng, 200, 131072)
    steps = rng.randint(4, 30) if n < 20000 else rng.randint(1, 3)
    return {"kind": kind, "n": n, "steps": steps, "every": rng.choice([1, 5, 10])}


# ----------------------------------------------------------------------------- the inputs
def _advection_state(case, seed):
    """A seeded mix of the study's two profiles: u0 = sin(pi x + a) and its critical-point form."""
    g = np.random.default_rng(seed)
    x, dx = inputs.advection_grid(case["n"])
    a, w = g.uniform(0.0, 2.0 * math.pi), g.uniform(0.0, 1.0)
    y = np.pi * x + a
    u = w * np.sin(y) + (1.0 - w) * np.sin(y - np.sin(y) / np.pi)
    return u.reshape(1, 1, -1).copy(), dx


def _flow_2d(case, seed):
    """Four-quadrant Riemann data (constant states split at the centre) with a few percent of
    smooth waves in every variable; periodic boxes take the waves alone."""
    nx, ny = case["nx"], case["ny"]
    q = torch.from_numpy(inputs.euler2d_params(seed)).cuda()
    g = np.random.default_rng(seed + 1)
    x = (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) / nx
    y = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny

    def waves(amp):
        w = torch.zeros((ny, nx), dtype=torch.float64, device="cuda")
        for _ in range(3):
            kx, ky = g.integers(1, 7, size=2)
            px, py = g.uniform(0.0, 2.0 * math.pi, size=2)
            w += amp / 3.0 * torch.sin(2.0 * math.pi * int(ky) * y + py)[:, None] * torch.sin(2.0 * math.pi * int(kx) * x + px)
        return w

    quad = (x > 0.5).long()[None, :] * 2 + (y > 0.5).long()[:, None]
    if case["bc"] == 0:
        quad = torch.zeros_like(quad)
    rho, u, v, p = (q[:, k][quad] for k in range(4))
    rho, p = rho * (1.0 + waves(0.1)), p * (1.0 + waves(0.1))
    u, v = u + waves(0.1), v + waves(0.1)
    return torch.stack([rho, rho * u, rho * v, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)]).contiguous()


def _line(case, seed):
    """Smooth waves with jumps, padded by three ghost cells on either side."""
    n = case["n"]
    g = np.random.default_rng(seed)
    x = torch.arange(n + 6, dtype=torch.float64, device="cuda") / n
    f = torch.zeros_like(x)
    for _ in range(4):
        f += g.uniform(0.2, 1.0) * torch.sin(2.0 * math.pi * float(g.uniform(1.0, 40.0)) * x + float(g.uniform(0.0, 6.28)))
    for at in g.uniform(0.0, 1.0, size=64):
        f += float(g.normal()) * (x > at)
    return f


def _batch(case, seed):
    """Sizes log-uniform in [n_min, n_max], fixed by the case; every instance's data by the seed."""
    g = np.random.default_rng(case["instances"])
    sizes = np.round(np.exp(g.uniform(math.log(case["n_min"]), math.log(case["n_max"]), case["instances"]))).astype(np.int64)
    off = np.concatenate([[0], np.cumsum(sizes)])
    U0 = np.concatenate([inputs.euler1d_ic(int(n), seed * 100003 + b)[:, 0] for b, n in enumerate(sizes)], 1)
    return sizes, off, U0


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "case": case}
    if kind == "advection":
        U0, dx = _advection_state(case, seed)
        st["U0"] = _cuda(U0)
        st["dt"] = 0.1 * dx ** (5.0 / 3.0)
        st["solver"] = W.Solver(W.wenozn_problem_init(W.WENOZN_ADVECTION_1D, case["n"], dx=dx, bc_x=W.WENOZN_BC_PERIODIC))
    elif kind == "euler1d":
        _, dx = inputs.euler1d_grid(case["n"])
        st["U0"] = _cuda(inputs.euler1d_ic(case["n"], seed))
        st["dt"] = 0.0
        st["solver"] = W.Solver(W.wenozn_problem_init(W.WENOZN_EULER_1D, case["n"], dx=dx))
    elif kind == "euler2d":
        st["U0"] = _flow_2d(case, seed)
        st["dt"] = 0.0
        st["solver"] = W.Solver(W.wenozn_problem_init(
            W.WENOZN_EULER_2D, case["nx"], case["ny"], 1.0 / case["nx"], 1.0 / case["ny"], bc_x=case["bc"],
            bc_y=case["bc"], split=case["split"], weights=case["weights"]))
    elif kind == "batch":
        sizes, off, U0 = _batch(case, seed)
        st["U0"] = _cuda(U0)
        st["batch"] = W.Batch(off, 10.0 / sizes, st["U0"])
    elif kind == "reconstruct":
        st["f"] = _line(case, seed)
        st["fhat"] = [torch.empty(case["n"] + 1, dtype=torch.float64, device="cuda") for _ in range(2)]
    else:
        n = case["n"]
        _, dx = inputs.euler1d_grid(n)
        st["p"] = W.wenozn_problem_init(W.WENOZN_EULER_1D, n, dx=dx, bc_x=W.WENOZN_BC_PERIODIC)
        st["ws"] = W.vjp_workspace(st["p"])
        st["U0"] = _cuda(inputs.adjoint_ic(n, seed)).requires_grad_(True)
        st["target"] = _cuda(inputs.adjoint_ic(n, seed + 1))[0]
        st["dt"] = rollout.cfl_step(st["p"], st["U0"].detach(), st["ws"])
    if kind in ("advection", "euler1d", "euler2d", "batch"):
        st["U"] = torch.empty_like(st["U0"])
    return st


def run(state):
    kind, case = state["kind"], state["case"]
    if kind in ("advection", "euler1d", "euler2d"):
        U = state["U"]
        U.copy_(state["U0"])                       # every pass starts from the initial state
        state["solver"].steps(U, case["steps"], state["dt"])
        return U
    if kind == "batch":
        U, b = state["U"], state["batch"]
        U.copy_(state["U0"])
        b.init(U)
        for _ in range(case["steps"]):
            b.step(U)
        return U
    if kind == "reconstruct":
        W.wenozn_reconstruct(state["f"], state["fhat"][0], 1)
        W.wenozn_reconstruct(state["f"], state["fhat"][1], -1)
        return state["fhat"]
    UT = rollout.rollout(state["U0"], state["p"], state["dt"], case["steps"], case["every"], state["ws"])
    loss = 0.5 * (UT[0] - state["target"]).square().sum()
    (grad,) = torch.autograd.grad(loss, state["U0"])
    return {"state": UT.detach(), "grad": grad}


# ------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Bytes: each input and output once.  Flops: one per add, sub, mul, div and sqrt of the
    scheme as written (tests/test_opcount*.py), per cell and RK3 step."""
    kind = case["kind"]
    if kind == "advection":
        return {"bytes": 16.0 * case["n"], "flops": 552.0 * case["n"] * case["steps"]}
    if kind == "euler1d":
        return {"bytes": 48.0 * case["n"], "flops": 2448.0 * case["n"] * case["steps"]}
    if kind == "euler2d":
        per = {0: 6984.0, 1: 7998.0, 2: 7968.0, 3: 7644.0}[case["split"]]
        if case["weights"]:
            per -= 3 * 2 * 8 * 12.0          # C and tau8 of each reconstruction are not part of these weights
        return {"bytes": 64.0 * case["nx"] * case["ny"], "flops": per * case["nx"] * case["ny"] * case["steps"]}
    if kind == "batch":
        mean = (case["n_max"] - case["n_min"]) / math.log(case["n_max"] / case["n_min"])
        cells = mean * case["instances"]
        return {"bytes": 48.0 * cells, "flops": 2448.0 * cells * case["steps"]}
    if kind == "reconstruct":
        return {"bytes": 24.0 * case["n"], "flops": 2 * 85.0 * case["n"]}
    # forward, and a reverse sweep of about three times the forward's operations
    return {"bytes": 80.0 * case["n"], "flops": 4.0 * 2448.0 * case["n"] * case["steps"]}


# ---------------------------------------------------------------- the same in plain 64 bits
def _zn(a, b, c, d, e, weights):
    is0 = 13.0 / 12.0 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2
    is1 = 13.0 / 12.0 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2
    is2 = 13.0 / 12.0 * (c - 2 * d + e) ** 2 + 0.25 * ((e - 4 * d) + 3 * c) ** 2
    q = ((2 * a - 7 * b + 11 * c) / 6, (-b + 5 * c + 2 * d) / 6, (2 * c + 5 * d - e) / 6)
    tau5 = (is0 - is2).abs()
    if weights == 0:
        # C and tau8 / (IS + eps) both times (tau5 + eps)^2 (the weights are normalised below), which
        # keeps torch's derivative of C accurate where tau5 nearly vanishes
        tau8 = ((a + e) - 4 * (b + d) + 6 * c) ** 2 * (tau5 + EPS) ** 2
        C = A_ZN * (2.0 * torch.minimum(is0, is2) + EPS) ** 2
        w = [ck * (C + tau8 / (s + EPS)) for ck, s in zip((0.1, 0.6, 0.3), (is0, is1, is2))]
    elif weights == 1:
        w = [ck * (1.0 + tau5 / (s + EPS)) for ck, s in zip((0.1, 0.6, 0.3), (is0, is1, is2))]
    else:
        w = [ck / (s + EPS) ** 2 for ck, s in zip((0.1, 0.6, 0.3), (is0, is1, is2))]
    return (w[0] * q[0] + w[1] * q[1] + w[2] * q[2]) / (w[0] + w[1] + w[2])


def _prims(U):
    """rho, normal velocity, tangential velocity (or None), pressure, sound speed."""
    rho, u = U[0], U[1] / U[0]
    v = U[2] / rho if len(U) == 4 else None
    kin = 0.5 * rho * (u * u if v is None else u * u + v * v)
    p = (GAMMA - 1.0) * (U[-1] - kin)
    return rho, u, v, p, torch.sqrt(GAMMA * p / rho)


def _split(U, split, alpha):
    """The split fluxes (F+, F-) of cells, alpha broadcastable to a component."""
    rho, u, v, p, c = _prims(U)
    if split == 3:
        out = []
        vv = 0.0 if v is None else v * v
        for s in (1.0, -1.0):
            l1, l2, l3 = (0.5 * (x + s * x.abs()) for x in (u - c, u, u + c))
            k, m = rho / (2 * GAMMA), 2 * (GAMMA - 1) * l2 + l1 + l3
            E = (GAMMA - 1) * l2 * (u * u + vv) + 0.5 * l1 * ((u - c) ** 2 + vv) + 0.5 * l3 * ((u + c) ** 2 + vv) \
                + (3 - GAMMA) * (l1 + l3) * c * c / (2 * (GAMMA - 1))
            mom = 2 * (GAMMA - 1) * l2 * u + l1 * (u - c) + l3 * (u + c)
            out.append([k * m, k * mom] + ([] if v is None else [k * m * v]) + [k * E])
        return out
    F = [U[1], U[1] * u + p] + ([] if v is None else [U[2] * u]) + [u * (U[-1] + p)]
    return [[0.5 * (f + s * alpha * w) for f, w in zip(F, U)] for s in (1.0, -1.0)]


def _interface_flux(S, split, weights, alpha):
    """F^ from the six stencil cells S[k] (nv, ...), k = 0..5.  alpha: the LF speed (global), the
    per-field speeds, or None (local LF, Steger-Warming)."""
    nv = len(S[0])
    rl, ul, vl, pl, _ = _prims(S[2])
    rr, ur, vr, pr, _ = _prims(S[3])
    a, b = torch.sqrt(rl), torch.sqrt(rr)
    u = (a * ul + b * ur) / (a + b)
    v = (a * vl + b * vr) / (a + b) if nv == 4 else torch.zeros_like(u)
    H = (a * (S[2][-1] + pl) / rl + b * (S[3][-1] + pr) / rr) / (a + b)
    q2 = u * u + v * v
    c = torch.sqrt((GAMMA - 1) * (H - 0.5 * q2))
    b1 = (GAMMA - 1) / (c * c)
    b2 = 0.5 * q2 * b1
    one, zero = torch.ones_like(u), torch.zeros_like(u)

    def cut(r):
        return r if nv == 4 else [r[0], r[1], r[3]]

    L = [cut([(b2 + u / c) / 2, -(b1 * u + 1 / c) / 2, -b1 * v / 2, b1 / 2]), cut([1 - b2, b1 * u, b1 * v, -b1])]
    R = [cut([one, u - c, v, H - u * c]), cut([one, u, v, 0.5 * q2])]
    if nv == 4:
        L.append([-v, zero, one, zero])
        R.append([zero, zero, one, v])
    L.append(cut([(b2 - u / c) / 2, -(b1 * u - 1 / c) / 2, -b1 * v / 2, b1 / 2]))
    R.append(cut([one, u + c, v, H + u * c]))
    if split == 2:
        sp = torch.stack([x[1].abs() + x[4] for x in map(_prims, S)])
        alpha = sp.amax(0)
    fields = [alpha[0]] + [alpha[1]] * (nv - 2) + [alpha[2]] if split == 1 else [alpha] * nv
    out = [0.0] * nv
    parts = None
    for k in range(nv):
        if parts is None or split == 1:
            parts = [_split(s, split, fields[k]) for s in S]
        gp = [sum(l * h for l, h in zip(L[k], parts[i][0])) for i in range(0, 5)]
        gm = [sum(l * h for l, h in zip(L[k], parts[i][1])) for i in range(5, 0, -1)]
        g = _zn(*gp, weights) + _zn(*gm, weights)
        out = [o + r * g for o, r in zip(out, R[k])]
    return torch.stack(out)


def _padded(U, bc):
    """Three ghost cells on either side of the last axis (component 1 is the normal momentum)."""
    n = U.shape[-1]
    g = torch.arange(-3, n + 3, device=U.device)
    if bc == 0:
        return U[..., g % n]
    if bc == 1:
        return U[..., g.clamp(0, n - 1)]
    P = U[..., torch.where(g < 0, -1 - g, torch.where(g >= n, 2 * n - 1 - g, g))].clone()
    P[1, ..., :3] *= -1.0
    P[1, ..., -3:] *= -1.0
    return P


def _sweep(U, bc, split, weights):
    """-dF along the last axis (not divided by dx), a few rows at a time."""
    nv, n = U.shape[0], U.shape[-1]
    _, u, _, _, c = _prims(U)
    alpha = None
    if split == 0:
        alpha = (u.abs() + c).reshape(-1).max(0).values
    elif split == 1:
        alpha = [(u - c).abs().max(), u.abs().max(), (u + c).abs().max()]
    rows = U.reshape(nv, -1, n)
    step = max(1, (1 << 20) // n)
    out = []
    for r in range(0, rows.shape[1], step):
        P = _padded(rows[:, r:r + step], bc)
        F = _interface_flux([P[..., k:k + n + 1] for k in range(6)], split, weights, alpha)
        out.append(F[..., :-1] - F[..., 1:])
    return torch.cat(out, 1).reshape(U.shape)


def _rhs(U, case, dx, dy):
    bc, split, weights = case.get("bc", 1), case.get("split", 0), case.get("weights", 0)
    L = _sweep(U, bc, split, weights) / dx
    if len(U) == 4:
        V = U[[0, 2, 1, 3]].transpose(1, 2).contiguous()
        L = L + _sweep(V, bc, split, weights)[[0, 2, 1, 3]].transpose(1, 2) / dy
    return L


def _rk3(U, rhs, dt):
    U1 = U + dt * rhs(U)
    U2 = 0.75 * U + 0.25 * (U1 + dt * rhs(U1))
    return U / 3.0 + 2.0 / 3.0 * (U2 + dt * rhs(U2))


def _speed(U, n):
    _, u, v, _, c = _prims(U)
    return ((u if n == 1 else v).abs() + c).max()


def exact(case, seed):
    kind = case["kind"]
    if kind == "reconstruct":
        f, n = _line(case, seed), case["n"]
        s = [f[k:k + n + 1] for k in range(6)]
        return [_zn(*s[:5], 0), _zn(*s[:0:-1], 0)]
    if kind == "advection":
        U0, dx = _advection_state(case, seed)
        U, dt = _cuda(U0), 0.1 * dx ** (5.0 / 3.0)

        def rhs(w):
            P, n = _padded(w, 0), w.shape[-1]
            F = _zn(*[P[..., k:k + n + 1] for k in range(5)], 0)      # speed 1: the minus part vanishes
            return (F[..., :-1] - F[..., 1:]) / dx

        for _ in range(case["steps"]):
            U = _rk3(U, rhs, dt)
        return U
    if kind == "euler2d":
        U = _flow_2d(case, seed)
        dx, dy = 1.0 / case["nx"], 1.0 / case["ny"]
        for _ in range(case["steps"]):
            tx, ty = dx / _speed(U, 1), dy / _speed(U, 2)
            U = _rk3(U, lambda w: _rhs(w, case, dx, dy), CFL * tx * ty / (tx + ty))
        return U
    if kind == "euler1d":
        _, dx = inputs.euler1d_grid(case["n"])
        U = _cuda(inputs.euler1d_ic(case["n"], seed))
        for _ in range(case["steps"]):
            U = _rk3(U, lambda w: _rhs(w, case, dx, 1.0), CFL * dx / _speed(U, 1))
        return U
    if kind == "batch":
        sizes, off, U0 = _batch(case, seed)
        U, dx, B = _cuda(U0), _cuda(10.0 / sizes), len(sizes)
        inst = torch.repeat_interleave(torch.arange(B, device="cuda"), _cuda(sizes))
        iface = torch.repeat_interleave(torch.arange(B, device="cuda"), _cuda(sizes) + 1)
        lo, hi = _cuda(off[:-1])[iface], _cuda(off[1:])[iface] - 1
        j = torch.arange(len(iface), device="cuda") - iface            # global cell right of the interface
        left = torch.arange(U.shape[1], device="cuda") + inst           # a cell's left interface

        def speeds(w):
            _, u, _, _, c = _prims(w)
            return torch.zeros(B, dtype=torch.float64, device="cuda").scatter_reduce(0, inst, u.abs() + c, "amax")

        def rhs(w):
            S = [w[:, torch.minimum(torch.maximum(j + k - 3, lo), hi)] for k in range(6)]
            F = _interface_flux(S, 0, 0, speeds(w)[iface])
            return (F[:, left] - F[:, left + 1]) / dx[inst]

        for _ in range(case["steps"]):
            U = _rk3(U, rhs, (CFL * dx / speeds(U))[inst])
        return U
    # rollout: the gradient by torch's own autograd through the plain scheme
    n = case["n"]
    _, dx = inputs.euler1d_grid(n)
    U0 = _cuda(inputs.adjoint_ic(n, seed)).requires_grad_(True)
    target = _cuda(inputs.adjoint_ic(n, seed + 1))[0]
    dt = (CFL * dx / _speed(U0.detach(), 1)).item()
    U = U0
    for _ in range(case["steps"]):
        U = _rk3(U, lambda w: _rhs(w, {"bc": 0}, dx, 1.0), dt)
    (grad,) = torch.autograd.grad(0.5 * (U[0] - target).square().sum(), U0)
    return {"state": U.detach(), "grad": grad}
