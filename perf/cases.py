"""What a user of this library has it compute, as cases that can be timed and checked.

Each case is one pass through the public entry points (`enomr.Solver`, `enomr.Batch`,
`enomr.rollout`): a few time steps of a 1D or 2D problem, a batched step, or a rollout with
its gradient.  `exact` restates the scheme in plain torch float64 without the library.
"""
from __future__ import annotations

import functools
import math
from fractions import Fraction

import numpy as np
import torch

from paper_2311_15504_gb300 import enomr, workloads

GAMMA = 1.4


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest run: the paper's scalar advection test, ten steps of a 200-cell line
        {"name": "advection_200", "kind": "advection", "n": 200, "order": 5, "steps": 10},
        # a long scalar line of odd length, smooth with a square pulse on it
        {"name": "advection_1m", "kind": "advection", "n": 1048573, "order": 9, "steps": 2},
        # a large scalar line of a nonlinear law, high order
        {"name": "burgers_4m", "kind": "burgers", "n": 4194304, "order": 13, "steps": 1},
        # shock / entropy-wave interaction at the sizes it is usually run at
        {"name": "shock_entropy_400", "kind": "euler1d", "n": 400, "order": 9, "steps": 4},
        {"name": "shock_entropy_6400", "kind": "euler1d", "n": 6400, "order": 17, "steps": 2},
        # thousands of independent Riemann problems of uneven size (parameter studies)
        {"name": "batch_4096", "kind": "batch", "nprob": 4096, "order": 9, "steps": 1},
        # a Riemann configuration on a grid of the size 2D papers show, at its start
        {"name": "riemann_801", "kind": "riemann", "nx": 801, "ny": 801, "order": 5,
         "developed": 0, "steps": 1},
        # the same problem some way into its run: the highest order, and the flagship grid
        {"name": "riemann_2048", "kind": "riemann", "nx": 2048, "ny": 2048, "order": 17,
         "developed": 24, "steps": 1},
        {"name": "riemann_4096", "kind": "riemann", "nx": 4096, "ny": 4096, "order": 9,
         "developed": 24, "steps": 1},
        # smooth flow: every cell differs from its neighbours
        {"name": "vortex_1024", "kind": "vortex", "nx": 1024, "ny": 1024, "order": 9, "steps": 1},
        # optimisation of an initial state: rollout and gradient of a density mismatch
        {"name": "vortex_grad_512", "kind": "grad", "nx": 512, "ny": 512, "order": 9, "steps": 2},
        # boundary sides of all kinds with a moving inflow: the double Mach reflection
        {"name": "double_mach_1200", "kind": "mach", "nx": 1200, "ny": 300, "order": 9, "steps": 1},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["advection", "burgers", "euler1d", "batch", "riemann", "riemann", "vortex",
                       "grad", "mach"])
    order = rng.choice([5, 7, 9, 11, 13, 15, 17])
    if kind in ("advection", "burgers"):
        n = _logint(rng, 128, 4000000)
        return {"kind": kind, "n": n, "order": order, "steps": 10 if n < 10000 else 1}
    if kind == "euler1d":
        n = _logint(rng, 200, 100000)
        return {"kind": kind, "n": n, "order": order, "steps": 4 if n < 10000 else 1}
    if kind == "batch":
        return {"kind": kind, "nprob": _logint(rng, 64, 2500), "order": order, "steps": 1}
    if kind == "riemann":
        return {"kind": kind, "nx": _logint(rng, 200, 2600), "ny": _logint(rng, 200, 2600),
                "order": order, "developed": rng.choice([0, 6, 24]), "steps": 1}
    if kind == "vortex":
        return {"kind": kind, "nx": _logint(rng, 64, 1024), "ny": _logint(rng, 64, 1024),
                "order": order, "steps": 1}
    if kind == "grad":
        return {"kind": kind, "nx": _logint(rng, 48, 512), "ny": _logint(rng, 48, 512),
                "order": rng.choice([5, 7, 9]), "steps": 2}
    n = _logint(rng, 75, 320)
    return {"kind": "mach", "nx": 4 * n, "ny": n, "order": rng.choice([5, 7, 9, 11]), "steps": 1}


CFL = {"mach": 0.1}  # others 0.5


def _cfl(case):
    return CFL.get(case["kind"], 0.5)


# ---------------------------------------------------------------------------
# inputs, on the GPU
# ---------------------------------------------------------------------------
def _dev():
    return torch.device("cuda")


def _riemann_state(case, seed):
    """Four constant states (seeded) meeting at (0.8, 0.8); 'developed' steps of a plain
    first-order scheme turn its jumps into the narrow fans, shocks and contacts of a run."""
    nx, ny = case["nx"], case["ny"]
    dx, dy = 1.0 / nx, 1.0 / ny
    x = (torch.arange(nx, device=_dev(), dtype=torch.float64) + 0.5) * dx
    y = (torch.arange(ny, device=_dev(), dtype=torch.float64) + 0.5) * dy
    st = torch.from_numpy(workloads.quadrant_states(seed)).to(_dev())
    right, up = x > 0.8, y > 0.8
    q = torch.where(up[:, None], torch.where(right, 0, 1)[None], torch.where(right, 3, 2)[None])
    U = _conserved(*(st[:, k][q] for k in range(4)))
    for _ in range(case["developed"]):
        s = [(U[1 + a] / U[0]).abs() + _sound(U) for a in (0, 1)]
        dt = 0.4 / float((s[0] / dx + s[1] / dy).max())
        D = torch.zeros_like(U)
        for axis, h in ((0, dx), (1, dy)):
            dim = 2 - axis
            n = U.shape[dim]
            E = torch.cat([U.narrow(dim, 0, 1), U, U.narrow(dim, n - 1, 1)], dim)
            F = _flux(E, axis)
            lam = float(s[axis].max())
            f = 0.5 * (F.narrow(dim, 0, n + 1) + F.narrow(dim, 1, n + 1)) - 0.5 * lam * (
                E.narrow(dim, 1, n + 1) - E.narrow(dim, 0, n + 1))
            D -= (f.narrow(dim, 1, n) - f.narrow(dim, 0, n)) / h
        U = U + dt * D
    return U.contiguous(), dx, dy


def _vortex_state(case, seed):
    """Isentropic vortex, periodic on [0, 10]^2, its centre off the grid lines (seeded)."""
    rng = np.random.default_rng(seed)
    cx, cy = 5.0 + rng.uniform(-0.4, 0.4, 2)
    strength = rng.uniform(4.0, 5.0)
    nx, ny = case["nx"], case["ny"]
    dx, dy = 10.0 / nx, 10.0 / ny
    x = (torch.arange(nx, device=_dev(), dtype=torch.float64) + 0.5) * dx - cx
    y = (torch.arange(ny, device=_dev(), dtype=torch.float64) + 0.5) * dy - cy
    X, Y = x[None, :].expand(ny, nx), y[:, None].expand(ny, nx)
    e = torch.exp(0.5 * (1.0 - X * X - Y * Y))
    T = 1.0 - (GAMMA - 1.0) * strength ** 2 / (8.0 * GAMMA * math.pi ** 2) * e * e
    rho = T ** (1.0 / (GAMMA - 1.0))
    k = strength / (2.0 * math.pi)
    prim = [rho, 1.0 - k * e * Y, 1.0 + k * e * X, rho ** GAMMA]
    if case["kind"] == "grad":  # weak waves over the whole domain
        for i, q in enumerate(prim):
            a, b, c = rng.uniform(-math.pi, math.pi, 3)
            prim[i] = q * (1.0 + 1e-2 * torch.sin(0.2 * math.pi * (X + cx) + a)
                           * torch.sin(0.4 * math.pi * (Y + cy) + b)
                           + 1e-2 * torch.sin(0.2 * math.pi * (X + Y) + c))
    return _conserved(*prim).contiguous(), dx, dy


def _batch_states(case, seed):
    """Riemann problems on [0, 1] packed one after another, their sizes log-uniform in
    [128, 8192] (the same ones for every seed) and their two states seeded."""
    n = case["nprob"]
    sizes = np.rint(np.exp(np.random.default_rng(n).uniform(math.log(128), math.log(8192), n)))
    sizes = sizes.astype(np.int64)
    prim = np.random.default_rng(seed).uniform([0.1, -1.0, 0.1], [2.0, 1.0, 10.0], size=(n, 2, 3))
    left = torch.arange(int(sizes.max()), device=_dev())
    U = torch.from_numpy(np.stack([workloads.conserved_1d(*q.T) for q in prim.transpose(1, 0, 2)],
                                  -1)).to(_dev())  # [3][problem][side]
    parts = []
    for p, m in enumerate(sizes.tolist()):
        parts.append(torch.where(left[:m] + 0.5 < 0.5 * m, U[:, p, :1], U[:, p, 1:]).reshape(-1))
    return sizes, torch.cat(parts), 1.0 / sizes


def _line_state(case, seed):
    rng = np.random.default_rng(seed)
    n = case["n"]
    if case["kind"] == "advection":
        x, h = workloads.periodic_grid(-1.0, 1.0, n)
        u = rng.uniform(0.5, 1.5) * np.sin(np.pi * (x + rng.uniform(-1.0, 1.0)))
        if n > 1000:  # the smooth wave of the accuracy test carries a square pulse
            u = u + np.where(np.abs(x - rng.uniform(-0.5, 0.5)) <= 0.25, 1.0, 0.0)
    elif case["kind"] == "burgers":
        x, h = workloads.periodic_grid(0.0, 2.0, n)
        u = 1.0 + rng.uniform(0.3, 0.6) * np.sin(np.pi * (x + rng.uniform(-1.0, 1.0))) ** 3
    else:
        x, h = workloads.centred_grid(-5.0, 5.0, n)
        left = x < -4.0
        wave = 1.0 + rng.uniform(0.15, 0.25) * np.sin(5.0 * x + rng.uniform(-1.0, 1.0))
        u = workloads.conserved_1d(np.where(left, 3.857143, wave), np.where(left, 2.629369, 0.0),
                                   np.where(left, 10.33333, 1.0))
    return torch.from_numpy(np.ascontiguousarray(u)).to(_dev()), h


def _mach_state(case, seed):
    """Double Mach reflection; the Mach number varies a little with the seed."""
    U, dx, dy, sides = workloads.double_mach(case["nx"], case["ny"])
    f = 1.0 + 0.02 * np.random.default_rng(seed).uniform(-1.0, 1.0)
    U[3] *= f  # a little more or less pressure and energy everywhere
    sides = tuple((k0, None if a is None else a * np.array([1, 1, 1, f]), k1,
                   None if b is None else b * np.array([1, 1, 1, f]), s0, r)
                  for k0, a, k1, b, s0, r in sides)
    return torch.from_numpy(U).to(_dev()), dx, dy, sides


def _initial(case, seed):
    """(state, dx, dy or None, sides or None)."""
    kind = case["kind"]
    if kind in ("advection", "burgers", "euler1d"):
        U, h = _line_state(case, seed)
        return U, h, None, None
    if kind == "riemann":
        return (*_riemann_state(case, seed), None)
    if kind in ("vortex", "grad"):
        return (*_vortex_state(case, seed), None)
    return _mach_state(case, seed)


def _target(case, U, seed):
    """The density a gradient case is compared with: the initial one, perturbed."""
    g = torch.Generator(device=U.device)
    g.manual_seed(seed)
    return U[0] * (1.0 + 1e-3 * torch.randn(U[0].shape, dtype=U.dtype, device=U.device,
                                            generator=g))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        sizes, U0, hs = _batch_states(case, seed)
        b = enomr.Batch(sizes, hs, order=case["order"], bc=enomr.TRANSMISSIVE)
        b.autotune(U0)
        return {"case": case, "batch": b, "U0": U0, "U": torch.empty_like(U0)}
    U0, dx, dy, sides = _initial(case, seed)
    eq = {"advection": enomr.ADVECTION, "burgers": enomr.BURGERS}.get(kind, enomr.EULER)
    bc = (enomr.PERIODIC if kind in ("advection", "burgers", "vortex", "grad")
          else enomr.TRANSMISSIVE)
    shape = case["n"] if dy is None else (case["ny"], case["nx"])
    solver = enomr.Solver(eq, shape, order=case["order"], dx=dx, dy=dy, bc=bc, gamma=GAMMA)
    state = {"case": case, "solver": solver, "U0": U0}
    if kind == "grad":
        state["target"] = _target(case, U0, seed)
        U0.requires_grad_(True)
    elif kind == "mach":
        solver.set_sides(sides)
        state["U"] = U0
    else:
        state["U"] = torch.empty_like(U0)
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind, steps, cfl = case["kind"], case["steps"], _cfl(case)
    if kind == "grad":
        U0 = state["U0"]
        U0.grad = None
        U = enomr.rollout(U0, state["solver"], steps, cfl=cfl)
        (0.5 * ((U[0] - state["target"]) ** 2).sum()).backward()
        return {"U": U.detach(), "grad": U0.grad}
    U = state["U"]
    if kind != "mach":  # the moving inflow goes on in time: that run continues instead
        U.copy_(state["U0"])
    if kind == "batch":
        for _ in range(steps):
            state["batch"].step(U, cfl)
    else:
        for _ in range(steps):
            state["solver"].step(U, 0.0, cfl)
    return U


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind, R, steps = case["kind"], case["order"], case["steps"]
    if kind in ("advection", "burgers"):
        # per cell and stage: one reconstruction (R products), the difference, the combination
        cells, comps, per = case["n"], 1, 2 * R + 8
    elif kind == "euler1d":
        cells, comps, per = case["n"], 3, 3 * 2 * 2 * R + 100
    elif kind == "batch":
        # log-uniform sizes in [128, 8192]; most cells lie on one of two constant states
        cells, comps, per = int(case["nprob"] * (8192 - 128) / math.log(64.0)), 3, 15
    else:
        cells, comps = case["nx"] * case["ny"], 4
        per = 2 * (4 * 2 * 2 * R + 100)  # two directions, both sides, four components
        if kind == "riemann":  # away from the fronts only the stage combination is left
            band = min(1.0, (2 * case["developed"] + 2 * R) * (case["nx"] + case["ny"]) / cells)
            per = band * per + 16
        elif kind == "mach":
            per = 0.2 * per + 16
    passes = steps * (4 if kind == "grad" else 1)  # the gradient: each stage again, and its transpose
    return {"bytes": 2 * 8 * comps * cells * (2 if kind == "grad" else 1),
            "flops": 3 * passes * per * cells}


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------
def _conserved(rho, u, v, p):
    return torch.stack([rho, rho * u, rho * v, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)])


def _pressure(U):
    m2 = sum(U[k] * U[k] for k in range(1, U.shape[0] - 1))
    return (GAMMA - 1.0) * (U[-1] - 0.5 * m2 / U[0])


def _sound(U):
    return torch.sqrt(GAMMA * _pressure(U) / U[0])


def _flux(U, axis):
    """Euler flux along `axis` (0: x), component order of U."""
    p, u = _pressure(U), U[1 + axis] / U[0]
    F = [U[k] * u for k in range(U.shape[0])]
    F[1 + axis] = F[1 + axis] + p
    F[-1] = F[-1] + p * u
    return torch.stack(F)


# the candidate stencils S(-m, n) in the order in which they are tested
_ORDERED = [(8, 8), (7, 8), (8, 7), (7, 7), (8, 6), (6, 7), (7, 6), (6, 6), (7, 5), (5, 6), (6, 5),
            (5, 5), (6, 4), (4, 5), (5, 4), (4, 4), (5, 3), (3, 4), (4, 3), (3, 3), (2, 3), (3, 2),
            (2, 2), (1, 2), (2, 1), (1, 1)]


@functools.lru_cache(None)
def _tables(order):
    """[(m, n, a, b)]: interface-value and undivided-difference weights over S(-m, n)."""
    g, rows = (order + 1) // 2, []
    for m, n in _ORDERED:
        if m > g - 1 or n > g - 1:
            continue
        k = m + n
        # moments: the cell averages of x^d over cell c are exact for the weights
        A = [[((Fraction(2 * c + 1, 2)) ** (d + 1) - (Fraction(2 * c - 1, 2)) ** (d + 1)) / (d + 1)
              for c in range(-m, n + 1)] + [Fraction(1, 2) ** d] for d in range(k + 1)]
        for i in range(k + 1):  # Gauss-Jordan elimination
            piv = next(r for r in range(i, k + 1) if A[r][i] != 0)
            A[i], A[piv] = A[piv], A[i]
            A[i] = [v / A[i][i] for v in A[i]]
            for r in range(k + 1):
                if r != i and A[r][i] != 0:
                    A[r] = [v - A[r][i] * w for v, w in zip(A[r], A[i])]
        a = [float(A[i][k + 1]) for i in range(k + 1)]
        b = [float((-1) ** (k - i) * math.comb(k, i)) for i in range(k + 1)]
        rows.append((m, n, a, b))
    return rows


def _reconstruct(v, order):
    """Value at the right face of the middle cell of the window v (a list of tensors)."""
    c = (order + 1) // 2 - 1
    with torch.no_grad():
        dl, dr = (v[c] - v[c - 1]).abs(), (v[c] - v[c + 1]).abs()
        dl = torch.maximum(dl, ((v[c] - 2 * v[c - 1]) + v[c - 2]).abs())
        dr = torch.maximum(dr, ((v[c] - 2 * v[c + 1]) + v[c + 2]).abs())
        base = torch.minimum(dl, dr)
        left = torch.ones_like(base, dtype=torch.bool)
    a1, b1 = v[c + 1] - v[c], v[c] - v[c - 1]
    small = torch.where(a1.abs() <= b1.abs(), a1, b1)
    same = ((a1 > 0) & (b1 > 0)) | ((a1 < 0) & (b1 < 0))
    value = v[c] + 0.5 * torch.where(same, small, torch.zeros_like(small))
    for m, n, a, b in _tables(order):
        with torch.no_grad():
            s = sum(w * v[c - m + i] for i, w in enumerate(b))
            hit = left & (s.abs() < base)
            left = left & ~hit
            if not bool(hit.any()):
                continue
        value = torch.where(hit, sum(w * v[c - m + i] for i, w in enumerate(a)), value)
    return value


def _pad(U, g, bc):
    """Ghost cells along the last dimension."""
    if bc == "periodic":
        return torch.cat([U[..., -g:], U, U[..., :g]], -1)
    lo = U[..., :1].expand(*U.shape[:-1], g)
    return torch.cat([lo, U, U[..., -1:].expand(*U.shape[:-1], g)], -1)


def _pad_sides(U, g, low, high, h_along, t):
    """As _pad with a side at each end; U [C][lines][n], components in line order."""
    ends = []
    for end, (k_lo, st_lo, k_hi, st_hi, split, rate) in enumerate((low, high)):
        edge = U[..., :1] if end == 0 else U[..., -1:]
        near = U[..., :g] if end == 0 else U[..., -g:]
        mirror = near.flip(-1) * torch.tensor([1.0, -1.0, 1.0, 1.0], device=U.device,
                                              dtype=U.dtype)[:, None, None]
        def ghost(kind, st):
            if kind == "inflow":
                return st[:, None, None].expand_as(near)
            return mirror if kind == "reflective" else edge.expand_as(near)
        pos = (torch.arange(U.shape[1], device=U.device, dtype=U.dtype) + 0.5) * h_along
        below = (pos < split + rate * t)[None, :, None]
        ends.append(torch.where(below, ghost(k_lo, st_lo), ghost(k_hi, st_hi)))
    return torch.cat([ends[0], U, ends[1]], -1)


def _speeds(U):
    u, c = U[1] / U[0], _sound(U)
    return (u - c).abs(), u.abs(), (u + c).abs()


def _sweep(U, E, order, h, alpha=None):
    """-dF/dx of Euler states U [C][lines][n] (line order), E with g ghost cells."""
    g, n, C = (order + 1) // 2, U.shape[-1], U.shape[0]
    if alpha is None:
        alpha = [s.max(-1, keepdim=True).values for s in _speeds(U)]
    F = _flux(E, 0)
    w = torch.sqrt(E[0])
    prim = [E[1] / E[0], E[2] / E[0] if C == 4 else None, (E[-1] + _pressure(E)) / E[0]]
    lo, hi = slice(g - 1, g + n), slice(g, g + n + 1)
    u, v, H = (None if q is None else (w[..., lo] * q[..., lo] + w[..., hi] * q[..., hi])
               / (w[..., lo] + w[..., hi]) for q in prim)
    q2 = 0.5 * (u * u + (v * v if C == 4 else 0.0))
    c2 = (GAMMA - 1.0) * (H - q2)
    c = torch.sqrt(c2)
    b = (GAMMA - 1.0) / c2
    one, nil = torch.ones_like(u), torch.zeros_like(u)
    if C == 4:
        L = [(0.5 * (b * q2 + u / c), -0.5 * (b * u + 1 / c), -0.5 * b * v, 0.5 * b),
             (1 - b * q2, b * u, b * v, -b), (-v, nil, one, nil),
             (0.5 * (b * q2 - u / c), -0.5 * (b * u - 1 / c), -0.5 * b * v, 0.5 * b)]
        R = [(one, u - c, v, H - u * c), (one, u, v, q2), (nil, nil, one, v),
             (one, u + c, v, H + u * c)]
        speed = [0, 1, 1, 2]
    else:
        L = [(0.5 * (b * q2 + u / c), -0.5 * (b * u + 1 / c), 0.5 * b), (1 - b * q2, b * u, -b),
             (0.5 * (b * q2 - u / c), -0.5 * (b * u - 1 / c), 0.5 * b)]
        R = [(one, u - c, H - u * c), (one, u, q2), (one, u + c, H + u * c)]
        speed = [0, 1, 2]
    out = [0.0] * C
    for l, r, k in zip(L, R, speed):
        vp, vm = [], []
        for j in range(2 * g):
            at = slice(j, j + n + 1)
            wU = sum(l[q] * E[q][..., at] for q in range(C))
            wF = sum(l[q] * F[q][..., at] for q in range(C))
            vp.append(0.5 * (wF + alpha[k] * wU))
            vm.append(0.5 * (wF - alpha[k] * wU))
        f = _reconstruct(vp[:-1], order) + _reconstruct(vm[:0:-1], order)
        out = [o + f * r[q] for q, o in enumerate(out)]
    f = torch.stack(out)
    return -(f[..., 1:] - f[..., :-1]) / h


_SWAP = [0, 2, 1, 3]


def _rhs(case, U, dx, dy, sides, t):
    order, kind = case["order"], case["kind"]
    g = (order + 1) // 2
    if kind == "advection":
        E = _pad(U, g, "periodic")
        f = _reconstruct([E[j:j + U.numel() + 1] for j in range(2 * g - 1)], order)
        return -(f[1:] - f[:-1]) / dx
    if kind == "burgers":  # u > 0: no split
        E = _pad(0.5 * U * U, g, "periodic")
        f = _reconstruct([E[j:j + U.numel() + 1] for j in range(2 * g - 1)], order)
        return -(f[1:] - f[:-1]) / dx
    bc = "periodic" if kind in ("vortex", "grad") else "transmissive"
    if kind == "euler1d":
        V = U[:, None, :]
        return _sweep(V, _pad(V, g, bc), order, dx)[:, 0]
    V = U[_SWAP].transpose(1, 2)
    if sides is None:
        Ex, Ey = _pad(U, g, bc), _pad(V, g, bc)
    else:
        def dev(s, swap):
            st = [None if a is None else torch.as_tensor(a, device=U.device, dtype=U.dtype)
                  for a in (s[1], s[3])]
            st = [a[_SWAP] if swap and a is not None else a for a in st]
            return s[0], st[0], s[2], st[1], s[4], s[5]
        Ex = _pad_sides(U, g, dev(sides[0], False), dev(sides[1], False), dy, t)
        Ey = _pad_sides(V, g, dev(sides[2], True), dev(sides[3], True), dx, t)
    if U.requires_grad or U.shape[1] * U.shape[2] < 1 << 20:
        return (_sweep(U, Ex, order, dx)
                + _sweep(V, Ey, order, dy).transpose(1, 2)[_SWAP])
    D = torch.empty_like(U)
    for a in range(0, U.shape[1], 512):  # some lines at a time
        D[:, a:a + 512] = _sweep(U[:, a:a + 512], Ex[:, a:a + 512], order, dx)
    for a in range(0, U.shape[2], 512):
        D[:, :, a:a + 512] += _sweep(V[:, a:a + 512], Ey[:, a:a + 512], order,
                                     dy).transpose(1, 2)[_SWAP]
    return D


def _time_step(case, U, dx, dy):
    cfl = _cfl(case)
    with torch.no_grad():
        if case["kind"] == "advection":
            return cfl * dx
        if case["kind"] == "burgers":
            return cfl / float(U.abs().max() * (1.0 / dx))
        c = _sound(U)
        s = ((U[1] / U[0]).abs() + c) * (1.0 / dx)
        if dy is not None:
            s = s + ((U[2] / U[0]).abs() + c) * (1.0 / dy)
        return cfl / float(s.max())


def _steps(case, U, dx, dy, sides):
    t = 0.0
    for _ in range(case["steps"]):
        dt = _time_step(case, U, dx, dy)
        U1 = U + dt * _rhs(case, U, dx, dy, sides, t)
        U2 = 0.75 * U + 0.25 * (U1 + dt * _rhs(case, U1, dx, dy, sides, t + dt))
        U = U / 3.0 + (2.0 / 3.0) * (U2 + dt * _rhs(case, U2, dx, dy, sides, t + 0.5 * dt))
        t += dt
    return U


def _batch_steps(case, sizes, packed, hs):
    """All problems as one line, each with its own ghost cells, split speeds and time step."""
    g, dev = (case["order"] + 1) // 2, packed.device
    n = torch.from_numpy(sizes).to(dev)
    base = torch.cumsum(n, 0) - n
    prob = torch.repeat_interleave(torch.arange(len(sizes), device=dev), n)
    cell = torch.arange(prob.numel(), device=dev) - base[prob]
    at = 3 * base[prob] + cell  # where component 0 of a cell is
    U = torch.stack([packed[at + q * n[prob]] for q in range(3)])
    wide = n + 2 * g
    start = torch.cumsum(wide, 0) - wide
    own = torch.repeat_interleave(torch.arange(len(sizes), device=dev), wide)
    j = torch.arange(own.numel(), device=dev) - start[own] - g
    ghosted = base[own] + torch.minimum(j.clamp_min(0), n[own] - 1)
    inner = start[prob] + cell  # a cell's place in the line without the line's first g cells
    own = own[g:own.numel() - g + 1]  # the problem of each face: the one of the cell to its right
    h = torch.from_numpy(hs).to(dev)

    def worst(s):
        return torch.zeros_like(h).scatter_reduce(0, prob, s, "amax")

    def rhs(U):
        E = U[:, None, ghosted]
        alpha = [worst(s)[own][None] for s in _speeds(U)]
        return _sweep(E[..., g:-g], E, case["order"], 1.0, alpha)[:, 0, inner] / h[prob]

    for _ in range(case["steps"]):
        s = _speeds(U)
        dt = (_cfl(case) / (torch.maximum(worst(s[0]), worst(s[2])) * (1.0 / h)))[prob]
        U1 = U + dt * rhs(U)
        U2 = 0.75 * U + 0.25 * (U1 + dt * rhs(U1))
        U = U / 3.0 + (2.0 / 3.0) * (U2 + dt * rhs(U2))
    out = torch.empty_like(packed)
    for q in range(3):
        out[at + q * n[prob]] = U[q]
    return out


def exact(case, seed):
    if case["kind"] == "batch":
        return _batch_steps(case, *_batch_states(case, seed))
    U0, dx, dy, sides = _initial(case, seed)
    if case["kind"] == "grad":
        target = _target(case, U0, seed)
        U0.requires_grad_(True)
        U = _steps(case, U0, dx, dy, sides)
        (0.5 * ((U[0] - target) ** 2).sum()).backward()
        return {"U": U.detach(), "grad": U0.grad}
    return _steps(case, U0, dx, dy, sides)
