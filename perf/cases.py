"""Workloads of the library as a user's program runs them, for timing and for comparing results.

A case is a dict of plain values.  ``path`` names what is called:

  step       one ``Hydro.step_cfl`` of a uniform lattice (the time loop of a run)
  advance    ``Hydro.advance`` over ``steps`` steps with the dt history kept
  graph      ``Hydro.advance_graph`` over ``steps`` steps (launch-bound runs)
  ensemble   one ``step_cfl`` of many independent periodic 2-D problems in one context
  two_level  one ``step_cfl`` of a two-level composite grid (a refined box)
  gradient   forward run and gradient through ``adjoint.run_differentiable``
  host       one ``Hydro.step_host_interior`` of a state in pinned host memory
  guards     ``fill_guardcells`` and ``compute_dt`` (start of a run, after a restart or for output)

Every state is FP64, the only type the library computes in.  ``exact`` is the same method
written with plain torch operations on global (unblocked) float64 arrays.
"""
from __future__ import annotations

import math

import numpy as np
import torch

GAMMA, CFL = 1.4, 0.8


def _case(name, path, ndim, n, nz, nb, ng=4, bc="ooo", problem="blast", stages=2, telescoping=False, steps=1,
          every=1, count=1, size=0):
    """bc: one letter per dimension, o(utflow) or p(eriodic).  size: an ensemble's largest problem, in cells."""
    c = {"path": path, "ndim": ndim, "n": n, "nz": nz, "nbx": nb[0], "nby": nb[1], "nbz": nb[2], "ng": ng, "bc": bc,
         "problem": problem, "stages": stages, "telescoping": telescoping, "steps": steps, "every": every,
         "count": count, "size": size}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest standard setup: a 2-D Sod tube of 128^2 in 64 blocks, one step
        _case("sod2d_128", "step", 2, 16, 1, (8, 8, 1), problem="sod"),
        # a launch-bound run: small blocks, an odd lattice, periodic, ten steps in one graph
        _case("kh2d_104x56_graph", "graph", 2, 8, 1, (13, 7, 1), bc="ppo", problem="kh", steps=10),
        # the batched ensemble: 96 independent periodic problems of 64^2 .. 512^2
        _case("ensemble2d_96", "ensemble", 2, 16, 1, (1, 1, 1), bc="ppo", problem="kh", count=96, size=512),
        # a smoke-test-sized 3-D blast: eight blocks
        _case("blast3d_32", "step", 3, 16, 16, (2, 2, 2)),
        # blocks of 8 x 8 x 12, an odd lattice, mixed boundaries, three-stage Runge-Kutta, a dt history
        _case("blast3d_40x24x84_rk3", "advance", 3, 8, 12, (5, 3, 7), bc="pop", stages=3, steps=3),
        # the mid-sized blast of the full-run checks
        _case("blast3d_128", "step", 3, 16, 16, (8, 8, 8)),
        # the headline size, 4096 blocks of 16^3
        _case("blast3d_256", "step", 3, 16, 16, (16, 16, 16)),
        # telescoping stages: one guard fill per step
        _case("telescoping3d_96", "step", 3, 16, 16, (6, 6, 6), telescoping=True),
        # a blast in a refined box: 512 coarse and 512 fine blocks
        _case("two_level3d_128", "two_level", 3, 16, 16, (8, 8, 8)),
        # gradient of a loss of the final state with respect to the initial fields, checkpointed
        _case("gradient2d_256", "gradient", 2, 16, 1, (16, 16, 1), problem="smooth", steps=4, every=2),
        # a state that lives in host memory, both copies in every step
        _case("host3d_128", "host", 3, 16, 16, (8, 8, 8)),
        # guard cells filled and the CFL time step reduced on a given state
        _case("guards3d_128", "guards", 3, 16, 16, (8, 8, 8)),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lattice3(rng, n, nz, cells):
    """Blocks per dimension of a 3-D lattice of about `cells` cells, uneven."""
    side = cells ** (1 / 3)
    return tuple(max(1, min(16 * 16 // b, int(round(side * rng.uniform(0.7, 1.4) / b)))) for b in (n, n, nz))


def draw(rng):
    path = rng.choice(["step", "step", "advance", "graph", "ensemble", "two_level", "gradient", "host", "guards"])
    n = rng.choice([4, 8, 16, 16, 16])
    bc = "".join(rng.choice("op") for _ in range(3))
    if path == "ensemble":
        return _case("", path, 2, rng.choice([8, 16, 16]), 1, (1, 1, 1), bc="ppo", problem="kh",
                     count=_log(rng, 3, 96), size=rng.choice([64, 128, 256, 512]))
    if path == "gradient":
        k = rng.randint(2, 5)
        return _case("", path, 2, n, 1, (_log(rng, 3, 24), _log(rng, 3, 24), 1), bc=bc[:2] + "o", problem="smooth",
                     steps=k, every=rng.randint(1, k))
    if path == "two_level":
        n = rng.choice([8, 16, 16])
        return _case("", path, 3, n, n, tuple(rng.randint(3, 8) for _ in range(3)), bc=bc)
    if path in ("step", "advance", "graph"):
        steps = 1 if path == "step" else rng.randint(2, 6)
        stages = rng.choice([2, 2, 3])
        tele = rng.random() < 0.3
        if tele:
            n = rng.choice([8, 16])
        ng = 2 * stages if tele else rng.choice([2, 4, 4]) if n == 4 else 4
        if rng.random() < 0.4:
            return _case("", path, 2, n, 1, (_log(rng, 2, 64), _log(rng, 2, 64), 1), ng=ng, bc=bc[:2] + "o",
                         problem=rng.choice(["sod", "kh"]), stages=stages, telescoping=tele, steps=steps)
        nz = rng.choice([n, n, n + 4])
        # a drawn case stays below one two-stage step of 256^3
        cells = _log(rng, 4e3, 1.2e7 / (steps * (stages - 1) * (2 if tele else 1)))
        return _case("", path, 3, n, nz, _lattice3(rng, n, nz, cells), ng=ng, bc=bc, stages=stages, telescoping=tele,
                     steps=steps)
    nz = rng.choice([n, n, n + 4])
    return _case("", path, 3, n, nz, _lattice3(rng, n, nz, _log(rng, 3e4, 5e6)), bc=bc)


# -- geometry ------------------------------------------------------------------

def _cells(case):
    """Global interior cells (x, y, z)."""
    return case["nbx"] * case["n"], case["nby"] * case["n"], case["nbz"] * case["nz"]


def _sizes(case):
    """Sizes of an ensemble's problems: uneven, up to case["size"], whole blocks."""
    rng = np.random.Generator(np.random.PCG64(7))
    choices = [s for s in (64, 128, 256, 512) if s <= case["size"]]
    return [int(choices[i]) for i in rng.integers(0, len(choices), case["count"])]


def _box(case):
    """The refined box of a two-level case, in coarse blocks."""
    nb = (case["nbx"], case["nby"], case["nbz"])
    lo = tuple(max(1, b // 4) for b in nb)
    return lo, tuple(max(l + 1, b - max(1, b // 4)) for l, b in zip(lo, nb))


def _width(case):
    """Equal cell widths in every dimension; the longest side has length 1."""
    return 1.0 / max(_cells(case)[: case["ndim"]])


def _to_blocks(G, n):
    """[5, nz, ny, nx] -> [blocks, 5, n2, n1, n0], x fastest."""
    s = G.shape
    b = [s[1 + d] // n[2 - d] for d in range(3)]
    v = G.reshape(5, b[0], n[2], b[1], n[1], b[2], n[0])
    return v.permute(1, 3, 5, 0, 2, 4, 6).reshape(-1, 5, n[2], n[1], n[0])


def _padded(B, ng, ndim):
    gz = ng if ndim == 3 else 0
    s = B.shape
    U = torch.zeros((s[0], 5, s[2] + 2 * gz, s[3] + 2 * ng, s[4] + 2 * ng), dtype=torch.float64, device=B.device)
    _interior(U, ng, ndim).copy_(B)
    return U


def _interior(U, ng, ndim):
    U = U[..., ng:-ng, ng:-ng]
    return U[:, :, ng:-ng] if ndim == 3 else U


# -- initial states --------------------------------------------------------------

def _centres(shape, h, origin, device):
    ax = [origin[d] + (torch.arange(shape[d], dtype=torch.float64, device=device) + 0.5) * h for d in range(3)]
    return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]


def _initial(problem, shape, h, origin, extent, seed, device, primitive=False, reach=None):
    """Global [5, nz, ny, nx] state of `shape` (x, y, z) cells of width h; `extent`: the domain's; `reach`: the
    width a blast's radius goes by (the refined box's, which holds the shock as a refinement criterion would)."""
    g = torch.Generator(device="cpu").manual_seed(seed)
    r = lambda lo, hi: lo + (hi - lo) * float(torch.rand((), generator=g, dtype=torch.float64))  # noqa: E731
    X, Y, Z = _centres(shape, h, origin, device)
    full = (shape[2], shape[1], shape[0])
    zero = torch.zeros(full, dtype=torch.float64, device=device)
    gd = torch.Generator(device=device).manual_seed(seed + 1)
    noise = torch.randn(full, generator=gd, dtype=torch.float64, device=device)
    if problem == "blast":
        # a blast wave after some time: a dense shell behind a strong shock, cold noisy gas outside
        two_d = shape[2] == 1
        c = [extent[d] * r(0.45, 0.55) for d in range(3)]
        R = r(0.2, 0.3) * (reach or min(extent[:2] if two_d else extent))
        dx, dy, dz = X - c[0], Y - c[1], (Z - c[2]) * (0.0 if two_d else 1.0)
        s = torch.sqrt(dx * dx + dy * dy + dz * dz) / R + zero
        inside = s < 1.0
        s4 = s ** 4
        rho = torch.where(inside, 0.05 + 4.0 * s4 * s4, 1.0) * torch.exp(0.02 * noise)
        p = torch.where(inside, 0.4 + 0.6 * s4, 1e-5 * (1.0 + 0.1 * torch.rand(full, generator=gd, dtype=torch.float64, device=device)))
        f = torch.where(inside, 0.9 / R, 0.0)
        u, v, w = dx * f, dy * f, dz * f
    elif problem == "sod":
        left = (X < extent[0] * r(0.4, 0.6)) & (zero == 0)
        rho = torch.where(left, 1.0, 0.125) * torch.exp(0.02 * noise)
        p = torch.where(left, 1.0, 0.1)
        u, v, w = zero, zero, zero
    elif problem == "kh":
        inner = ((Y - 0.5 * extent[1]).abs() < 0.25 * extent[1]) & (zero == 0)
        rho = torch.where(inner, 2.0, 1.0) * torch.exp(0.1 * noise)
        u = torch.where(inner, 0.5, -0.5)
        v = 0.01 * torch.sin(4.0 * math.pi * (X / extent[0] + r(0, 1))) + zero
        w, p = zero, zero + 2.5
    else:
        # a smoothed Sod jump with 2-D modulations of every field: no field is locally constant
        x, y = X / extent[0], Y / extent[1]
        a, b, k = r(0, 1), r(0, 1), 2.0 * math.pi
        s = 0.5 * (1.0 - torch.tanh((X - 0.5 * extent[0]) / (2.0 * h)))
        mod = 1.0 + 0.05 * torch.sin(k * x + 0.3 + a) * torch.sin(k * y + 0.7 + b)
        rho, p = (0.125 + 0.875 * s) * mod * torch.exp(0.01 * noise), (0.1 + 0.9 * s) * (2.0 - mod)
        u = 0.05 * torch.sin(k * y + 0.2 + a) * torch.cos(math.pi * x + 0.1) + zero
        v = 0.05 * torch.cos(k * x + 0.4 + b) * torch.sin(k * y + 0.9) + zero
        w = zero
    W = torch.stack([q + zero for q in (rho, u, v, w, p)])
    return W if primitive else _conserved(W)


def _conserved(W):
    rho, u, v, w, p = W
    return torch.stack([rho, rho * u, rho * v, rho * w, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v + w * w)])


def _globals(case, seed, device):
    """The case's initial data as a list of global arrays (an ensemble's problems; a two-level grid's coarse
    and fine arrays) with the cell width of each."""
    if case["path"] == "ensemble":
        out = []
        for i, s in enumerate(_sizes(case)):
            kind = "kh" if i % 2 else "sod"
            out.append((_initial(kind, (s, s, 1), 1.0 / s, (0.0,) * 3, (1.0,) * 3, seed * 1000 + i, device), 1.0 / s))
        return out
    h = _width(case)
    shape = _cells(case)
    extent = [shape[d] * h for d in range(3)]
    if case["path"] == "two_level":
        lo, hi = _box(case)
        n = (case["n"], case["n"], case["nz"])
        fine = tuple(2 * (hi[d] - lo[d]) * n[d] for d in range(3))
        reach = 0.5 * h * min(fine)
        return [(_initial(case["problem"], shape, h, (0.0,) * 3, extent, seed, device, reach=reach), h),
                (_initial(case["problem"], fine, 0.5 * h, [lo[d] * n[d] * h for d in range(3)], extent, seed, device,
                          reach=reach), 0.5 * h)]
    return [(_initial(case["problem"], shape, h, (0.0,) * 3, extent, seed, device, case["problem"] == "smooth"), h)]


# -- what a user's program has in hand ---------------------------------------------

class _Lat:
    """A lattice as Hydro.from_lattice and its relatives take it."""

    def __init__(self, case, cells=None, h=None):
        n = (case["n"], case["n"], case["nz"])
        cells = _cells(case) if cells is None else cells
        h = _width(case) if h is None else h
        self.ndim, self.n, self.ng = case["ndim"], n, case["ng"]
        self.nb = tuple(cells[d] // n[d] for d in range(3))
        self.bc = tuple("periodic" if b == "p" else "outflow" for b in case["bc"])
        self.extent = tuple(cells[d] * h for d in range(3))
        self.dx = (h,) * 3


class _TwoLevel:
    def __init__(self, case):
        self.coarse = _Lat(case)
        self.lo, self.hi = _box(case)


def prepare(case, seed):
    from paper_2401_03378_gb300 import Hydro

    n, ng, nd = (case["n"], case["n"], case["nz"]), case["ng"], case["ndim"]
    blocks = torch.cat([_to_blocks(G, n) for G, _ in _globals(case, seed, "cuda")])
    if case["path"] == "ensemble":
        h = Hydro.from_batch([_Lat(case, (s, s, 1), 1.0 / s) for s in _sizes(case)], gamma=GAMMA, cfl=CFL)
    elif case["path"] == "two_level":
        h = Hydro.from_two_level(_TwoLevel(case), gamma=GAMMA, cfl=CFL)
    else:
        h = Hydro.from_lattice(_Lat(case), gamma=GAMMA, cfl=CFL)
    if case["stages"] != 2:
        h.set_rk_stages(case["stages"])
    if case["telescoping"]:
        h.set_telescoping(True)
    U = _padded(blocks, ng, nd)
    state = {"case": case, "h": h, "U": U}
    if case["path"] == "gradient":
        g = torch.Generator(device="cuda").manual_seed(seed + 5)
        state["W"] = U.requires_grad_(True)
        state["g"] = torch.randn(U.shape, generator=g, dtype=torch.float64, device="cuda")
        return state
    state["dt"] = h.compute_dt(U)
    if case["path"] == "advance":
        state["hist"] = torch.zeros(case["steps"], dtype=torch.float64, device="cuda")
    if case["path"] == "host":
        state["U_host"] = torch.empty(blocks.shape, dtype=torch.float64, pin_memory=True)
        state["U_host"].copy_(blocks)
        state["dt_host"] = state["dt"].cpu().numpy()
        del state["U"]
    return state


def run(state):
    case, h = state["case"], state["h"]
    path, ng, nd = case["path"], case["ng"], case["ndim"]
    if path == "gradient":
        from paper_2401_03378_gb300.adjoint import run_differentiable

        U = run_differentiable(h, state["W"], case["steps"], case["every"])
        (gW,) = torch.autograd.grad(U, state["W"], state["g"])
        return {"U": _interior(U.detach(), ng, nd), "gradient": _interior(gW, ng, nd)}
    if path == "host":
        h.step_host_interior(state["U_host"], state["dt_host"])
        return {"U": state["U_host"], "dt": state["dt_host"]}
    U, dt = state["U"], state["dt"]
    if path == "guards":
        h.fill_guardcells(U)
        return {"U": U, "dt": h.compute_dt(U)}
    if path == "advance":
        h.advance(U, case["steps"], dt, state["hist"])
        return {"U": _interior(U, ng, nd), "dt": dt, "history": state["hist"]}
    if path == "graph":
        h.advance_graph(U, case["steps"], dt)
    else:
        h.step_cfl(U, dt)
    # guard cells hold unspecified values after a step
    return {"U": _interior(U, ng, nd), "dt": dt}


def work(case):
    """Bytes: the state's interior read once and written once.  Flops of the method on an unblocked grid
    (+ - * / sqrt one each): conversion 13, slopes and face states 11 per variable and dimension, HLLC 114 a
    face, update 3 per variable and dimension plus the combine, signal speed 11."""
    nd, S = case["ndim"], case["stages"]
    if case["path"] == "ensemble":
        zones = sum(s * s for s in _sizes(case))
    else:
        x, y, z = _cells(case)
        zones = x * y * z
    if case["path"] == "two_level":
        lo, hi = _box(case)
        box = math.prod((hi[d] - lo[d]) * (case["n"], case["n"], case["nz"])[d] for d in range(3))
        zones += box * 2 ** nd - box
    stage = 13 + 55 * nd + 114 * nd + 5 * (3 * nd + 1)
    flops = (S * stage + (S - 1) * 15 + 11) * zones * case["steps"]
    nbytes = 80 * zones
    if case["path"] == "gradient":
        # the reverse of every operation costs about two
        return {"bytes": 2 * nbytes, "flops": 3 * flops}
    if case["path"] == "guards":
        ng = case["ng"]
        padded = (case["n"] + 2 * ng) ** 2 * (case["nz"] + 2 * ng) / (case["n"] ** 2 * case["nz"])
        return {"bytes": int(40 * zones * padded), "flops": 24 * zones}
    return {"bytes": nbytes, "flops": flops}


# -- the method in plain torch on global arrays ---------------------------------------

def _axis(d):
    """Array axis of dimension d (0 = x) of [5, nz, ny, nx]."""
    return 3 - d


def _pad(A, d, width, periodic):
    k = A.shape[_axis(d)]
    i = torch.arange(-width, k + width, device=A.device)
    return A.index_select(_axis(d), i % k if periodic else i.clamp(0, k - 1))


def _cut(A, d, lo, hi):
    return A.narrow(_axis(d), lo, A.shape[_axis(d)] - lo - hi)


def _primitive(U):
    u, v, w = U[1] / U[0], U[2] / U[0], U[3] / U[0]
    return torch.stack([U[0], u, v, w, (GAMMA - 1.0) * (U[4] - 0.5 * U[0] * (u * u + v * v + w * w))])


def _mc(dm, dp):
    """The MC-limited slope."""
    m = torch.where(dm.abs() < dp.abs(), 2.0 * dm.abs(), 2.0 * dp.abs())
    c = 0.5 * (dm + dp).abs()
    m = torch.where(c < m, c, m)
    return torch.where(dm * dp > 0.0, torch.sign(dp) * m, torch.zeros_like(m))


def _flux(W, d):
    """HLLC fluxes at the faces of dimension d; W holds two more cells there on each side."""
    dq = _cut(W, d, 1, 0) - _cut(W, d, 0, 1)
    s = 0.5 * _mc(_cut(dq, d, 0, 1), _cut(dq, d, 1, 0))
    q = _cut(W, d, 1, 1)
    L, R = _cut(q + s, d, 0, 1), _cut(q - s, d, 1, 0)
    n, a, b = d + 1, (2, 1, 1)[d], (3, 3, 2)[d]
    rl, ul, pl, rr, ur, pr = L[0], L[n], L[4], R[0], R[n], R[4]
    cl, cr = torch.sqrt(GAMMA * pl / rl), torch.sqrt(GAMMA * pr / rr)
    el = pl / (GAMMA - 1.0) + 0.5 * rl * (L[1] ** 2 + L[2] ** 2 + L[3] ** 2)
    er = pr / (GAMMA - 1.0) + 0.5 * rr * (R[1] ** 2 + R[2] ** 2 + R[3] ** 2)
    sl, sr = torch.sqrt(rl), torch.sqrt(rr)
    wl, wr = sl / (sl + sr), sr / (sl + sr)
    u = wl * ul + wr * ur
    jump = (L[1] - R[1]) ** 2 + (L[2] - R[2]) ** 2 + (L[3] - R[3]) ** 2
    c = torch.sqrt(wl * cl ** 2 + wr * cr ** 2 + 0.5 * (GAMMA - 1.0) * wl * wr * jump)
    SL = torch.where(ul - cl < u - c, ul - cl, u - c)
    SR = torch.where(ur + cr > u + c, ur + cr, u + c)
    ml, mr = rl * (SL - ul), rr * (SR - ur)
    S = (pr - pl + ml * ul - mr * ur) / (ml - mr)
    left = S >= 0.0
    pick = lambda x, y: torch.where(left, x, y)  # noqa: E731
    r, v, p, e, SK = pick(rl, rr), pick(ul, ur), pick(pl, pr), pick(el, er), pick(SL, SR)
    va, vb = pick(L[a], R[a]), pick(L[b], R[b])
    outside = torch.where(left, SL >= 0.0, SR <= 0.0)
    k = r * (SK - v) / (SK - S)
    ek = k * (e / r + (S - v) * (S + p / (r * (SK - v))))
    F = [None] * 5
    for i, plain, state, star in ((0, r * v, r, k), (n, r * v * v + p, r * v, k * S), (a, r * v * va, r * va, k * va),
                                  (b, r * v * vb, r * vb, k * vb), (4, (e + p) * v, e, ek)):
        F[i] = torch.where(outside, plain, plain + SK * (star - state))
    return torch.stack(F)


def _rate(P, nd, width, h):
    """-div F on P's cells less `width` - 2 .. : P holds `width` more cells per side in every dimension and the
    result holds width - 2 of them."""
    out = 0.0
    for d in range(nd):
        Q = P
        for o in range(nd):
            if o != d:
                Q = _cut(Q, o, 2, 2)
        F = _flux(_primitive(Q), d)
        out = out - (_cut(F, d, 1, 0) - _cut(F, d, 0, 1)) / h
    return out


_STAGES = {2: ((0.0, 1.0), (0.5, 0.5)), 3: ((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0))}


def _shrink(P, nd, by):
    for d in range(nd):
        if by:
            P = _cut(P, d, by, by)
    return P


def _step(U, dt, case, h):
    nd, S, per = case["ndim"], case["stages"], [b == "p" for b in case["bc"]]
    reach = 2 * S if case["telescoping"] else 2
    X, width, base = U, 0, U
    for s, (a, b) in enumerate(_STAGES[S]):
        if not width:
            width = reach
            X = base if s == 0 else X
            for d in range(nd):
                X = _pad(X, d, reach, per[d])
            if s == 0:
                U0 = X
        R = _rate(X, nd, width, h)
        new = _shrink(X, nd, 2) + dt * R
        width -= 2
        X = a * _shrink(U0, nd, reach - width) + b * new if s else new
    return X


def _speed(U, nd, h):
    W = _primitive(U)
    c = torch.sqrt(GAMMA * W[4] / W[0])
    return sum((W[1 + d].abs() + c) / h for d in range(nd))


def _mean(A, dims):
    for d in dims:
        s = list(A.shape)
        ax = _axis(d)
        A = A.reshape(s[:ax] + [s[ax] // 2, 2] + s[ax + 1:]).mean(ax + 1)
    return A


def _window(A, lo, hi):
    for d in range(3):
        A = A.narrow(_axis(d), lo[d], hi[d] - lo[d])
    return A


def _two_level_stage(C, F, lo, hi, h, per, dt):
    """(C, F) + dt L with the fine fluxes on the coarse side of the box; lo, hi in coarse cells."""
    C = C.clone()
    _window(C, lo, hi).copy_(_mean(F, range(3)))
    wide = _window(C, [x - 2 for x in lo], [x + 2 for x in hi])
    P = _shrink(wide, 3, 1)
    for d in range(3):
        P = P.repeat_interleave(2, _axis(d))
    for d in range(3):
        q = wide
        for o in range(3):
            if o != d:
                q = _cut(q, o, 1, 1)
        dq = _cut(q, d, 1, 0) - _cut(q, d, 0, 1)
        s = 0.25 * _mc(_cut(dq, d, 0, 1), _cut(dq, d, 1, 0))
        shape = list(s.shape)
        ax = _axis(d)
        s = torch.stack([-s, s], ax + 1).reshape(shape[:ax] + [2 * shape[ax]] + shape[ax + 1:])
        for o in range(3):
            if o != d:
                s = s.repeat_interleave(2, _axis(o))
        P = P + s
    _shrink(P, 3, 2).copy_(F)
    RC, RF = 0.0, 0.0
    for d in range(3):
        Q = P
        for o in range(3):
            if o != d:
                Q = _cut(Q, o, 2, 2)
        ff = _flux(_primitive(Q), d)
        fc = _flux(_primitive(_pad(C, d, 2, per[d])), d)
        other = [o for o in range(3) if o != d]
        for end, at in ((0, lo[d]), (ff.shape[_axis(d)] - 1, hi[d])):
            face = _mean(ff.narrow(_axis(d), end, 1), other)
            l, u = list(lo), list(hi)
            l[d], u[d] = at, at + 1
            _window(fc, l, u).copy_(face)
        RC = RC - (_cut(fc, d, 1, 0) - _cut(fc, d, 0, 1)) / h
        RF = RF - (_cut(ff, d, 1, 0) - _cut(ff, d, 0, 1)) / (0.5 * h)
    return C, C + dt * RC, F + dt * RF


def _two_level(case, data):
    (C0, h), (F0, _) = data
    n = (case["n"], case["n"], case["nz"])
    lo, hi = ([b[d] * n[d] for d in range(3)] for b in _box(case))
    per = [b == "p" for b in case["bc"]]

    def leaf_dt(C, F):
        sc = _speed(C, 3, h).unsqueeze(0)
        _window(sc, lo, hi).zero_()
        return CFL / torch.maximum(sc.max(), _speed(F, 3, 0.5 * h).max())

    dt = leaf_dt(C0, F0)
    C0, C1, F1 = _two_level_stage(C0, F0, lo, hi, h, per, dt)
    _, C2, F2 = _two_level_stage(C1, F1, lo, hi, h, per, dt)
    C, F = 0.5 * C0 + 0.5 * C2, 0.5 * F0 + 0.5 * F2
    dt = leaf_dt(C, F)
    _window(C, lo, hi).copy_(_mean(F, range(3)))
    return {"U": torch.cat([_to_blocks(C, n), _to_blocks(F, n)]), "dt": dt.reshape(1)}


def exact(case, seed):
    data = _globals(case, seed, "cuda" if torch.cuda.is_available() else "cpu")
    n, nd, ng = (case["n"], case["n"], case["nz"]), case["ndim"], case["ng"]
    if case["path"] == "two_level":
        return _two_level(case, data)
    if case["path"] == "guards":
        (U, h), = data
        P = U
        for d in range(nd):
            P = _pad(P, d, ng, case["bc"][d] == "p")
        for d in range(nd):
            P = P.unfold(_axis(d), n[d] + 2 * ng, n[d])
        # [5, bz, by, bx, x, y, z] -> [blocks, 5, z, y, x]
        P = P.permute(1, 2, 3, 0, 6, 5, 4).reshape(-1, 5, n[2] + 2 * ng, n[1] + 2 * ng, n[0] + 2 * ng)
        return {"U": P, "dt": (CFL / _speed(U, nd, h).max()).reshape(1)}
    if case["path"] == "gradient":
        (W, h), = data
        g = torch.Generator(device=W.device).manual_seed(seed + 5)
        blocks = _to_blocks(W, n)
        gz = ng if nd == 3 else 0
        gU = torch.randn((blocks.shape[0], 5, n[2] + 2 * gz, n[1] + 2 * ng, n[0] + 2 * ng), generator=g,
                         dtype=torch.float64, device=W.device)
        W.requires_grad_(True)
        U = _conserved(W)
        for _ in range(case["steps"]):
            dt = CFL / _speed(U.detach(), nd, h).max()
            U = _step(U, dt, case, h)
        out = _to_blocks(U, n)
        (gW,) = torch.autograd.grad(out, W, _interior(gU, ng, nd).contiguous())
        return {"U": out.detach(), "gradient": _to_blocks(gW, n)}
    blocks, dts, hist = [], [], []
    for U, h in data:
        dt = CFL / _speed(U, nd, h).max()
        for _ in range(case["steps"]):
            hist.append(dt)
            U = _step(U, dt, case, h)
            dt = CFL / _speed(U, nd, h).max()
        blocks.append(_to_blocks(U, n))
        dts.append(dt)
    out = {"U": torch.cat(blocks), "dt": torch.stack(dts)}
    if case["path"] == "advance":
        out["history"] = torch.stack(hist)
    return out
