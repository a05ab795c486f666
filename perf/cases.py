"""Performance cases of the HDG library: what a solver built on it asks for at every Newton step.

A case names an operation on one mesh:

* ``linearize``  one Newton linearization: linearize + condense + assemble, the trace blocks and right-hand
  side, one trace matvec and the interior recovery (the library's core loop body);
* ``solve``      one linear solve of an assembled trace system: additive Schwarz set-up and GMRES;
* ``newton``     a whole Newton solve of one DIRK stage, state in, converged state out;
* ``step``       one SDIRK3 time step, captured as a CUDA graph and replayed.

The meshes and flows are those of the paper's evaluation in the sizes one GPU takes quickly: periodic quads with a
sinusoidal freestream, the Taylor-Green vortex on hexes (nearly incompressible, or at M = 1.25 with Sutherland's
law and artificial viscosity), a wall layer on graded hexes (isothermal wall, inflow, outflow), and curved
anisotropic tetrahedra of mixed degree over a bumped wall.  Everything is made here from the seed; nothing of it
comes from files.

``exact`` is the same mathematics in FP64 by another route: plain torch, pointwise fluxes differentiated by
forward-mode automatic differentiation, dense per-element solves, Krylov iterations taken to convergence.
"""
from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

from paper_2608_27863_gb300 import hdg as H

DEV = "cuda"
F64 = torch.float64
GAMMA = 1.4


# ----------------------------------------------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------------------------------------------
def _case(op, flow, p, nx, ny, nz, prec):
    return {"op": op, "flow": flow, "p": p, "nx": nx, "ny": ny, "nz": nz, "prec": prec}


def listed():
    def named(name, *a):
        return dict(_case(*a), name=name)

    return [
        # a small 2-D run: latency, launches and the serial pivot chain set the time
        named("quad-p2-8x8-fp64", "linearize", "wave", 2, 8, 8, 0, "fp64"),
        # an ordinary 2-D mesh in the fast form, odd sizes
        named("quad-p3-61x47-mixed", "linearize", "wave", 3, 61, 47, 0, "mixed"),
        # low order with walls, inflow and outflow (boundary rows, graded cells, Sutherland's law)
        named("hex-p1-11x9x7-wall-fp64", "linearize", "wall", 1, 11, 9, 7, "fp64"),
        # the Taylor-Green vortex at the paper's order, both precisions
        named("hex-p2-8x8x8-tgv-fp64", "linearize", "tgv", 2, 8, 8, 8, "fp64"),
        named("hex-p2-16x16x16-tgv-mixed", "linearize", "tgv", 2, 16, 16, 16, "mixed"),
        # the compressible vortex at p = 3 with shock capturing, both precisions
        named("hex-p3-7x6x5-shock-fp64", "linearize", "shock", 3, 7, 6, 5, "fp64"),
        named("hex-p3-12x11x10-shock-mixed", "linearize", "shock", 3, 12, 11, 10, "mixed"),
        # curved tetrahedra of degrees 1..4, both precisions (the bench's default workload, smaller)
        named("tet-p1to4-10x20x3-fp64", "linearize", "layer", 0, 10, 20, 3, "fp64"),
        named("tet-p1to4-10x20x6-mixed", "linearize", "layer", 0, 10, 20, 6, "mixed"),
        # the linear solver on the assembled tetrahedral system
        named("tet-p1to4-7x12x5-solve-mixed", "solve", "layer", 0, 7, 12, 5, "mixed"),
        # a whole Newton solve of a stage and a whole time step
        named("hex-p2-8x8x8-newton-mixed", "newton", "tgv", 2, 8, 8, 8, "mixed"),
        named("quad-p2-8x8-step-fp64", "step", "wave", 2, 8, 8, 0, "fp64"),
    ]


# elements that one linearization of a drawn case may have, by flow dimension and degree
_MOST = {("wave", 1): 12000, ("wave", 2): 6000, ("wave", 3): 3000, ("hex", 1): 8000, ("hex", 2): 2000, ("hex", 3): 500}


def draw(rng):
    op = rng.choice(("linearize",) * 7 + ("solve", "newton", "step"))
    prec = rng.choice(("fp64", "mixed"))
    if op == "step":
        return _case(op, "wave", rng.randint(1, 3), rng.randint(3, 14), rng.randint(3, 14), 0, "fp64")
    if op == "newton":
        n = [rng.randint(3, 9) for _ in range(3)]
        return _case(op, "tgv", rng.randint(1, 2), *n, prec)
    if op == "solve":
        return _case(op, "layer", 0, rng.randint(3, 8), rng.randint(3, 14), rng.randint(3, 5), prec)
    flow = rng.choice(("wave", "tgv", "shock", "wall", "layer"))
    if flow == "layer":
        return _case(op, flow, 0, rng.randint(3, 10), rng.randint(2, 20), rng.randint(3, 3 if prec == "fp64" else 6), prec)
    p = rng.randint(1, 3)
    dim = 2 if flow == "wave" else 3
    most = _MOST[("wave" if dim == 2 else "hex", p)] * (1 if prec == "fp64" else 2)
    e = math.exp(rng.uniform(math.log(3 ** dim), math.log(most)))
    side = e ** (1.0 / dim)
    n = [max(3, round(side * rng.uniform(0.75, 1.25))) for _ in range(dim)]
    while math.prod(n) > most:
        n[n.index(max(n))] -= 1
    return _case(op, flow, p, n[0], n[1], n[2] if dim == 3 else 0, prec)


# ----------------------------------------------------------------------------------------------------------------
# meshes (host arrays as the library takes them)
# ----------------------------------------------------------------------------------------------------------------
def _box(coords, periodic, tags):
    """Structured box of quads or hexes: vertices, element vertices, periodic masters, boundary tags."""
    d = len(coords)
    n = [len(c) - 1 for c in coords]
    nv = [k + 1 for k in n]
    strides = np.cumprod([1] + nv[:-1])
    ii = np.stack(np.unravel_index(np.arange(int(np.prod(nv))), nv, order="F"), axis=1)
    vert = np.stack([np.asarray(coords[r])[ii[:, r]] for r in range(d)], axis=1)
    jj = np.where(np.array(periodic) & (ii == np.array(n)), 0, ii)
    pmap = jj @ strides
    ei = np.stack(np.unravel_index(np.arange(int(np.prod(n))), n, order="F"), axis=1)
    corner = np.array([[(c >> r) & 1 for r in range(d)] for c in range(2 ** d)])
    ev = (ei[:, None, :] + corner[None]) @ strides
    tag = np.zeros((len(ei), 2 * d), np.int32)
    for (r, s), t in tags.items():
        tag[ei[:, r] == (0 if s == 0 else n[r] - 1), 2 * r + s] = t
    return {"dim": d, "vert": vert.astype(np.float64), "ev": ev.astype(np.int64), "pmap": pmap.astype(np.int64),
            "tag": tag}


def _graded(n, length, first):
    lo, hi = 1.0 + 1e-9, 4.0
    for _ in range(200):
        r = 0.5 * (lo + hi)
        lo, hi = (lo, r) if first * (r ** n - 1.0) / (r - 1.0) > length else (r, hi)
    x = np.concatenate([[0.0], np.cumsum(first * lo ** np.arange(n))])
    return x * (length / x[-1])


_EDGES = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))


def _bump(x):
    y = np.array(x, copy=True)
    y[..., 1] += 0.05 * np.sin(np.pi * x[..., 0]) * (1.0 - x[..., 1]) ** 2
    return y


def _layer(nx, ny, nz):
    """Kuhn tetrahedra over a bumped wall: x and z periodic, y graded from the wall by 1.2 (wall cell dx / 1000)."""
    dx = 1.0 / nx
    h1 = dx / 1e3
    ys = np.concatenate([[0.0], np.cumsum(h1 * 1.2 ** np.arange(ny))])
    b = _box([np.linspace(0, 1, nx + 1), ys, np.linspace(0, nz * dx, nz + 1)], (True, False, True), {})
    comp, ev8 = b["vert"], b["ev"]
    phys = _bump(comp)
    tets, corner = [], []
    for perm in itertools.permutations(range(3)):
        c = [0, 1 << perm[0], (1 << perm[0]) | (1 << perm[1]), 7]
        tets.append(ev8[:, c])
        corner.append(np.broadcast_to(np.array(c), (len(ev8), 4)))
    ev = np.stack(tets, axis=1).reshape(-1, 4)
    cs = np.stack(corner, axis=1).reshape(-1, 4).copy()
    X = phys[ev]
    flip = np.linalg.det(X[:, 1:] - X[:, :1]) < 0
    ev[flip] = ev[flip][:, [0, 2, 1, 3]]
    cs[flip] = cs[flip][:, [0, 2, 1, 3]]
    row = np.repeat(np.unravel_index(np.arange(len(ev8)), (nx, ny, nz), order="F")[1], 6)
    vrow = row[:, None] + ((cs >> 1) & 1)
    tag = np.zeros((len(ev), 4), np.int32)
    for f in range(4):
        loc = [v for v in range(4) if v != f]
        tag[np.all(vrow[:, loc] == 0, axis=1), f] = 4
        tag[np.all(vrow[:, loc] == ny, axis=1), f] = 1
    sag = 0.05 * np.pi ** 2 * dx * dx / 8.0
    curved_rows = next((j for j in range(ny) if h1 * 1.2 ** j >= 6.0 * sag), ny)
    geo = np.zeros((len(ev), 10, 3))
    geo[:, :4] = phys[ev]
    for c, (i, j) in enumerate(_EDGES):
        straight = 0.5 * (phys[ev[:, i]] + phys[ev[:, j]])
        bent = _bump(0.5 * (comp[ev[:, i]] + comp[ev[:, j]]))
        geo[:, 4 + c] = np.where((np.maximum(vrow[:, i], vrow[:, j]) <= curved_rows)[:, None], bent, straight)
    ep = (1 + np.random.default_rng(3).integers(0, 4, len(ev))).astype(np.int32)
    return {"dim": 3, "vert": phys, "ev": ev.astype(np.int64), "pmap": b["pmap"], "tag": tag, "ep": ep, "geo": geo}


@functools.lru_cache(maxsize=16)
def _mesh(flow, nx, ny, nz):
    if flow == "layer":
        return _layer(nx, ny, nz)
    if flow == "wave":
        return _box([np.linspace(0, 1, nx + 1), np.linspace(0, 1, ny + 1)], (True, True), {})
    if flow == "wall":
        return _box([np.linspace(0.1, 1.1, nx + 1), _graded(ny, 0.1, 0.02 / ny), np.linspace(0, 0.05, nz + 1)],
                    (False, False, True), {(0, 0): 1, (0, 1): 2, (1, 0): 3, (1, 1): 1})
    return _box([np.linspace(0, 2 * np.pi, k + 1) for k in (nx, ny, nz)], (True, True, True), {})


@functools.lru_cache(maxsize=16)
def _faces(flow, nx, ny, nz):
    """Global faces numbered by first encounter: e2f [E][nf], number of faces, the master ids of every face's corners."""
    m = _mesh(flow, nx, ny, nz)
    ids = m["pmap"][m["ev"]]
    d = m["dim"]
    if flow == "layer":
        corners = [[v for v in range(4) if v != f] for f in range(4)]
    else:
        corners = [[(f & 1) << (f >> 1) | sum(((c >> a) & 1) << k for a, k in enumerate(r for r in range(d) if r != f >> 1))
                    for c in range(2 ** (d - 1))] for f in range(2 * d)]
    fid = np.stack([ids[:, c] for c in corners], axis=1)
    key = np.sort(fid.reshape(-1, fid.shape[-1]), axis=1)
    _, first, inv = np.unique(key, axis=0, return_index=True, return_inverse=True)
    rank = np.empty(len(first), np.int64)
    rank[np.argsort(first)] = np.arange(len(first))
    return rank[inv.reshape(-1)].reshape(fid.shape[:2]), len(first), fid, corners


# ----------------------------------------------------------------------------------------------------------------
# physics and states
# ----------------------------------------------------------------------------------------------------------------
def _physics(case):
    flow, d = case["flow"], 2 if case["flow"] == "wave" else 3
    P = {"d": d, "re": 1600.0, "pr": 0.71, "mach": 0.1, "visc": 0, "c1": 1.4042, "s": 0.40417, "tau": 5.0,
         "tau_mode": 0, "dt": 1e-2, "a": 0.29, "tw": 1.0}
    if flow == "wave":
        P.update(re=100.0, pr=0.72, mach=0.3)
    elif flow == "shock":
        P.update(mach=1.25, visc=1)
    elif flow == "wall":
        t_aw = 1.0 + math.sqrt(0.72) * (GAMMA - 1.0) * 3.0 ** 2 / 2.0
        P.update(re=1e4, pr=0.72, mach=3.0, visc=1, s=110.4 / 51.86, c1=1.0 + 110.4 / 51.86, dt=1e-3, tau_mode=1,
                 tw=0.5 * t_aw)
    elif flow == "layer":
        P.update(re=1e5, pr=0.72, mach=0.5, dt=1e-3, a=0.4358665215, c1=1.0, s=0.0)
    vel = 0.0 if flow in ("tgv", "shock") else 1.0
    pres = 1.0 / (GAMMA * P["mach"] ** 2)
    P["ub"] = [1.0, vel] + [0.0] * (d - 1) + [pres / (GAMMA - 1.0) + 0.5 * vel]
    return P


def _conserved(rho, vel, pres):
    return torch.stack([rho] + [rho * v for v in vel] + [pres / (GAMMA - 1.0) + 0.5 * rho * sum(v * v for v in vel)], -1)


def _flow(case, P, r):
    """The state function x [..., d] -> u [..., m], with seeded phases r."""
    flow, mach = case["flow"], P["mach"]
    ub = torch.tensor(P["ub"], dtype=F64, device=DEV)
    p0 = 1.0 / (GAMMA * mach * mach)
    tau = 2 * math.pi

    def wave(x):
        u = ub.expand(x.shape[:-1] + (ub.numel(),)).clone()
        j = 1 if flow == "wave" else 2
        s = sum(torch.sin(tau * ((1 + k % 3) * x[..., 0] + (1 + k // 2) * x[..., j]) + tau * r[k]) for k in range(4))
        amp = 1e-2 if flow == "wave" else 1e-3
        for a in (0, 1, u.shape[-1] - 1):
            u[..., a] += amp * s
        return u

    def vortex(x):
        X, Y, Z = x[..., 0] + tau * r[0], x[..., 1] + tau * r[1], x[..., 2] + tau * r[2]
        pres = p0 + (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2.0) / 16.0
        return _conserved(GAMMA * mach * mach * pres, [torch.sin(X) * torch.cos(Y) * torch.cos(Z),
                                                      -torch.cos(X) * torch.sin(Y) * torch.cos(Z), 0.0 * Z], pres)

    def wall(x):
        y = x[..., 1] / 0.02
        prof = torch.tanh(y)
        T = P["tw"] + (1.0 - P["tw"]) * prof + 0.4 * prof * (1.0 - prof)
        vel = [prof, 0.0 * y, 0.0 * y]
        vel = [v + 1e-3 * y * torch.exp(-y) * torch.sin(tau * (x[..., 0] + 20 * x[..., 2] * (k > 0) + r[k]))
               for k, v in enumerate(vel)]
        return _conserved(1.0 / T, vel, p0 + 0.0 * y)

    return {"wave": wave, "layer": wave, "tgv": vortex, "shock": vortex, "wall": wall}[flow]


def _gll(p):
    a = {1: [], 2: [0.0], 3: [-math.sqrt(0.2), math.sqrt(0.2)]}[p]
    return np.array([-1.0] + a + [1.0])


def _tri_n(p):
    return (p + 1) * (p + 2) // 2


def _lattice(p):
    return np.array([(i, j, k) for k in range(p + 1) for j in range(p + 1 - k) for i in range(p + 1 - j - k)])


def _p2_shape(lam):
    """Quadratic tetrahedral shape functions [..., 10] at barycentric coordinates lam [..., 4]."""
    return torch.stack([lam[..., v] * (2 * lam[..., v] - 1) for v in range(4)] +
                       [4 * lam[..., a] * lam[..., b] for a, b in _EDGES], -1)


def _node_xyz(case, m):
    """Physical node positions: a tensor [E, Np, d], or for tetrahedra {degree: (elements, [n, Np, 3])}."""
    t = functools.partial(torch.as_tensor, device=DEV)
    if case["flow"] == "layer":
        out = {}
        for p in range(1, 5):
            idx = np.nonzero(m["ep"] == p)[0]
            l3 = t(_lattice(p) / p, dtype=F64)
            lam = torch.cat([1.0 - l3.sum(-1, keepdim=True), l3], -1)
            out[p] = (t(idx), torch.einsum("nc,eck->enk", _p2_shape(lam), t(m["geo"][idx])))
        return out
    d, p = m["dim"], case["p"]
    s = 0.5 * (_gll(p) + 1.0)
    jj = np.stack(np.unravel_index(np.arange((p + 1) ** d), (p + 1,) * d, order="F"), 1)
    w = np.ones((len(jj), 2 ** d))
    for c in range(2 ** d):
        for r in range(d):
            w[:, c] *= s[jj[:, r]] if (c >> r) & 1 else 1.0 - s[jj[:, r]]
    return torch.einsum("nc,ecx->enx", t(w), t(m["vert"][m["ev"]]))


def _gradient(fun, x, h=1e-5):
    d = x.shape[-1]
    eye = torch.eye(d, dtype=F64, device=DEV) * h
    return torch.stack([(fun(x + eye[k]) - fun(x - eye[k])) / (2 * h) for k in range(d)], -2)     # [..., d, m]


def _inputs(case, seed):
    """The state arrays of a case in the library's layouts, all on the GPU."""
    m, P = _mesh(case["flow"], case["nx"], case["ny"], case["nz"]), _physics(case)
    e2f, nF, _, _ = _faces(case["flow"], case["nx"], case["ny"], case["nz"])
    g = torch.Generator(device=DEV).manual_seed(int(seed))

    def noise(n):
        return torch.randn(n, generator=g, dtype=F64, device=DEV)

    r = torch.rand(8, generator=g, dtype=F64, device=DEV)
    fun = _flow(case, P, r)
    x = _node_xyz(case, m)
    ub = torch.tensor(P["ub"], dtype=F64, device=DEV)
    scale = ub.abs() + 1.0
    nu = None
    if case["flow"] == "layer":
        npe = (m["ep"] + 1) * (m["ep"] + 2) * (m["ep"] + 3) // 6
        off = np.concatenate([[0], np.cumsum(5 * npe)])
        U = torch.empty(int(off[-1]), dtype=F64, device=DEV)
        for p, (idx, xp) in x.items():
            u = fun(xp).transpose(1, 2).reshape(len(idx), -1)
            at = torch.as_tensor(off[:-1], device=DEV)[idx][:, None] + torch.arange(u.shape[1], device=DEV)
            U[at.reshape(-1)] = u.reshape(-1)
        U += 1e-4 * noise(U.shape)
        Q = 1e-2 * noise(3 * U.numel())
        fp = np.zeros(nF, np.int64)
        np.maximum.at(fp, e2f.reshape(-1), np.repeat(m["ep"], 4))
        nfp = torch.as_tensor((fp + 1) * (fp + 2) // 2, device=DEV)
        comp = torch.arange(5, device=DEV).repeat(nF).repeat_interleave(nfp.repeat_interleave(5))
        UH = ub[comp] + 1e-3 * scale[comp] * noise(comp.shape)
    else:
        u = fun(x)
        U = u.transpose(1, 2).contiguous()
        U += 1e-4 * noise(U.shape)
        Q = _gradient(fun, x).permute(0, 2, 3, 1).contiguous()
        shape = (nF, len(P["ub"]), (case["p"] + 1) ** (P["d"] - 1))
        UH = ub[None, :, None] + 1e-3 * scale[None, :, None] * noise(shape)
        if case["flow"] == "shock":
            nu = 2e-3 * (1.0 + 0.5 * torch.prod(torch.sin(x + 2 * math.pi * r[3:6]), -1)).contiguous()
    x1 = 1e-2 * noise(UH.shape) * (scale[comp] if case["flow"] == "layer" else scale[None, :, None])
    return m, P, {"U": U, "Q": Q.contiguous(), "UH": UH.contiguous(), "Us": U.clone(), "nu": nu, "x": x1.contiguous()}


# ----------------------------------------------------------------------------------------------------------------
# what a program has in hand, and one pass
# ----------------------------------------------------------------------------------------------------------------
class _Handle:
    """A library handle that goes when its owner does."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        if H is not None and self.h:
            H.hdg_destroy(self.h)
            self.h = None


#: Krylov settings of the whole calls
_SOLVE = {"restart": 120, "max_iter": 960, "rtol": 1e-8}
_NEWTON = {"tol": 1e-8, "max_newton": 10, "restart": 100, "max_gmres": 300, "gmres_rtol": 1e-6}
_STEP = {"n_newton": 4, "m": 40}


def prepare(case, seed):
    m, P, a = _inputs(case, seed)
    layer = case["flow"] == "layer"
    tag = m["tag"] if m["tag"].any() else None
    if layer:
        h = H.hdg_create_tet(m["vert"], m["ev"], m["pmap"], tag, m["ep"], m["geo"], GAMMA, P["re"], P["pr"], P["mach"])
    else:
        h = H.hdg_create(m["dim"], m["vert"], m["ev"], m["pmap"], tag, case["p"], GAMMA, P["re"], P["pr"], P["mach"])
    own = _Handle(h)
    H.hdg_set_params(h, tau=P["tau"], visc_law=P["visc"], suth_c1=P["c1"], suth_s=P["s"], tau_mode=P["tau_mode"],
                     precision=H.HDG_PREC_FP64 if case["prec"] == "fp64" else H.HDG_PREC_MIXED_3XTF32)
    H.hdg_set_stream(h, torch.cuda.current_stream().cuda_stream)
    if tag is not None and (tag == 1).any():
        H.hdg_set_bc_state(h, 1, np.array(P["ub"]))
    if tag is not None and (tag == 3).any():
        H.hdg_set_bc_state(h, 3, np.array([P["tw"]]))
    st = dict(a, case=case, own=own, P=P)
    if case["op"] == "linearize":
        if layer:
            n = H.hdg_tet_query(h)["n_vals"]
        else:
            s = H.hdg_query_sizes(h)
            n = s["nnzb"] * s["block"] ** 2
        st["S"] = torch.empty(n, dtype=F64 if case["prec"] == "fp64" else torch.float32, device=DEV)
        st["g"], st["y"] = torch.empty_like(a["UH"]), torch.empty_like(a["UH"])
        st["dQ"], st["dU"] = torch.empty_like(a["Q"]), torch.empty_like(a["U"])
    elif case["op"] == "solve":
        H.hdg_set_preconditioner(h, H.HDG_PC_SCHWARZ)
        H.hdg_linearize_condense(h, a["U"], a["Q"], a["UH"], a["Us"], a["nu"], P["dt"], P["a"])
        st["g"], st["sol"] = torch.empty_like(a["UH"]), torch.empty_like(a["UH"])
        H.hdg_trace_rhs(h, st["g"])
    else:
        if case["op"] == "newton":
            H.hdg_set_preconditioner(h, H.HDG_PC_SCHWARZ)
        st["W"] = [torch.empty_like(a[k]) for k in ("U", "Q", "UH")]
    return st


def run(state):
    case, h, P = state["case"], state["own"].h, state["P"]
    if case["op"] == "linearize":
        H.hdg_linearize_condense(h, state["U"], state["Q"], state["UH"], state["Us"], state["nu"], P["dt"], P["a"])
        H.hdg_get_blocks(h, state["S"])
        H.hdg_trace_rhs(h, state["g"])
        H.hdg_trace_matvec(h, state["x"], state["y"])
        H.hdg_recover_interior(h, state["x"], state["dQ"], state["dU"])
        return {k: state[k] for k in ("S", "g", "y", "dQ", "dU")}
    if case["op"] == "solve":
        H.hdg_schwarz_setup(h)
        state["sol"].zero_()
        H.hdg_gmres(h, state["g"], state["sol"], **_SOLVE)
        return {"x": state["sol"]}
    U, Q, UH = state["W"]
    for w, k in zip((U, Q, UH), ("U", "Q", "UH")):
        w.copy_(state[k])
    if case["op"] == "newton":
        H.hdg_newton(h, U, Q, UH, state["Us"], state["nu"], P["dt"], P["a"], raise_on_noconv=False, **_NEWTON)
    else:
        H.hdg_dirk_step(h, U, Q, UH, state["nu"], P["dt"], **_STEP)
    return {"U": U, "Q": Q, "UH": UH}


# ----------------------------------------------------------------------------------------------------------------
# work and tolerance
# ----------------------------------------------------------------------------------------------------------------
def _sizes(case):
    """Per element class (count, n_u, t, columns of the contraction, points): and the trace blocks' values."""
    m = _mesh(case["flow"], case["nx"], case["ny"], case["nz"])
    e2f, nF, _, _ = _faces(case["flow"], case["nx"], case["ny"], case["nz"])
    d = m["dim"]
    mm = d + 2
    E, nf = e2f.shape
    if case["flow"] == "layer":
        fp = np.zeros(nF, np.int64)
        np.maximum.at(fp, e2f.reshape(-1), np.repeat(m["ep"], nf))
        bs = mm * (fp + 1) * (fp + 2) // 2
        nu = mm * (m["ep"] + 1) * (m["ep"] + 2) * (m["ep"] + 3) // 6
    else:
        bs = np.full(nF, mm * (case["p"] + 1) ** (d - 1))
        nu = np.full(E, mm * (case["p"] + 1) ** d)
    t = bs[e2f].sum(1)
    pair = (e2f[:, :, None] * nF + e2f[:, None, :]).reshape(-1)
    key = np.unique(pair)
    return nu.astype(float), t.astype(float), float(bs.sum()), float((bs[key // nF] * bs[key % nF]).sum()), d


def work(case):
    """Inputs and outputs moved once; the arithmetic of the condensation (interior LU, two triangular solves, Schur
    product) once per linearization.  Newton and time steps: three linearizations, and one per stage."""
    nu, t, nt, nv, d = _sizes(case)
    width = 8.0 if case["prec"] == "fp64" else 4.0
    lin = float((2.0 / 3.0 * nu ** 3 + 2.0 * nu ** 2 * t + 2.0 * t ** 2 * nu).sum())
    state = 8.0 * (nu.sum() * (2 + d) + nt)
    if case["op"] == "linearize":
        return {"bytes": state + width * nv + 8.0 * (nu.sum() * (1 + d) + 3 * nt), "flops": lin}
    if case["op"] == "solve":
        return {"bytes": width * nv + 16.0 * nt, "flops": float((2.0 / 3.0 * t ** 3).sum())}
    k = 3.0
    return {"bytes": 2 * state + k * width * nv, "flops": k * lin}


def tolerance(case):
    """About four times the largest error against ``exact`` that the cases and draws showed: FP64 blocks and
    corrections to 2e-12, the mixed form's to 9e-6 (5e-5 through a linear solve), Newton and time steps as far as
    the stage residual is driven (2e-9 and 8e-12)."""
    fp64 = case["prec"] == "fp64"
    if case["op"] == "linearize":
        return {"rel": 1e-11, "max": 1e-8} if fp64 else {"rel": 4e-5, "max": 1e-2}
    if case["op"] == "solve":
        return {"rel": 1e-6, "max": 1e-4} if fp64 else {"rel": 3e-4, "max": 3e-2}
    return {"rel": 2e-8, "max": 1e-6} if case["op"] == "newton" else {"rel": 1e-9, "max": 1e-7}


# ----------------------------------------------------------------------------------------------------------------
# the same in plain torch, FP64
# ----------------------------------------------------------------------------------------------------------------
def _flux(u, q, nu, P):
    """F^c - F^v at one point: u [m], q [m, d] (q[a, k] = d u_a / d x_k) -> [m, d]."""
    d = q.shape[1]
    rho, v, E = u[0], u[1:d + 1] / u[0], u[d + 1] / u[0]
    pres = (GAMMA - 1.0) * (u[d + 1] - 0.5 * rho * (v * v).sum())
    eye = torch.eye(d, dtype=u.dtype, device=u.device)
    Fc = torch.cat([(rho * v)[None], rho * v[:, None] * v[None] + pres * eye, ((u[d + 1] + pres) * v)[None]])
    mu = torch.ones_like(rho) / P["re"]
    if P["visc"]:
        T = GAMMA * P["mach"] ** 2 * pres / rho
        mu = P["c1"] * T ** 1.5 / (T + P["s"]) / P["re"]
    dv = (q[1:d + 1] - v[:, None] * q[0][None]) / rho
    de = (q[d + 1] - E * q[0]) / rho - v @ dv
    tau = mu * (dv + dv.T - (2.0 / 3.0) * torch.trace(dv) * eye)
    Fv = torch.cat([torch.zeros_like(q[:1]), tau, (v @ tau + GAMMA * mu / P["pr"] * de)[None]]) + nu * q
    return Fc - Fv


def _face_terms(u, uh, q, nu, nw, hk, tag, P):
    """(fhat, bhat) at one face point, both times w |J|: nw is the weighted outward normal."""
    d = q.shape[1]
    nrm = torch.sqrt((nw * nw).sum())
    live = nrm > 0
    n = nw / torch.where(live, nrm, torch.ones_like(nrm))
    tau = P["tau"] * torch.ones_like(nrm)
    if P["tau_mode"]:
        rho, v = uh[0], uh[1:d + 1] / uh[0]
        pres = (GAMMA - 1.0) * (uh[d + 1] - 0.5 * rho * (v * v).sum())
        mu = torch.ones_like(rho) / P["re"]
        if P["visc"]:
            T = GAMMA * P["mach"] ** 2 * pres / rho
            mu = P["c1"] * T ** 1.5 / (T + P["s"]) / P["re"]
        tau = torch.abs(v @ n) + torch.sqrt(GAMMA * pres / rho) + mu / hk
    f = _flux(uh, q, nu, P) @ nw + nrm * tau * (u - uh)
    ub = torch.tensor(P["ub"], dtype=u.dtype, device=u.device)
    ew = P["tw"] / (GAMMA * (GAMMA - 1.0) * P["mach"] ** 2)
    wall = torch.cat([f[:1], nrm * uh[1:d + 1]])
    b = torch.where(tag == 1, nrm * (uh - ub), f)
    b = torch.where(tag == 2, nrm * (uh - u), b)
    b = torch.where(tag == 3, torch.cat([wall, (nrm * (uh[d + 1] - uh[0] * ew))[None]]), b)
    b = torch.where(tag == 4, torch.cat([wall, f[d + 1:]]), b)
    return f, b


def _lagrange(nodes, x):
    """Values and derivatives [..., n] of the 1-D Lagrange basis at x [...]."""
    n = len(nodes)
    val, der = [], []
    for j in range(n):
        k = [i for i in range(n) if i != j]
        f = [(x - nodes[i]) / (nodes[j] - nodes[i]) for i in k]
        val.append(functools.reduce(torch.mul, f, torch.ones_like(x)))
        der.append(sum(functools.reduce(torch.mul, [f[b] for b in range(n - 1) if b != a], torch.ones_like(x)) /
                       (nodes[j] - nodes[k[a]]) for a in range(n - 1)))
    return torch.stack(val, -1), torch.stack(der, -1)


def _tensor_basis(p, x, grad=False):
    """Tensor Gauss-Lobatto basis at x [..., d], first direction fastest; with grad, the derivatives [..., d, Np]."""
    d = x.shape[-1]
    vd = [_lagrange(_gll(p), x[..., r]) for r in range(d)]

    def prod(tabs):
        out = tabs[0]
        for t in tabs[1:]:
            out = (t[..., :, None] * out[..., None, :]).flatten(-2)
        return out

    if not grad:
        return prod([v for v, _ in vd])
    return torch.stack([prod([vd[r][1] if r == k else vd[r][0] for r in range(d)]) for k in range(d)], -2)


def _simplex_basis(p, x, grad=False):
    """Lagrange basis of the equispaced lattice of degree p at barycentric tails x [..., dim]."""
    dim = x.shape[-1]
    ex = _lattice(p)
    ex = ex if dim == 3 else ex[ex[:, 2] == 0][:, :2]
    nodes = torch.as_tensor(ex / p, dtype=F64, device=x.device)

    def mono(y, e):
        return functools.reduce(torch.mul, [torch.stack([y[..., r] ** int(k) for k in e[:, r]], -1) for r in range(dim)])

    inv = torch.linalg.inv(mono(nodes, ex))
    if not grad:
        return mono(x, ex) @ inv
    out = []
    for r in range(dim):
        e = ex.copy()
        e[:, r] = np.maximum(e[:, r] - 1, 0)
        out.append((mono(x, e) * torch.as_tensor(ex[:, r], dtype=F64, device=x.device)) @ inv)
    return torch.stack(out, -2)


def _jacobi_rule(n, alpha):
    """Gauss rule of weight (1 - x)^alpha on [-1, 1], mapped to [0, 1] with weight (1 - s)^alpha."""
    k = np.arange(n)
    a = np.where(2 * k + alpha == 0, -alpha / (alpha + 2.0), -alpha ** 2 / np.maximum((2 * k + alpha) * (2 * k + alpha + 2.0), 1e-300))
    if alpha == 0:
        a = np.zeros(n)
    k = np.arange(1, n)
    s = 2 * k + alpha
    b = 4.0 * k ** 2 * (k + alpha) ** 2 / (s ** 2 * (s + 1.0) * (s - 1.0))
    w, v = np.linalg.eigh(np.diag(a) + np.diag(np.sqrt(b), 1) + np.diag(np.sqrt(b), -1))
    return 0.5 * (w + 1.0), v[0] ** 2 / (alpha + 1.0)


def _simplex_rule(n, dim):
    """Collapsed rule on the unit simplex: barycentric tails [n^dim, dim] and weights."""
    (a, wa), (b, wb), (c, wc) = (_jacobi_rule(n, k) for k in range(3))
    if dim == 2:
        B, A = (t.reshape(-1) for t in np.meshgrid(b, a, indexing="ij"))
        return np.stack([A * (1 - B), B], 1), np.outer(wb, wa).reshape(-1)
    C, B, A = (t.reshape(-1) for t in np.meshgrid(c, b, a, indexing="ij"))
    return np.stack([A * (1 - B) * (1 - C), B * (1 - C), C], 1), np.einsum("i,j,k->ijk", wc, wb, wa).reshape(-1)


class _Disc:
    """The discretization of a case as batched tables: groups of elements of one degree, faces padded to one size."""

    def __init__(self, case):
        self.case = case
        self.P = _physics(case)
        m = self.m = _mesh(case["flow"], case["nx"], case["ny"], case["nz"])
        e2f, self.nF, fid, corners = _faces(case["flow"], case["nx"], case["ny"], case["nz"])
        self.tet = case["flow"] == "layer"
        d, E, nf = m["dim"], *e2f.shape
        self.d, self.mm, self.nf = d, d + 2, nf
        t = self.t = functools.partial(torch.as_tensor, device=DEV)
        if self.tet:
            fp = np.zeros(self.nF, np.int64)
            np.maximum.at(fp, e2f.reshape(-1), np.repeat(m["ep"], nf))
            nfp = (fp + 1) * (fp + 2) // 2
        else:
            fp = np.full(self.nF, case["p"])
            nfp = np.full(self.nF, (case["p"] + 1) ** (d - 1))
        self.L, bs = int(nfp.max()), self.mm * nfp
        hoff = np.concatenate([[0], np.cumsum(bs)])
        # padded trace vectors [nF, m, L] <-> the library's packed ones
        lab = np.arange(self.L)
        at = hoff[:-1, None, None] + np.arange(self.mm)[None, :, None] * nfp[:, None, None] + lab
        self.live = t(np.broadcast_to(lab < nfp[:, None, None], at.shape).copy())
        self.pos = t(np.where(lab < nfp[:, None, None], at, 0))
        self.e2f = t(e2f)
        # block pattern: (row face, column face) sorted, values column-major per block
        pair = (e2f[:, :, None] * self.nF + e2f[:, None, :]).reshape(-1)
        key, inv = np.unique(pair, return_inverse=True)
        boff = np.concatenate([[0], np.cumsum(bs[key // self.nF] * bs[key % self.nF])])
        self.nvals = int(boff[-1])
        self.boff = t(boff[:-1][inv.reshape(-1)].reshape(E, nf, nf))
        self.nfp = t(nfp)
        npe = (m["ep"] + 1) * (m["ep"] + 2) * (m["ep"] + 3) // 6 if self.tet else np.full(E, (case["p"] + 1) ** d)
        self.uoff = np.concatenate([[0], np.cumsum(self.mm * npe)])
        self.groups = [self._group(p, np.nonzero(m["ep"] == p)[0], fp, fid, corners) for p in range(1, 5)
                       if (m["ep"] == p).any()] if self.tet else [self._group(case["p"], np.arange(E), fp, fid, corners)]

    def _group(self, p, idx, fp, fid, corners):
        """Tables of the elements idx (all of degree p), in chunks."""
        t, d, m = self.t, self.d, self.m
        chunk = max(1, int(3e9 / (8.0 * ((p + 2) ** d * self.mm ** 2 * d * (p + 1) ** d * 6 + 1e4))))
        out = []
        for c0 in range(0, len(idx), chunk):
            ii = idx[c0:c0 + chunk]
            G = {"idx": t(ii), "n": len(ii)}
            if self.tet:
                xq, wq = _simplex_rule(p + 2, 3)
                xq = t(xq)
                G["phi"], dphi = _simplex_basis(p, xq), _simplex_basis(p, xq, True)
                geo = t(m["geo"][ii])

                def jac(x):
                    x = x.expand(len(ii), -1, -1)
                    lam = torch.cat([1 - x.sum(-1, keepdim=True), x], -1)
                    dl = torch.cat([-torch.ones(1, 3, dtype=F64, device=DEV), torch.eye(3, dtype=F64, device=DEV)])
                    dN = torch.stack([(4 * lam[..., v, None] - 1) * dl[v] for v in range(4)] +
                                     [4 * (lam[..., a, None] * dl[b] + lam[..., b, None] * dl[a]) for a, b in _EDGES], -2)
                    return torch.einsum("ngcr,nck->ngkr", dN, geo)

                verts = np.concatenate([np.zeros((1, 3)), np.eye(3)])
            else:
                x1, w1 = _jacobi_rule(p + 2, 0)
                gi = np.stack(np.unravel_index(np.arange((p + 2) ** d), (p + 2,) * d, order="F"), 1)
                xq, wq = t(2 * x1[gi] - 1), np.prod(2 * w1[gi], 1)
                G["phi"], dphi = _tensor_basis(p, xq), _tensor_basis(p, xq, True)
                X = m["vert"][m["ev"][ii]]
                J = t(np.stack([(X[:, 1 << r] - X[:, 0]) / 2 for r in range(d)], -1))          # [n, k, r]

                def jac(x):
                    return J[:, None].expand(len(ii), x.shape[-2], d, d)

                verts = np.array([[2.0 * ((c >> r) & 1) - 1 for r in range(d)] for c in range(2 ** d)])
            Jq = jac(xq)
            Ji = torch.linalg.inv(Jq)
            G["W"] = t(wq) * torch.linalg.det(Jq)
            G["dphi"] = torch.einsum("ngrk,gri->ngik", Ji, dphi)
            G["hk"] = G["W"].sum(1) ** (1.0 / d)
            # faces: points, trace basis and weighted normals in the face's canonical frame
            ids = fid[ii]
            nq = max((int(q) + 2) for q in fp) ** (d - 1)
            n = len(ii)
            phif = torch.zeros(n, self.nf, nq, G["phi"].shape[1], dtype=F64, device=DEV)
            mu = torch.zeros(n, self.nf, nq, self.L, dtype=F64, device=DEV)
            nw = torch.zeros(n, self.nf, nq, d, dtype=F64, device=DEV)
            centre = verts.mean(0)
            for f in range(self.nf):
                c = np.array(corners[f])
                if self.tet:
                    frame = c[np.argsort(ids[:, f], axis=1)]                                    # origin, then the axes' ends
                elif d == 2:
                    frame = c[np.argsort(ids[:, f], axis=1)]
                else:
                    o = np.argmin(ids[:, f], axis=1)
                    nb = np.stack([o ^ 1, o ^ 2], 1)
                    first = np.argmin(np.take_along_axis(ids[:, f], nb, 1), axis=1)
                    frame = c[np.stack([o, nb[np.arange(n), first], nb[np.arange(n), 1 - first]], 1)]
                V = verts[frame]                                                                # [n, d, d]
                ax = V[:, 1:] - V[:, :1]
                if d == 3:
                    area = np.cross(ax[:, 0], ax[:, 1])
                else:
                    area = np.stack([ax[:, 0, 1], -ax[:, 0, 0]], 1)
                out_dir = verts[c].mean(0) - centre
                area *= np.sign(area @ out_dir)[:, None]
                for q in np.unique(fp[self.e2f[t(ii), f].cpu().numpy()]):
                    sel = np.nonzero(fp[self.e2f[t(ii), f].cpu().numpy()] == q)[0]
                    if self.tet:
                        xs, ws = _simplex_rule(int(q) + 2, 2)
                        tb = _simplex_basis(int(q), t(xs))
                    else:
                        x1, w1 = _jacobi_rule(p + 2, 0)
                        gi = np.stack(np.unravel_index(np.arange((p + 2) ** (d - 1)), (p + 2,) * (d - 1), order="F"), 1)
                        xs, ws = x1[gi], np.prod(w1[gi], 1)
                        tb = _tensor_basis(p, t(2 * xs - 1))
                    x = t(V[sel][:, None, 0] + np.einsum("sa,nak->nsk", xs, ax[sel]))
                    s = t(sel)
                    full = torch.zeros(n, len(ws), d, dtype=F64, device=DEV)
                    full[s] = x
                    Jf = jac(full)[s]
                    nws = torch.einsum("nsrk,nr->nsk", torch.linalg.inv(Jf), t(area[sel])) * (t(ws) * torch.linalg.det(Jf))[..., None]
                    basis = _simplex_basis(p, x) if self.tet else _tensor_basis(p, x)
                    phif[s, f, :len(ws)] = basis
                    mu[s, f, :len(ws), :tb.shape[1]] = tb
                    nw[s, f, :len(ws)] = nws
                    # padded points: weight zero, at a valid place so that the state there is admissible
                    phif[s, f, len(ws):] = basis[:, :1]
                    mu[s, f, len(ws):, :tb.shape[1]] = tb[:1]
            G.update(phif=phif, mu=mu, nw=nw, tag=t(m["tag"][ii].astype(np.int64)))
            M = torch.einsum("ng,gi,gj->nij", G["W"], G["phi"], G["phi"])
            G["M"] = M
            E_ = torch.einsum("ng,ngik,gj->nkij", G["W"], G["dphi"], G["phi"])
            B_ = -torch.einsum("nfsi,nfsl,nfsk->nkifl", phif, mu, nw).flatten(3)
            G["G"] = torch.linalg.solve(M[:, None], E_)                                          # q = -G u - H uh
            G["H"] = torch.linalg.solve(M[:, None], B_)
            off = t(self.uoff)[G["idx"]]
            G["u_at"] = off[:, None, None] + (torch.arange(self.mm * G["phi"].shape[1], device=DEV)).reshape(1, self.mm, -1)
            G["q_at"] = d * off[:, None, None, None] + torch.arange(d * self.mm * G["phi"].shape[1], device=DEV).reshape(1, d, self.mm, -1)
            out.append(G)
        return out

    def chunks(self):
        return (G for g in self.groups for G in g)

    def pad(self, x):
        return x.reshape(-1)[self.pos] * self.live

    def unpad(self, x, like):
        out = torch.empty(like.numel(), dtype=F64, device=DEV)
        out[self.pos[self.live]] = x[self.live]
        return out.reshape(like.shape)

    def condense(self, G, a, dt, aii):
        """S^K, g^K in padded element trace order, and (X, y) with dU = -y - X duh, q_lift - q, for one chunk."""
        P, mm, d, L, n = self.P, self.mm, self.d, self.L, G["n"]
        U, Q, Us = a["U"].reshape(-1)[G["u_at"]], a["Q"].reshape(-1)[G["q_at"]], a["Us"].reshape(-1)[G["u_at"]]
        uh = self.pad(a["UH"])[self.e2f[G["idx"]]]                                               # [n, f, m, L]
        phi, W, dphi, phif, mu, nw = (G[k] for k in ("phi", "W", "dphi", "phif", "mu", "nw"))
        Np, T = phi.shape[1], self.nf * L
        uht = uh.transpose(1, 2).reshape(n, mm, T)
        ql = -torch.einsum("nkij,naj->nkai", G["G"], U) - torch.einsum("nkic,nac->nkai", G["H"], uht)
        vm = torch.func.vmap
        nug = torch.zeros(n, phi.shape[0], dtype=F64, device=DEV)
        nuf = torch.zeros(phif.shape[:3], dtype=F64, device=DEV)
        if a["nu"] is not None:
            nun = a["nu"][G["idx"]]
            nug, nuf = nun @ phi.T, torch.einsum("nfsi,ni->nfs", phif, nun)
        # volume
        u = torch.einsum("gi,nai->nga", phi, U).reshape(-1, mm)
        q = torch.einsum("gi,nkai->ngak", phi, Q).reshape(-1, mm, d)
        fl = lambda u_, q_, v_: _flux(u_, q_, v_, P)
        F = vm(fl)(u, torch.einsum("gi,nkai->ngak", phi, ql).reshape(-1, mm, d), nug.reshape(-1)).reshape(n, -1, mm, d)
        Fu, Fq = (j.reshape((n, -1) + j.shape[1:]) for j in vm(torch.func.jacfwd(fl, (0, 1)))(u, q, nug.reshape(-1)))
        # columns: q varies by -G (u columns) and -H (trace columns)
        psi = torch.cat([torch.einsum("gi,nkij->ngkj", phi, G["G"]), torch.einsum("gi,nkic->ngkc", phi, G["H"])], -1)
        col = -torch.einsum("ngakbl,nglc->ngakbc", Fq, psi)
        col[..., :Np] += Fu[..., None] * phi[None, :, None, None, None]
        R = torch.einsum("ng,ngik->ngki", W, dphi)
        A = -dt * torch.einsum("ngki,ngakbc->naibc", R, col)
        ru = -dt * torch.einsum("ngki,ngak->nai", R, F) + torch.einsum("nij,naj->nai", G["M"], U - Us) / aii
        for c in range(mm):
            A[:, c, :, c, :Np] += G["M"] / aii
        del col, Fu, Fq, psi
        # faces
        nS = phif.shape[2]
        us = torch.einsum("nfsi,nai->nfsa", phif, U).reshape(-1, mm)
        uhs = torch.einsum("nfsl,nfal->nfsa", mu, uh).reshape(-1, mm)
        qs = torch.einsum("nfsi,nkai->nfsak", phif, Q).reshape(-1, mm, d)
        qls = torch.einsum("nfsi,nkai->nfsak", phif, ql).reshape(-1, mm, d)
        rest = (nuf.reshape(-1), nw.reshape(-1, d), G["hk"][:, None, None].expand(nuf.shape).reshape(-1),
                G["tag"][:, :, None].expand(nuf.shape).reshape(-1))
        ft = lambda u_, h_, q_, *r: _face_terms(u_, h_, q_, *r, P)
        f, b = (v.reshape(n, self.nf, nS, mm) for v in vm(ft)(us, uhs, qls, *rest))
        Jf, Jb = vm(torch.func.jacfwd(ft, (0, 1, 2)))(us, uhs, qs, *rest)
        psif = torch.cat([torch.einsum("nfsi,nkij->nfskj", phif, G["G"]), torch.einsum("nfsi,nkic->nfskc", phif, G["H"])], -1)
        rows = []
        for J in (Jf, Jb):
            ju, jh, jq = (j.reshape((n, self.nf, nS) + j.shape[1:]) for j in J)
            c = -torch.einsum("nfsabl,nfslc->nfsabc", jq, psif)
            c[..., :Np] += ju[..., None] * phif[:, :, :, None, None]
            for k in range(self.nf):
                c[:, k, ..., Np + k * L:Np + (k + 1) * L] += jh[:, k, ..., None] * mu[:, k, :, None, None]
            rows.append(c)
        A += dt * torch.einsum("nfsi,nfsabc->naibc", phif, rows[0])
        ru += dt * torch.einsum("nfsi,nfsa->nai", phif, f)
        C = torch.einsum("nfsl,nfsabc->nfalbc", mu, rows[1])
        rh = torch.einsum("nfsl,nfsa->nfal", mu, b)
        # order: u columns (b, j), trace columns (f, b, l)
        Au = A[..., :Np].reshape(n, mm * Np, mm * Np)
        B = A[..., Np:].reshape(n, mm, Np, mm, self.nf, L).transpose(3, 4).reshape(n, mm * Np, -1)
        Cu = C[..., :Np].reshape(n, -1, mm * Np)
        D = C[..., Np:].reshape(n, self.nf, mm, L, mm, self.nf, L).transpose(4, 5).reshape(n, self.nf * mm * L, -1)
        sol = torch.linalg.solve(Au, torch.cat([B, ru.reshape(n, -1, 1)], -1))
        X, y = sol[..., :-1], sol[..., -1]
        S = D - Cu @ X
        g = -rh.reshape(n, -1) + torch.einsum("nrc,nc->nr", Cu, y)
        return S, g, X, y, ql - Q

    def recover(self, G, X, y, dq0, dx):
        """dU, dQ of one chunk for the padded trace correction dx."""
        n, mm = G["n"], self.mm
        duh = dx[self.e2f[G["idx"]]]
        dU = (-y - torch.einsum("nrc,nc->nr", X, duh.reshape(n, -1))).reshape(n, mm, -1)
        dt_ = duh.transpose(1, 2).reshape(n, mm, -1)
        dQ = dq0 - torch.einsum("nkij,naj->nkai", G["G"], dU) - torch.einsum("nkic,nac->nkai", G["H"], dt_)
        return dU, dQ

    def scatter(self, G, v, out):
        return out.index_add_(0, self.e2f[G["idx"]].reshape(-1), v.reshape(-1, self.mm, self.L))

    def block_index(self, G):
        """Position of every entry of S^K in the block values, -1 for padding."""
        mm, L, nf = self.mm, self.L, self.nf
        k = self.nfp[self.e2f[G["idx"]]]                                                         # [n, f]
        a, l = torch.arange(mm, device=DEV), torch.arange(L, device=DEV)
        loc = a[None, None, :, None] * k[:, :, None, None] + l                                   # [n, f, m, L]
        ok = (l < k[:, :, None, None]).expand(loc.shape)
        bF = (mm * k)[:, :, None, None, None, None, None]
        at = self.boff[G["idx"]][:, :, None, None, :, None, None] + loc[:, None, None, None] * bF + loc[:, :, :, :, None, None, None]
        return torch.where(ok[:, :, :, :, None, None, None] & ok[:, None, None, None], at, -1).reshape(G["n"], nf * mm * L, -1)


class _System:
    """An assembled trace system kept by elements: matvec, block-Jacobi GMRES, recovery."""

    def __init__(self, D, a, dt, aii):
        self.D, self.parts = D, []
        bs = D.mm * D.L
        self.g = torch.zeros(D.nF, D.mm, D.L, dtype=F64, device=DEV)
        diag = torch.zeros(D.nF, bs, bs, dtype=F64, device=DEV)
        for G in D.chunks():
            S, g, X, y, dq0 = D.condense(G, a, dt, aii)
            D.scatter(G, g, self.g)
            for f in range(D.nf):
                diag.index_add_(0, D.e2f[G["idx"], f], S[:, f * bs:(f + 1) * bs, f * bs:(f + 1) * bs])
            self.parts.append((G, S, X, y, dq0))
        dead = (~D.live).reshape(D.nF, bs)
        diag += torch.diag_embed(dead.to(F64))
        self.inv = torch.linalg.inv(diag)

    def matvec(self, x):
        D = self.D
        out = torch.zeros_like(x)
        for G, S, *_ in self.parts:
            D.scatter(G, torch.einsum("nrc,nc->nr", S, x[D.e2f[G["idx"]]].reshape(G["n"], -1)), out)
        return out

    def solve(self, rtol=1e-12, m=400, cycles=6):
        shape = self.g.shape
        pre = lambda v: (self.inv @ v.reshape(shape[0], -1, 1)).reshape(-1)
        x = torch.zeros_like(self.g).reshape(-1)
        b0 = float(pre(self.g).norm())
        for _ in range(cycles):
            r = pre(self.g - self.matvec(x.reshape(shape)))
            beta = float(r.norm())
            if beta <= rtol * b0:
                break
            V = torch.empty(m + 1, r.numel(), dtype=F64, device=DEV)
            Hm = np.zeros((m + 1, m))
            V[0] = r / beta
            y = None
            for k in range(m):
                w = pre(self.matvec(V[k].reshape(shape)))
                h = torch.zeros(k + 1, dtype=F64, device=DEV)
                for _ in range(2):
                    c = V[:k + 1] @ w
                    w = w - c @ V[:k + 1]
                    h += c
                hn = float(w.norm())
                Hm[:k + 1, k], Hm[k + 1, k] = h.cpu().numpy(), hn
                V[k + 1] = w / max(hn, 1e-300)
                if k % 20 == 19 or k == m - 1 or hn < 1e-14 * beta:
                    e = np.zeros(k + 2)
                    e[0] = beta
                    y = np.linalg.lstsq(Hm[:k + 2, :k + 1], e, rcond=None)[0]
                    if np.linalg.norm(Hm[:k + 2, :k + 1] @ y - e) <= 0.3 * rtol * b0:
                        break
            x = x + torch.as_tensor(y, device=DEV) @ V[:len(y)]
        return x.reshape(shape)


def _newton_exact(D, a, dt, aii, iters):
    for _ in range(iters):
        s = _System(D, a, dt, aii)
        dx = s.solve()
        U, Q = a["U"].reshape(-1).clone(), a["Q"].reshape(-1).clone()
        for G, S, X, y, dq0 in s.parts:
            dU, dQ = D.recover(G, X, y, dq0, dx)
            U[G["u_at"].reshape(-1)] += dU.reshape(-1)
            Q[G["q_at"].reshape(-1)] += dQ.reshape(-1)
        a = dict(a, U=U.reshape(a["U"].shape), Q=Q.reshape(a["Q"].shape), UH=a["UH"] + D.unpad(dx, a["UH"]))
    return a


def _sdirk3():
    """Alexander's three-stage, third-order, stiffly accurate SDIRK."""
    g = next(float(r.real) for r in np.roots([1.0, -3.0, 1.5, -1.0 / 6.0]) if 1.0 / 3.0 < r.real < 0.5)
    return np.array([[g, 0.0, 0.0], [(1.0 - g) / 2.0, g, 0.0],
                     [-(6 * g * g - 16 * g + 1) / 4.0, (6 * g * g - 20 * g + 5) / 4.0, g]])


def exact(case, seed):
    m, P, a = _inputs(case, seed)
    D = _Disc(case)
    if case["op"] == "linearize":
        vals = torch.zeros(D.nvals + 1, dtype=F64, device=DEV)
        g = torch.zeros(D.nF, D.mm, D.L, dtype=F64, device=DEV)
        y = torch.zeros_like(g)
        x = D.pad(a["x"])
        dU, dQ = torch.empty(a["U"].numel(), dtype=F64, device=DEV), torch.empty(a["Q"].numel(), dtype=F64, device=DEV)
        for G in D.chunks():
            S, gk, X, yk, dq0 = D.condense(G, a, P["dt"], P["a"])
            at = D.block_index(G)
            vals.index_add_(0, torch.where(at < 0, D.nvals, at).reshape(-1), S.reshape(-1))
            D.scatter(G, gk, g)
            D.scatter(G, torch.einsum("nrc,nc->nr", S, x[D.e2f[G["idx"]]].reshape(G["n"], -1)), y)
            u, q = D.recover(G, X, yk, dq0, x)
            dU[G["u_at"].reshape(-1)] = u.reshape(-1)
            dQ[G["q_at"].reshape(-1)] = q.reshape(-1)
        return {"S": vals[:-1], "g": D.unpad(g, a["UH"]), "y": D.unpad(y, a["UH"]), "dQ": dQ.reshape(a["Q"].shape),
                "dU": dU.reshape(a["U"].shape)}
    if case["op"] == "solve":
        return {"x": D.unpad(_System(D, a, P["dt"], P["a"]).solve(), a["UH"])}
    if case["op"] == "newton":
        a = _newton_exact(D, a, P["dt"], P["a"], 4)
        return {k: a[k] for k in ("U", "Q", "UH")}
    A = _sdirk3()
    dinv = np.linalg.inv(A)
    Un, stages = a["U"].clone(), []
    for i in range(3):
        Us = Un.clone()
        for j in range(i):
            Us -= A[i, i] * dinv[i, j] * (stages[j] - Un)
        a = _newton_exact(D, dict(a, Us=Us), P["dt"], float(A[i, i]), 4)
        stages.append(a["U"])
    return {k: a[k] for k in ("U", "Q", "UH")}
