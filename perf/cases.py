"""The workloads this solver is timed on: calls that a user's program makes, over the range of sizes,
meshes, fluxes, boundary conditions and precisions of the repository's own configurations.

A case names a flow (one of FLOWS: box, boundary planes, parameters and initial field of a configuration of
bench.py, cases.py or the tests), the layer pattern and size of its mesh, the call that is made and the
arithmetic. The mesh of a case is built once in a process; a state holds a solver on it and an initial field
of its own (a seeded perturbation and phase).

The mixed path computes the reconstruction and the flux in FP32, so its results carry single precision; a
program that chose it takes them over as float32, and so do these cases. FP64 results stay FP64.

`exact` is the method of the paper written with numpy and torch alone, in FP64: topology by sorting, least
squares by orthogonalisation, the kinetic moments by their recurrences, every slope by forward-mode
derivatives of the moments, and the adjoint by torch's reverse mode.
"""
import functools
import math

import numpy as np
import torch

import paper_2203_09047_gb300 as gks
from paper_2203_09047_gb300 import inputs as I
from paper_2203_09047_gb300.autograd import s2o4_rollout

GAMMA = 1.4
PERIODIC, SLIP, NOSLIP, FAR = 0, 1, 2, 3
MIXED = {"mixed": gks.GKS_PREC_MIXED, "fp64": gks.GKS_PREC_FP64, "mixed64": gks.GKS_PREC_MIXED_FP64UPD}
EXACT_CELLS = 70000  # above this the plain evaluation takes too long

_LID = [[0.0] * 3 for _ in range(6)]
_LID[4][0] = 0.15
_SOD = [[1.0, 0.0, 0.0, 0.0, 1.0] for _ in range(6)]
_SOD[3] = [0.125, 0.0, 0.0, 0.0, 0.1]

# box, boundary planes per axis, jitter, enlarged stencils, CFL number, parameters
FLOWS = {
    # Section 5.1 accuracy test, the bench's headline: Euler, smooth flux, zero collision time
    "advection": dict(lo=(0, 0, 0), hi=(2, 2, 2), bc=(0, 0, 0), jitter=0.1, min_stencil=18, cfl=0.5, prm={}),
    # the same field, Navier-Stokes with the full flux: the configuration of the adjoint runs
    "navier": dict(lo=(0, 0, 0), hi=(2, 2, 2), bc=(0, 0, 0), jitter=0.1, min_stencil=18, cfl=0.5,
                   prm=dict(flux_mode=1, tau_model=2, mu=1e-3)),
    # Taylor-Green vortex, Re 1600, Pr 0.72
    "tgv": dict(lo=(0, 0, 0), hi=(2 * math.pi,) * 3, bc=(0, 0, 0), jitter=0.05, min_stencil=18, cfl=0.5,
                prm=dict(flux_mode=0, tau_model=2, mu=1.0 / 1600.0, Pr=0.72)),
    # Section 5 spherical explosion in a reflecting box: full flux, inviscid collision time
    "explosion": dict(lo=(-1, -1, -1), hi=(1, 1, 1), bc=(1, 1, 1), jitter=0.1, min_stencil=18, cfl=0.5,
                      prm=dict(flux_mode=1, tau_model=1, gp_fallback=1)),
    # Section 5 Riemann tube (Sod): far-field ends, slip sides
    "tube": dict(lo=(0, 0, 0), hi=(1, 0.1, 0.1), bc=(3, 1, 1), jitter=0.0, min_stencil=0, cfl=0.5,
                 prm=dict(flux_mode=1, tau_model=1, gp_fallback=1, farfield=_SOD)),
    # Section 5.3 lid-driven cavity: no-slip isothermal walls, lid at Ma 0.15, Re 1000, implicit steps
    "cavity": dict(lo=(0, 0, 0), hi=(1, 1, 1), bc=(2, 2, 2), jitter=0.1, min_stencil=0, cfl=2.0,
                   prm=dict(flux_mode=1, tau_model=2, mu=1.5e-4, wall_u=_LID, wall_T=[1.0 / GAMMA] * 6)),
}


def listed():
    return [
        # the smallest mesh of the tests and smoke(): ten steps of a debugging or coupling run, launch bound
        dict(name="step-small-mixed", flow="advection", layers="hybrid8", n=8, nx=8, call="step", steps=10, prec="mixed"),
        # the bench's headline workload, 1,048,576 cells
        dict(name="step-large-mixed", flow="advection", layers="hybrid8", n=64, nx=64, call="step", steps=4, prec="mixed"),
        # the FP64 reference path on a mid-size mesh of the convergence study
        dict(name="step-mid-fp64", flow="advection", layers="hybrid8", n=32, nx=32, call="step", steps=2, prec="fp64"),
        # 10^3 hexahedra (the paper's coarsest accuracy mesh): single residual calls of an outer solver
        dict(name="residual-hex-fp64", flow="navier", layers="hex", n=10, nx=10, call="residual", steps=1, prec="fp64"),
        # single residual calls in FP32 on an odd-sized box
        dict(name="residual-mid-mixed", flow="advection", layers="hybrid8", n=24, nx=23, call="residual", steps=1, prec="mixed"),
        # the explosion with the time step re-evaluated every step, as the configuration runs it
        dict(name="explosion-mixed", flow="explosion", layers="hybrid8", n=48, nx=48, call="adaptive", steps=3, prec="mixed"),
        # Taylor-Green vortex on its layer pattern, FP32 flux with the FP64 update
        dict(name="tgv-mixed64", flow="tgv", layers="tgv48", n=43, nx=43, call="step", steps=3, prec="mixed64"),
        # Sod tube on Kuhn tetrahedra, 100 x 10 x 10 cubes
        dict(name="tube-tet-fp64", flow="tube", layers="tet", n=10, nx=100, call="adaptive", steps=2, prec="fp64"),
        # the bench's implicit workload: lid-driven cavity of the paper's size
        dict(name="cavity-mixed", flow="cavity", layers="hybrid8", n=32, nx=32, call="implicit", steps=5, prec="mixed"),
        # the cavity on 20^3 cubes of tetrahedra in FP64
        dict(name="cavity-tet-fp64", flow="cavity", layers="tet", n=20, nx=20, call="implicit", steps=2, prec="fp64"),
        # the residual's vector-Jacobian product on the adjoint configuration (32 cubes, full flux)
        dict(name="vjp-mid", flow="navier", layers="hybrid8", n=32, nx=32, call="vjp", steps=1, prec="fp64"),
        # gradient through a short differentiable rollout (smooth flux)
        dict(name="rollout-grad", flow="advection", layers="hybrid8", n=16, nx=16, call="rollout", steps=2, prec="fp64"),
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["explicit", "explicit", "residual", "explosion", "tgv", "tube", "cavity", "vjp", "rollout"])
    prec = rng.choice(["mixed", "mixed", "fp64", "mixed64"])
    top = 40 if prec == "fp64" else 64
    if kind == "explicit":
        layers = rng.choice(["hybrid8", "hybrid8", "hex", "prism", "tet"])
        nx = _log_int(rng, 6, 28 if layers == "tet" else top)
        n = 8 * max(1, round(nx / 8)) if layers == "hybrid8" else nx
        c = dict(flow="advection", layers=layers, n=n, nx=nx, call="step", steps=rng.randint(1, 6), prec=prec)
        if prec == "fp64":
            c["steps"] = rng.randint(1, 2)
        elif nx > 54:
            c["steps"] = rng.randint(1, 4)
    elif kind == "residual":
        n = 8 * rng.randint(1, 5)
        c = dict(flow=rng.choice(["advection", "navier"]), layers="hybrid8", n=n, nx=rng.randint(max(6, n - 8), n + 6),
                 call="residual", steps=1, prec=rng.choice(["mixed", "fp64"]))
    elif kind == "explosion":
        n = 8 * rng.randint(2, 6)
        c = dict(flow="explosion", layers="hybrid8", n=n, nx=max(9, n + rng.randint(-5, 4)), call="adaptive",
                 steps=rng.randint(1, 3), prec=rng.choice(["mixed", "mixed64"]))
    elif kind == "tgv":
        n = _log_int(rng, 9, 32 if prec == "fp64" else 50)
        c = dict(flow="tgv", layers="tgv48", n=n, nx=n, call="step", steps=rng.randint(1, 2 if prec == "fp64" else 3), prec=prec)
    elif kind == "tube":
        n = rng.randint(4, 13)
        c = dict(flow="tube", layers=rng.choice(["hex", "tet"]), n=n, nx=10 * n + rng.randint(-9, 9), call="adaptive", steps=rng.randint(1, 2),
                 prec=rng.choice(["mixed", "fp64"]))
    elif kind == "cavity":
        layers = rng.choice(["hybrid8", "tet", "hex"])
        nx = _log_int(rng, 8, 22 if layers == "tet" else 40)
        n = 8 * max(1, round(nx / 8)) if layers == "hybrid8" else nx
        p = rng.choice(["mixed", "fp64"])
        c = dict(flow="cavity", layers=layers, n=n, nx=nx, call="implicit", steps=rng.randint(1, 6 if p == "mixed" else 2), prec=p)
    elif kind == "vjp":
        n = 8 * rng.randint(1, 4)
        c = dict(flow=rng.choice(["advection", "navier"]), layers="hybrid8", n=n, nx=rng.randint(max(6, n - 9), n + 1),
                 call="vjp", steps=1, prec="fp64")
    else:
        n = 8 * rng.randint(1, 2)
        c = dict(flow=rng.choice(["advection", "navier"]), layers="hybrid8", n=n, nx=rng.randint(6, 19),
                 call="rollout", steps=rng.randint(1, 2), prec="fp64")
    return draw(rng) if any(dict(c, name=x["name"]) == x for x in listed()) else c


def _ny(c):
    return c["n"] if c["flow"] == "tube" else c["nx"]


def _mesh_dict(c):
    f = FLOWS[c["flow"]]
    return I.layered_box_mesh(c["n"], c["layers"], lo=f["lo"], hi=f["hi"], bc=f["bc"], jitter=f["jitter"],
                              shape=(c["nx"], _ny(c)))


@functools.lru_cache(maxsize=None)
def _mesh(flow, layers, n, nx):
    c = dict(flow=flow, layers=layers, n=n, nx=nx)
    m = _mesh_dict(c)
    return m, gks.Mesh(m, min_stencil=FLOWS[flow]["min_stencil"])


def _field(c, m, seed):
    """The flow's initial field [5, cells] with a seeded phase and a seeded perturbation of every value."""
    u = I.uniform01(seed + 1, np.arange(4, dtype=np.uint64))
    flow = c["flow"]
    if flow in ("advection", "navier"):
        x = I.vertex_mean(m) + 2.0 * u[:3]
        q = I.primitive_to_conserved(*I.advection_primitive(x))
        amp = 0.03
    elif flow == "tgv":
        q = I.taylor_green_state(m)
        amp = 0.01
    elif flow in ("explosion", "tube"):
        # the printed states, their jump spread over about three cells as the first steps leave it: on the bare
        # jump one perturbed field in some hundreds meets a non-physical interface state and is refused
        x = I.vertex_mean(m)
        if flow == "explosion":
            d, h = 0.4 - np.sqrt((x * x).sum(axis=1)), 2.0 / c["nx"]
        else:
            d, h = 0.5 - x[:, 0], 1.0 / c["nx"]
        one = 0.5 * (1.0 + np.tanh(d / (1.5 * h)))
        q = I.primitive_to_conserved(0.125 + 0.875 * one, np.zeros_like(x), 0.1 + 0.9 * one)
        amp = 0.001
    else:  # the gas of the cavity at rest
        q = np.zeros((5, len(m["cell_type"])))
        q[0] = 1.0
        q[4] = 1.0 / GAMMA / (GAMMA - 1.0)
        amp = 0.01
    return I.perturbed_state(np.ascontiguousarray(q), seed + 7, amp)


def prepare(case, seed):
    m, mesh = _mesh(case["flow"], case["layers"], case["n"], case["nx"])
    f = FLOWS[case["flow"]]
    S = gks.Solver(mesh, precision=MIXED[case["prec"]], **f["prm"])
    q = _field(case, m, seed)
    Q = torch.from_numpy(q).cuda()
    s = dict(case=case, S=S, Q=Q, cfl=f["cfl"])
    S.set_state(Q)
    s["dt"] = S.max_dt(f["cfl"])
    if case["call"] == "vjp":
        g = I.normal_directions(q.shape, 2, seed + 3)
        s["gL"], s["gLt"] = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in g)
    elif case["call"] == "rollout":
        s["g"] = torch.from_numpy(np.ascontiguousarray(I.normal_directions(q.shape, 1, seed + 3)[0])).cuda()
    return s


def run(s):
    case, S, Q, dt = s["case"], s["S"], s["Q"], s["dt"]
    call, steps = case["call"], case["steps"]
    if call == "residual":
        out = S.residual(Q, dt)
    elif call == "vjp":
        return S.residual_vjp(Q, dt, s["gL"], s["gLt"])
    elif call == "rollout":
        x = Q.detach().requires_grad_(True)
        y = s2o4_rollout(x, S, dt, steps)
        (gx,) = torch.autograd.grad(y, x, s["g"])
        return y.detach(), gx
    else:
        S.set_state(Q)
        if call == "step":
            S.step(dt, steps)
        elif call == "implicit":
            S.step_implicit(dt, steps)
        else:  # the time step of every step from the state before it
            for _ in range(steps):
                S.step(S.max_dt(s["cfl"]), 1)
        out = (S.get_state(),)
    return tuple(x if case["prec"] == "fp64" else x.float() for x in out)


# ------------------------------------------------------------------------------------------ work
_CELLS = {"hex": {8: 1}, "prism": {6: 2}, "trans": {5: 5, 4: 2}, "transm": {5: 5, 4: 2}, "tet": {4: 6}}
_FACES = {4: 4, 5: 5, 6: 5, 8: 6}
_MEMBERS = {4: 18, 5: 18, 6: 19, 8: 24}  # cells of a big stencil
_PAIRS = {4: 24, 5: 46, 6: 18, 8: 24}    # (sub-stencil, member) pairs


def work(case):
    """Bytes: the state (or cotangents) in and out once per pass, and per residual the state, the least-squares
    weights of every member, the face points and the new state, each once, in the working precision. Flops: the
    least-squares products, the weights, and the flux of every face point."""
    layers = I.layer_pattern(case["layers"], case["n"])
    cells = {}
    for k in layers:
        for t, v in _CELLS[k].items():
            cells[t] = cells.get(t, 0) + v * case["nx"] * _ny(case)
    nc = sum(cells.values())
    nf = sum(_FACES[t] * v for t, v in cells.items()) / 2
    mem = sum(_MEMBERS[t] * v for t, v in cells.items())
    pairs = sum(_PAIRS[t] * v for t, v in cells.items())
    full = FLOWS[case["flow"]]["prm"].get("flux_mode", 0)
    r = 8 if case["prec"] == "fp64" else 4
    byte = 80 * nc + r * (9 * mem + 3 * pairs + 40 * nf)
    flop = 90 * mem + 30 * pairs + 500 * nc + (1800 if full else 1000) * 4 * nf
    stages = {"residual": 1, "vjp": 3, "implicit": 1}.get(case["call"], 2) * case["steps"]
    if case["call"] == "rollout":
        stages *= 5  # forward, recomputation and a reverse of twice its work
    if case["call"] == "implicit":
        byte += 3 * (10 * r + 16) * nc
        flop += 3 * 100 * 2 * nf
    return {"bytes": 80.0 * nc + byte * stages, "flops": float(flop * stages)}


# ------------------------------------------------------------------------------------------ exact
_SLOTS = {4: (0, 1, 2, 4), 5: (0, 1, 2, 3, 4), 6: (0, 1, 2, 4, 5, 6), 8: tuple(range(8))}
_LOCAL = {
    4: ((1, 2, 3), (1, 2, 4), (2, 3, 4), (3, 1, 4)),
    5: ((1, 2, 5), (2, 3, 5), (3, 4, 5), (4, 1, 5), (1, 2, 3, 4)),
    6: ((1, 2, 3), (4, 5, 6), (1, 2, 5, 4), (2, 3, 6, 5), (3, 1, 4, 6)),
    8: ((1, 2, 3, 4), (1, 2, 6, 5), (2, 3, 7, 6), (3, 4, 8, 7), (4, 1, 5, 8), (5, 6, 7, 8)),
}
# sub-stencils: three faces, and the face whose neighbour's neighbours join (0: none)
_SUBS = {
    8: ((1, 2, 3, 0), (1, 3, 4, 0), (1, 4, 5, 0), (1, 5, 2, 0), (6, 2, 3, 0), (6, 3, 4, 0), (6, 4, 5, 0), (6, 5, 2, 0)),
    6: ((1, 3, 4, 0), (1, 4, 5, 0), (1, 5, 3, 0), (2, 3, 4, 0), (2, 4, 5, 0), (2, 5, 3, 0)),
    4: ((1, 2, 3, 1), (1, 2, 4, 2), (2, 3, 4, 3), (3, 1, 4, 4)),
    5: ((1, 2, 3, 1), (2, 3, 4, 2), (3, 4, 1, 3), (4, 1, 2, 4), (1, 2, 5, 1), (2, 3, 5, 2), (3, 4, 5, 3), (4, 1, 5, 4)),
}


def _topology(m, min_stencil):
    """Faces, stencil members (cell, mirror signs, shift, planes crossed) and sub-stencil membership."""
    xyz, ctype, cn = m["xyz"], m["cell_type"].astype(np.int64), m["cell_nodes"]
    lo, hi, bc = (np.asarray(m[k]) for k in ("lo", "hi", "bc"))
    nc, ext = len(ctype), float((hi - lo).max())
    w = xyz.copy()
    for a in range(3):
        if bc[a] == PERIODIC:
            w[np.abs(w[:, a] - hi[a]) < 1e-9 * ext, a] = lo[a]
    key = np.round((w - lo) / (1e-7 * ext)).astype(np.int64)
    rep = np.unique(key, axis=0, return_inverse=True)[1].reshape(-1)
    # one record per (cell, local face), nodes in label order
    cell, lf, nodes = [], [], []
    for t, faces in _LOCAL.items():
        c = np.nonzero(ctype == t)[0]
        for p, labels in enumerate(faces):
            v = cn[c][:, [_SLOTS[t][k - 1] for k in labels]]
            nodes.append(v if len(labels) == 4 else np.concatenate([v, np.full((len(c), 1), -1)], axis=1))
            cell.append(c)
            lf.append(np.full(len(c), p))
    cell, lf, nodes = np.concatenate(cell), np.concatenate(lf), np.concatenate(nodes)
    ids = np.where(nodes >= 0, rep[nodes], -1)
    by = np.argsort(ids, axis=1)
    ids, snodes = np.take_along_axis(ids, by, 1), np.take_along_axis(nodes, by, 1)
    o = np.lexsort((lf, cell, ids[:, 3], ids[:, 2], ids[:, 1], ids[:, 0]))
    cell, lf, nodes, ids, snodes = cell[o], lf[o], nodes[o], ids[o], snodes[o]
    first = np.ones(len(cell), bool)
    first[1:] = (ids[1:] != ids[:-1]).any(1)
    at = np.nonzero(first)[0]
    two = np.zeros(len(at), bool)
    two[:-1] = np.diff(at) == 2
    two[-1] = len(cell) - at[-1] == 2
    own, other = at, np.where(two, at + 1, at)
    shift = np.where(two[:, None], xyz[snodes[own, 3]] - xyz[snodes[other, 3]], 0.0)
    shift[np.abs(shift) < 1e-9 * ext] = 0.0
    plane = np.full(len(at), -1)
    for a in range(3):
        if bc[a] == PERIODIC:
            continue
        for side, at_x in ((0, lo[a]), (1, hi[a])):
            x = np.where(nodes[own] >= 0, xyz[nodes[own], a], at_x)
            plane[~two & (plane < 0) & (np.abs(x - at_x) < 1e-9 * ext).all(1)] = a + 3 * side
    assert ((plane >= 0) | two).all()
    f_nb = np.where(two, cell[other], -1)
    # neighbour of every (cell, local face): cell, signs, shift, plane
    N = np.full((nc, 6), -1)
    Ns, Nt, Nw = np.ones((nc, 6, 3)), np.zeros((nc, 6, 3)), np.full((nc, 6), -1)
    N[cell[own], lf[own]] = np.where(two, f_nb, cell[own])
    Nt[cell[own], lf[own]] = shift
    k = np.nonzero(two)[0]
    N[cell[other[k]], lf[other[k]]] = cell[own[k]]
    Nt[cell[other[k]], lf[other[k]]] = -shift[k]
    k = np.nonzero(~two)[0]
    ax = plane[k] % 3
    Ns[cell[own[k]], lf[own[k]], ax] = -1
    Nt[cell[own[k]], lf[own[k]], ax] = 2.0 * np.where(plane[k] < 3, lo[ax], hi[ax])
    Nw[cell[own[k]], lf[own[k]]] = plane[k]

    def through(c0, s0, t0, w0, f):
        """The neighbour across face f of the image (c0, s0, t0, planes w0 [.., 3], innermost first)."""
        ok = (c0 >= 0) & (N[c0, f] >= 0)
        c = np.where(ok, N[c0, f], -1)
        s, t = s0 * Ns[c0, f], s0 * Nt[c0, f] + t0
        add = Nw[c0, f]
        ww = np.where((add >= 0)[..., None], np.concatenate([add[..., None], w0[..., :-1]], -1), w0)
        lost = (add >= 0) & (w0[..., -1] >= 0)
        ww[lost, -1] = 9  # more planes than are kept
        return c, s, t, ww

    everyone = np.arange(nc)
    one = (N, Ns, Nt, np.concatenate([Nw[..., None], np.full((nc, 6, 2), -1)], -1))
    r2 = through(one[0][:, :, None], one[1][:, :, None], one[2][:, :, None],
                 np.broadcast_to(one[3][:, :, None], (nc, 6, 6, 3)), np.arange(6)[None, None])
    C = np.concatenate([one[0], r2[0].reshape(nc, 36)], 1)
    Sg = np.concatenate([one[1], r2[1].reshape(nc, 36, 3)], 1)
    T = np.concatenate([one[2], r2[2].reshape(nc, 36, 3)], 1)
    W = np.concatenate([one[3], r2[3].reshape(nc, 36, 3)], 1)

    def keys(c, s, t):
        q = np.round(t / ext * 1000.0).astype(np.int64) + 4096
        code = (s < 0).astype(np.int64) @ np.array([1, 2, 4])
        return ((((c * 8 + code) * 8192 + q[..., 0]) * 8192) + q[..., 1]) * 8192 + q[..., 2]

    K = np.where(C >= 0, keys(C, Sg, T), -1)
    self_key = keys(everyone, np.ones((nc, 3)), np.zeros((nc, 3)))
    place = np.broadcast_to(np.arange(42), (nc, 42)).copy()  # where a slot's image is first listed
    for j in range(42):
        for i in range(j):
            same = (place[:, j] == j) & (K[:, j] == K[:, i])
            place[same, j] = place[same, i]
    place[(C < 0) | (K == self_key[:, None])] = -1
    valid = place == np.arange(42)
    # enlarged stencils: the face neighbours of the members, in order, until there are enough
    extra = []
    count = valid.sum(1)
    need = np.nonzero(count < min_stencil)[0]
    if len(need):
        rank = np.argsort(~valid[need], axis=1, kind="stable")  # members first, in slot order
        n2, cnt = count[need].copy(), count[need].copy()
        extra = [dict(c=np.full(nc, -1), s=np.ones((nc, 3)), t=np.zeros((nc, 3)), w=np.full((nc, 3), -1))
                 for _ in range(int(min_stencil - cnt.min()))]
        more = np.full((len(need), len(extra)), -1)
        for k in range(int(n2.max())):
            at_k = rank[:, k]
            img = tuple(v[need, at_k] for v in (C, Sg, T, W))
            for f in range(6):
                act = (k < n2) & (cnt < min_stencil)
                if not act.any():
                    break
                c, s, t, ww = through(*img, f)
                kk = np.where(c >= 0, keys(c, s, t), -1)
                act &= (c >= 0) & (ww[:, 2] < 0) & (kk != self_key[need])
                act &= ~(kk[:, None] == np.where(valid[need], K[need], -2)).any(1) & ~(kk[:, None] == more).any(1)
                a = np.nonzero(act)[0]
                for j in np.unique(cnt[a] - n2[a]):
                    b = a[cnt[a] - n2[a] == j]
                    e = extra[j]
                    e["c"][need[b]], e["s"][need[b]], e["t"][need[b]], e["w"][need[b]] = c[b], s[b], t[b], ww[b]
                    more[b, j] = kk[b]
                cnt[a] += 1
    sub = np.zeros((nc, 8, 42 + len(extra)), bool)
    nsub = np.zeros(nc, np.int64)
    for t, rules in _SUBS.items():
        c = np.nonzero(ctype == t)[0]
        nsub[c] = len(rules)
        for s, rule in enumerate(rules):
            slots = [f - 1 for f in rule[:3]] + ([6 + 6 * (rule[3] - 1) + q for q in range(6)] if rule[3] else [])
            for q in slots:
                p = place[c, q]
                sub[c[p >= 0], s, p[p >= 0]] = True
    if extra:
        C = np.concatenate([np.where(valid, C, -1)] + [e["c"][:, None] for e in extra], 1)
        Sg = np.concatenate([Sg] + [e["s"][:, None] for e in extra], 1)
        T = np.concatenate([T] + [e["t"][:, None] for e in extra], 1)
        W = np.concatenate([W] + [e["w"][:, None] for e in extra], 1)
    else:
        C = np.where(valid, C, -1)
    # face vertices of the owner, oriented outwards, smallest node id first, triangles (a, b, c, c)
    fv, oc = nodes[own].copy(), cell[own]
    tri = fv[:, 3] < 0
    x = xyz[np.where(fv < 0, fv[:, 2:3], fv)]
    xe = 0.5 * (-x[:, 0] - x[:, 1] + x[:, 2] + x[:, 3])
    xz = 0.5 * (-x[:, 0] + x[:, 1] + x[:, 2] - x[:, 3])
    out = (np.cross(xe, xz) * (x.mean(1) - xyz[cn[oc]].mean(1))).sum(1) < 0
    fv[out & ~tri] = fv[out & ~tri][:, ::-1]
    fv[out & tri, :3] = fv[out & tri, :3][:, ::-1]
    for sel, n in ((tri, 3), (~tri, 4)):
        v = fv[sel, :n]
        r = (np.arange(n)[None] + v.argmin(1)[:, None]) % n
        fv[sel, :n] = np.take_along_axis(v, r, 1)
    fv[tri, 3] = fv[tri, 2]
    return dict(nc=nc, f_own=oc, f_nb=f_nb, f_shift=shift, f_plane=plane, f_x=xyz[fv], C=C, S=Sg, T=T, W=W,
                sub=sub, nsub=nsub, cell_x=xyz[cn])


def _pinv(A):
    """Pseudo-inverse of full-rank tall matrices [..., m, n] by twice-iterated Gram-Schmidt."""
    n = A.shape[-1]
    V, cols, R = A, [], torch.zeros(A.shape[:-2] + (n, n), dtype=A.dtype, device=A.device)
    for j in range(n):
        v = V[..., j]
        for _ in range(2):
            for i, q in enumerate(cols):
                r = (q * v).sum(-1)
                R[..., i, j] += r
                v = v - r[..., None] * q
        R[..., j, j] = v.norm(dim=-1)
        cols.append(v / R[..., j, j][..., None])
    return torch.linalg.solve_triangular(R, torch.stack(cols, -2), upper=True)


class _Plain:
    """The method of the paper on one mesh, in FP64 torch."""

    def __init__(self, case):
        f = FLOWS[case["flow"]]
        m = _mesh_dict(case)
        top = _topology(m, f["min_stencil"])
        dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(dev)
        self.dev, self.bc, self.nc = dev, f["bc"], top["nc"]
        p = dict(flux_mode=0, tau_model=0, mu=0.0, Pr=1.0, gp_fallback=0, wall_u=[[0.0] * 3] * 6, wall_T=[0.0] * 6,
                 farfield=[[1.0, 0, 0, 0, 1 / GAMMA]] * 6)
        p.update(f["prm"])
        self.p = p
        self.K = (5 - 3 * GAMMA) / (GAMMA - 1)
        # cell volumes, centroids and scaled central second moments by the 27-point rule
        x = t(top["cell_x"])
        org = x.mean(1)
        x = x - org[:, None]
        g = torch.tensor([-math.sqrt(0.6) / 2, 0.0, math.sqrt(0.6) / 2], dtype=torch.float64, device=dev)
        gw = torch.tensor([5 / 18, 8 / 18, 5 / 18], dtype=torch.float64, device=dev)
        sg = torch.tensor([[-1, -1, -1], [1, -1, -1], [1, 1, -1], [-1, 1, -1], [-1, -1, 1], [1, -1, 1], [1, 1, 1],
                           [-1, 1, 1]], dtype=torch.float64, device=dev)
        m0, m1, m2 = 0.0, 0.0, 0.0
        for a in range(3):
            for b in range(3):
                for c in range(3):
                    fx, fy, fz = (0.5 + sg[:, k] * v for k, v in enumerate((g[a], g[b], g[c])))
                    pt = (x * (fx * fy * fz)[None, :, None]).sum(1)
                    J = torch.stack([(x * d[None, :, None]).sum(1) for d in
                                     (sg[:, 0] * fy * fz, fx * sg[:, 1] * fz, fx * fy * sg[:, 2])], 1)
                    wt = gw[a] * gw[b] * gw[c] * torch.linalg.det(J)
                    m0, m1 = m0 + wt, m1 + wt[:, None] * pt
                    m2 = m2 + wt[:, None, None] * pt[:, :, None] * pt[:, None, :]
        self.vol, cc = m0, m1 / m0[:, None]
        self.cen, self.h = org + cc, m0 ** (1 / 3)
        mom = (m2 / m0[:, None, None] - cc[:, :, None] * cc[:, None, :]) / (self.h ** 2)[:, None, None]
        pa, pb = [0, 1, 2, 0, 0, 1], [0, 1, 2, 1, 2, 2]
        self.mom = mom[:, pa, pb]
        # stencils: rows of scaled monomial means, pseudo-inverses
        C, Sg, T = t(top["C"]), t(top["S"]), t(top["T"])
        self.valid, self.C = C >= 0, C.clamp(min=0)
        self.W = t(top["W"])
        d = (Sg * self.cen[self.C] + T - self.cen[:, None]) / self.h[:, None, None]
        r2 = (self.h[self.C] / self.h[:, None]) ** 2
        mj = self.mom[self.C] * Sg[..., pa] * Sg[..., pb] * r2[..., None]
        A = torch.cat([d, d[..., pa] * d[..., pb] + mj - self.mom[:, None]], -1) * self.valid[..., None]
        self.A = _pinv(A)
        self.sub, self.M = t(top["sub"]), t(top["nsub"])
        on = torch.arange(8, device=dev)[None] < self.M[:, None]
        self.on = on
        fake = torch.zeros_like(A[:, :, :3])
        fake[:, 0, 0] = fake[:, 1, 1] = fake[:, 2, 2] = 1.0
        self.B = torch.stack([_pinv(torch.where(on[:, s, None, None], A[:, :, :3] * self.sub[:, s, :, None], fake)) *
                              on[:, s, None, None] for s in range(8)], 1)
        # faces: 2 x 2 Gauss points, unit normals, weights; offsets from both centroids
        v, self.o, self.nb = t(top["f_x"]), t(top["f_own"]), t(top["f_nb"])
        self.plane = t(top["f_plane"])
        self.inner = self.nb >= 0
        nbc = torch.where(self.inner, self.nb, self.o)
        self.nbc = nbc
        cn = torch.where(self.inner[:, None], self.cen[nbc] + t(top["f_shift"]), self.cen[self.o])
        q = math.sqrt(3) / 6
        se, sz = torch.tensor([-1.0, -1, 1, 1], device=dev).double(), torch.tensor([-1.0, 1, 1, -1], device=dev).double()
        pts, nrm = [], []
        for eta in (-q, q):
            for zeta in (-q, q):
                fe, fz = 0.5 + se * eta, 0.5 + sz * zeta
                ein = lambda u: (v * u[None, :, None]).sum(1)
                pts.append(ein(fe * fz))
                nrm.append(torch.linalg.cross(ein(se * fz), ein(fe * sz)))
        xg, ng = torch.stack(pts, 1), torch.stack(nrm, 1)
        ln = ng.norm(dim=-1)
        self.n, self.w = ng / ln[..., None], 0.25 * ln
        self.dl, self.dr = xg - self.cen[self.o][:, None], xg - cn[:, None]
        av = 0.5 * torch.linalg.cross(v[:, 3] - v[:, 1], v[:, 2] - v[:, 0])
        self.area = av.norm(dim=-1)
        self.fn = av / self.area[:, None]
        amax = torch.zeros(self.nc, dtype=torch.float64, device=dev)
        wsum = self.w.sum(1)
        amax.scatter_reduce_(0, self.o, wsum, "amax")
        amax.scatter_reduce_(0, nbc, wsum, "amax")
        self.hdt = self.vol / amax

    # -- boundary maps -----------------------------------------------------------------------
    def far_state(self, q, plane):
        """The characteristic state of q [..., 5] at the far-field planes plane [...]."""
        inf = torch.tensor(self.p["farfield"], dtype=torch.float64, device=self.dev)[plane.clamp(0, 5)]
        ax, sg = plane.clamp(min=0) % 3, torch.where(plane >= 3, 1.0, -1.0).double()
        U = q[..., 1:4] / q[..., :1]
        p = (GAMMA - 1) * (q[..., 4] - 0.5 * q[..., 0] * (U * U).sum(-1))
        c = (GAMMA * p / q[..., 0]).sqrt()
        pick = lambda v: torch.gather(v, -1, ax[..., None])[..., 0]
        un, uinf = sg * pick(U), sg * pick(inf[..., 1:4])
        cinf = (GAMMA * inf[..., 4] / inf[..., 0]).sqrt()
        g1 = GAMMA - 1
        rp, rm = un + 2 * c / g1, uinf - 2 * cinf / g1
        unb, cb = 0.5 * (rp + rm), 0.25 * g1 * (rp - rm)
        leave = unb >= 0
        s = torch.where(leave, p / q[..., 0] ** GAMMA, inf[..., 4] / inf[..., 0] ** GAMMA)
        Ub = torch.where(leave[..., None], U, inf[..., 1:4]).scatter(-1, ax[..., None], (sg * unb)[..., None])
        rb = (cb * cb / (GAMMA * s)) ** (1 / g1)
        pb = rb * cb * cb / GAMMA
        into = un <= -c
        rb, pb = torch.where(into, inf[..., 0], rb), torch.where(into, inf[..., 4], pb)
        Ub = torch.where(into[..., None], inf[..., 1:4], Ub)
        b = torch.cat([rb[..., None], rb[..., None] * Ub, (pb / g1 + 0.5 * rb * (Ub * Ub).sum(-1))[..., None]], -1)
        return torch.where((un >= c)[..., None], q, b)

    def plane_kind(self, plane):
        return torch.tensor(self.bc, device=self.dev)[plane.clamp(min=0) % 3]

    def image(self, q, plane):
        """The flow variables q [..., 5] of a cell mirrored at a plane (ghost cells: walls are adiabatic)."""
        if not any(self.bc):
            return q
        kind = self.plane_kind(plane)
        on = plane >= 0
        flip = torch.nn.functional.one_hot(plane.clamp(min=0) % 3, 3).double()
        uw = torch.tensor(self.p["wall_u"], dtype=torch.float64, device=self.dev)[plane.clamp(0, 5)]
        m = q[..., 1:4]
        slip = torch.cat([q[..., :1], m * (1 - 2 * flip), q[..., 4:]], -1)
        wall = torch.cat([q[..., :1], 2 * uw * q[..., :1] - m,
                          (q[..., 4] + 2 * (uw * uw).sum(-1) * q[..., 0] - 2 * (uw * m).sum(-1))[..., None]], -1)
        r = torch.where((on & (kind == SLIP))[..., None], slip, q)
        r = torch.where((on & (kind == NOSLIP))[..., None], wall, r)
        if FAR in self.bc:
            r = torch.where((on & (kind == FAR))[..., None], self.far_state(q, plane), r)
        return r

    def ghost(self, v, g, plane):
        """Ghost value [N, 5] and gradient [N, 3, 5] at the boundary points of `plane`."""
        kind = self.plane_kind(plane)
        flip = 1 - 2 * torch.nn.functional.one_hot(plane % 3, 3).double()
        uw = torch.tensor(self.p["wall_u"], dtype=torch.float64, device=self.dev)[plane]
        Tw = torch.tensor(self.p["wall_T"], dtype=torch.float64, device=self.dev)[plane]

        def wall(q):
            m = q[..., 1:4]
            e = 2 * (uw * uw).sum(-1) * q[..., 0] - 2 * (uw * m).sum(-1)
            iso = 2 * q[..., 0] * Tw / (GAMMA - 1) - q[..., 4] + (m * m).sum(-1) / q[..., 0]
            return torch.cat([q[..., :1], 2 * uw * q[..., :1] - m,
                              (e + torch.where(Tw > 0, iso, q[..., 4]))[..., None]], -1)

        def slip(q):
            return torch.cat([q[..., :1], q[..., 1:4] * flip, q[..., 4:]], -1)

        vg, gg = v, torch.zeros_like(g)
        for code, fn in ((SLIP, slip), (NOSLIP, wall)):
            if code in self.bc:
                on = kind == code
                dv = torch.stack([torch.func.jvp(fn, (v,), (g[:, d],))[1] for d in range(3)], 1)
                vg = torch.where(on[:, None], fn(v), vg)
                gg = torch.where(on[:, None, None], flip[:, :, None] * dv, gg)
        if FAR in self.bc:
            vg = torch.where((kind == FAR)[:, None], self.far_state(v, plane), vg)
        return vg, gg

    # -- reconstruction ----------------------------------------------------------------------
    def polynomials(self, Q):
        """Gradient b [nc, 5, 3] and Hessian H [nc, 5, 6] (xx yy zz xy xz yz) and value at the centroid."""
        q = Q.T
        mem = self.image(self.image(q[self.C], self.W[..., 0]), self.W[..., 1])
        dq = (mem - q[:, None]) * self.valid[..., None]                       # [nc, S, 5]
        a = self.A @ dq                                                       # [nc, 9, 5]
        b = self.B.reshape(self.nc, 24, -1) @ dq
        b = b.reshape(self.nc, 8, 3, 5)
        m2 = self.mom[:, :, None]
        gr = [(2 * a[:, 3], a[:, 6], a[:, 7]), (a[:, 6], 2 * a[:, 4], a[:, 8]), (a[:, 7], a[:, 8], 2 * a[:, 5])]
        beta0 = (a[:, :3] ** 2).sum(1) + 4 * (a[:, 3:6] ** 2).sum(1) + (a[:, 6:] ** 2).sum(1)
        for g in gr:
            beta0 = beta0 + (m2[:, 0] * g[0] ** 2 + m2[:, 1] * g[1] ** 2 + m2[:, 2] * g[2] ** 2 +
                             2 * (m2[:, 3] * g[0] * g[1] + m2[:, 4] * g[0] * g[2] + m2[:, 5] * g[1] * g[2]))
        bet = (b ** 2).sum(2)                                                 # [nc, 8, 5]
        on = self.on[..., None].double()
        M = self.M[:, None].double()
        x = beta0[:, None] - bet
        tau = (torch.where(x < 0, -x, x) * on).sum(1) / M
        wg, eps = 0.0125, 1e-8
        g0 = 1 - wg * M
        w0 = g0 * (1 + tau / (beta0 + eps))
        wm = wg * (1 + tau[:, None] / (bet + eps)) * on
        tot = w0 + wm.sum(1)
        wb0, wbm = w0 / tot, wm / tot[:, None]
        c = (wb0 / g0)[:, None] * a
        lin = c[:, :3] + (((wbm - (wb0 * wg / g0)[:, None] * on))[:, :, None] * b).sum(1)
        quad = c[:, 3:]
        val = q - (quad * self.mom[:, :, None]).sum(1)
        return val, lin / self.h[:, None, None], quad / (self.h ** 2)[:, None, None]

    def evaluate(self, poly, cell, d):
        """Values [F, 4, 5] and gradients [F, 4, 3, 5] at offsets d [F, 4, 3] of the cells [F]."""
        val, b, hq = (p[cell] for p in poly)
        d = d[..., None]
        x, y, z = d[:, :, 0], d[:, :, 1], d[:, :, 2]
        b, hq = b[:, None], hq[:, None]
        v = (val[:, None] + b[:, :, 0] * x + b[:, :, 1] * y + b[:, :, 2] * z + hq[:, :, 0] * x * x + hq[:, :, 1] * y * y +
             hq[:, :, 2] * z * z + hq[:, :, 3] * x * y + hq[:, :, 4] * x * z + hq[:, :, 5] * y * z)
        g = torch.stack([b[:, :, 0] + 2 * hq[:, :, 0] * x + hq[:, :, 3] * y + hq[:, :, 4] * z,
                         b[:, :, 1] + 2 * hq[:, :, 1] * y + hq[:, :, 3] * x + hq[:, :, 5] * z,
                         b[:, :, 2] + 2 * hq[:, :, 2] * z + hq[:, :, 4] * x + hq[:, :, 5] * y], 2)
        return v, g

    # -- kinetic flux ------------------------------------------------------------------------
    def moments(self, q, powers, side=0):
        """rho <u^a v^b w^c psi> of the Maxwellian of q [N, 5] for each (a, b, c) of `powers`, over the whole line
        (side 0) or u > 0 (1) or u < 0 (-1): the usual recurrences."""
        rho = q[:, 0]
        U = [q[:, k] / rho for k in (1, 2, 3)]
        p = (GAMMA - 1) * (q[:, 4] - 0.5 * rho * (U[0] ** 2 + U[1] ** 2 + U[2] ** 2))
        hil = p / rho
        one = torch.ones_like(rho)

        def line(u, start):
            m = list(start)
            while len(m) < 6:
                m.append(u * m[-1] + (len(m) - 1) * hil * m[-2])
            return m

        if side:
            lam = 0.5 / hil
            a0 = 0.5 * torch.special.erfc(-side * lam.sqrt() * U[0])
            first = (a0, U[0] * a0 + side * 0.5 * torch.exp(-lam * U[0] ** 2) / (math.pi * lam).sqrt())
        else:
            first = (one, U[0])
        mu, mv, mw = line(U[0], first), line(U[1], (one, U[1])), line(U[2], (one, U[2]))
        xi2 = self.K * hil
        out = []
        for a, b, c in powers:
            f = lambda i, j, k: mu[a + i] * mv[b + j] * mw[c + k]
            e = 0.5 * (f(2, 0, 0) + f(0, 2, 0) + f(0, 0, 2) + f(0, 0, 0) * xi2)
            out.append(torch.stack([rho * f(0, 0, 0), rho * f(1, 0, 0), rho * f(0, 1, 0), rho * f(0, 0, 1), rho * e], 1))
        return out

    def along(self, q, dq, powers, side=0):
        """Derivatives of `moments` along dq."""
        return torch.func.jvp(lambda x: self.moments(x, powers, side), (q,), (dq,))[1]

    def point_flux(self, ql, dl, qr, dr, dt):
        """F^n and dF/dt [N, 5] in the local frame from states [N, 5] and slopes [N, 3, 5] of both sides."""
        p = self.p
        axis = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
        second = [(2, 0, 0), (1, 1, 0), (1, 0, 1)]
        zero = [(0, 0, 0)]
        q0 = self.moments(ql, zero, 1)[0] + self.moments(qr, zero, -1)[0]
        dW = [self.along(ql, dl[:, d], zero, 1)[0] + self.along(qr, dr[:, d], zero, -1)[0] for d in range(3)]
        dWt = -sum(self.along(q0, dW[d], [axis[d]])[0] for d in range(3))
        E0 = self.moments(q0, [axis[0]])[0]
        E2 = self.along(q0, dWt, [axis[0]])[0]
        pres = lambda q: (GAMMA - 1) * (q[:, 4] - 0.5 * (q[:, 1:4] ** 2).sum(1) / q[:, 0])
        pl, pr, p0 = pres(ql), pres(qr), pres(q0)
        x = (pl - pr) / (pl + pr)
        jump = torch.where(x < 0, -x, x)
        tau = {0: lambda: torch.zeros_like(p0), 1: lambda: (0.01 + jump) * dt,
               2: lambda: p["mu"] / p0 + jump * dt}[p["tau_model"]]()[:, None]
        E1 = sum(self.along(q0, dW[d], [second[d]])[0] for d in range(3))
        if not p["flux_mode"]:
            Fn, Ft = E0 - tau * (E1 + E2), E2
            if p["Pr"] != 1.0:
                U = q0[:, 1:4] / q0[:, :1]
                u2 = (U * U).sum(1)

                def heat(F, m):
                    return (F[:, 4] - (U * F[:, 1:4]).sum(1) + 0.5 * u2 * F[:, 0] - U[:, 0] * m[:, 4] +
                            U[:, 0] * (U * m[:, 1:4]).sum(1) - 0.5 * U[:, 0] * u2 * m[:, 0])
                fix = 1 / p["Pr"] - 1
                add = lambda F, h: torch.cat([F[:, :4], (F[:, 4] + fix * h)[:, None]], 1)
                Fn, Ft = add(Fn, heat(Fn, q0)), add(Ft, heat(Ft, dWt))
            return Fn, Ft
        N0, N1, N2 = 0.0, 0.0, 0.0
        for q, dq, s in ((ql, dl, 1), (qr, dr, -1)):
            N0 = N0 + self.moments(q, [axis[0]], s)[0]
            N1 = N1 + sum(self.along(q, dq[:, d], [second[d]], s)[0] for d in range(3))
            dtq = -sum(self.along(q, dq[:, d], [axis[d]])[0] for d in range(3))
            N2 = N2 + self.along(q, dtq, [axis[0]], s)[0]

        def total(d):  # time integral of the flux over [0, d]
            e = torch.exp(-d / tau)
            om = 1 - e
            return (E0 * (d - tau * om) + E1 * (2 * tau * tau * om - tau * d * (1 + e)) +
                    E2 * (0.5 * d * d - tau * d + tau * tau * om) + N0 * tau * om +
                    N1 * (tau * d * e - 2 * tau * tau * om) - N2 * tau * tau * om)
        half, whole = total(0.5 * dt), total(dt)
        return (4 * half - whole) / dt, 4 * (whole - 2 * half) / dt ** 2

    def faces(self, Q, dt):
        """Face sums of F^n and dF/dt, [F, 5] each, out of the owner."""
        poly = self.polynomials(Q)
        vl, gl = self.evaluate(poly, self.o, self.dl)
        vr, gr = self.evaluate(poly, self.nbc, self.dr)
        flat = lambda x: x.reshape((-1,) + x.shape[2:])
        vl, gl, vr, gr = flat(vl), flat(gl), flat(vr), flat(gr)
        rep = lambda x: x[:, None].expand(-1, 4).reshape(-1)
        if self.p["gp_fallback"]:
            def safe(v, g, cell):
                bad = ~((v[:, 0] > 0) & (v[:, 0] * v[:, 4] > 0.5 * (v[:, 1:4] ** 2).sum(1)))
                return torch.where(bad[:, None], Q.T[cell], v), torch.where(bad[:, None, None], torch.zeros_like(g), g)
            vl, gl = safe(vl, gl, rep(self.o))
            vr, gr = safe(vr, gr, rep(self.nbc))
        plane = rep(self.plane)
        edge = plane >= 0
        if edge.any():
            vg, gg = self.ghost(vl, gl, plane.clamp(min=0))
            vr, gr = torch.where(edge[:, None], vg, vr), torch.where(edge[:, None, None], gg, gr)
        n1 = self.n.reshape(-1, 3)
        e = torch.nn.functional.one_hot(n1.abs().argmin(1), 3).double()
        n2 = torch.linalg.cross(n1, e)
        n2 = n2 / n2.norm(dim=1, keepdim=True)
        R = torch.stack([n1, n2, torch.linalg.cross(n1, n2)], 1)              # rows: local axes

        def turn(v):  # momentum into the local frame
            return torch.cat([v[..., :1], torch.einsum("...nj,...jk->...nk", v[..., 1:4].unsqueeze(-2),
                                                       R.transpose(1, 2) if v.dim() == 2 else
                                                       R.transpose(1, 2)[:, None]).squeeze(-2), v[..., 4:]], -1)
        gl, gr = R @ gl, R @ gr                                               # derivatives along the local axes
        out = []
        for F in self.point_flux(turn(vl), turn(gl), turn(vr), turn(gr), dt):
            F = torch.cat([F[:, :1], (F[:, 1:4].unsqueeze(1) @ R).squeeze(1), F[:, 4:]], 1)
            F = (F.reshape(-1, 4, 5) * self.w[..., None]).sum(1)
            if edge.any():
                kind = self.plane_kind(self.plane)
                on = ~self.inner
                keep = torch.nn.functional.one_hot(self.plane.clamp(min=0) % 3, 3).double()
                z = torch.zeros_like(F[:, :1])
                slip = torch.cat([z, F[:, 1:4] * keep, z], 1)
                pl = self.plane.clamp(min=0)
                uw = torch.tensor(self.p["wall_u"], dtype=torch.float64, device=self.dev)[pl]
                Tw = torch.tensor(self.p["wall_T"], dtype=torch.float64, device=self.dev)[pl]
                en = torch.where(Tw > 0, F[:, 4], (uw * F[:, 1:4]).sum(1))[:, None]
                F = torch.where((on & (kind == SLIP))[:, None], slip,
                                torch.where((on & (kind == NOSLIP))[:, None], torch.cat([z, F[:, 1:4], en], 1), F))
            out.append(F)
        return out

    def sums(self, F):
        """-sum_f s_f F_f of every cell, [nc, 5]."""
        s = torch.zeros(self.nc, 5, dtype=torch.float64, device=self.dev).index_add(0, self.o, -F)
        k = self.inner.nonzero()[:, 0]
        return s.index_add(0, self.nb[k], F[k])

    def residual(self, Q, dt):
        Fn, Ft = self.faces(Q, dt)
        return (self.sums(Fn) / self.vol[:, None]).T, (self.sums(Ft) / self.vol[:, None]).T

    def step(self, Q, dt):
        L, Lt = self.residual(Q, dt)
        _, Ls = self.residual(Q + dt / 2 * L + dt * dt / 8 * Lt, dt)
        return Q + dt * L + dt * dt / 6 * (Lt + 2 * Ls)

    def max_dt(self, Q, cfl):
        U2 = (Q[1:4] ** 2).sum(0) / Q[0] ** 2
        c = (GAMMA * (GAMMA - 1) * (Q[4] - 0.5 * Q[0] * U2) / Q[0]).sqrt()
        return cfl * float((self.hdt / (U2.sqrt() + c + 2 * self.p["mu"] / (Q[0] * self.hdt))).min())

    def implicit(self, Q, dt, kmax=3):
        """Backward Euler with the split flux Jacobian, kmax Jacobi iterations."""
        Fn, Ft = self.faces(Q, dt)
        res = self.sums(Fn) + 0.5 * dt * self.sums(Ft)
        q = Q.T
        other = lambda x: torch.where(self.inner[:, None], x[self.nbc], self.edge(x[self.o]))

        def speed(v):
            U = v[:, 1:4] / v[:, :1]
            p = (GAMMA - 1) * (v[:, 4] - 0.5 * v[:, 0] * (U * U).sum(1))
            return (U * self.fn).sum(1).abs() + (GAMMA * p / v[:, 0]).sqrt()

        def euler(v):
            un = (v[:, 1:4] * self.fn).sum(1) / v[:, 0]
            p = (GAMMA - 1) * (v[:, 4] - 0.5 * (v[:, 1:4] ** 2).sum(1) / v[:, 0])
            return torch.cat([(v[:, 0] * un)[:, None], v[:, 1:4] * un[:, None] + p[:, None] * self.fn,
                              ((v[:, 4] + p) * un)[:, None]], 1)
        qo, qn = q[self.o], other(q)
        r = 0.5 * torch.maximum(speed(qo), speed(qn)) * self.area
        k = self.inner.nonzero()[:, 0]
        D = (self.vol / dt).index_add(0, self.o, r).index_add(0, self.nb[k], r[k])[:, None]
        dq = res / D
        for _ in range(kmax):
            do = dq[self.o]
            dn = torch.where(self.inner[:, None], dq[self.nbc], self.edge(qo + do) - self.edge(qo))
            hS = 0.5 * self.area[:, None]
            to = hS * (euler(qn + dn) - euler(qn)) - r[:, None] * dn     # the owner's row sees the neighbour
            tn = -hS * (euler(qo + do) - euler(qo)) - r[:, None] * do    # and the neighbour's row the owner
            acc = torch.zeros_like(res).index_add(0, self.o, to).index_add(0, self.nb[k], tn[k])
            dq = (res - acc) / D
        return Q + dq.T

    def edge(self, v):
        """The boundary ghost's value of every face's owner state."""
        if not any(self.bc):
            return v
        return self.ghost(v, torch.zeros(v.shape[0], 3, 5, dtype=v.dtype, device=v.device), self.plane.clamp(min=0))[0]


@functools.lru_cache(maxsize=1)
def _plain(flow, layers, n, nx):
    return _Plain(dict(flow=flow, layers=layers, n=n, nx=nx))


def exact(case, seed):
    m = _mesh_dict(case)
    if len(m["cell_type"]) > EXACT_CELLS:
        return None
    P = _plain(case["flow"], case["layers"], case["n"], case["nx"])
    f = FLOWS[case["flow"]]
    q = _field(case, m, seed)
    Q = torch.from_numpy(q).to(P.dev)
    dt, call = P.max_dt(Q, f["cfl"]), case["call"]
    put = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(P.dev)
    if call == "vjp":
        g = I.normal_directions(q.shape, 2, seed + 3)
        x = Q.requires_grad_(True)
        return torch.autograd.grad(P.residual(x, dt), x, (put(g[0]), put(g[1])))[0]
    if call == "rollout":
        g = put(I.normal_directions(q.shape, 1, seed + 3)[0])
        xs = [Q]
        with torch.no_grad():
            for _ in range(case["steps"]):
                xs.append(P.step(xs[-1], dt))
        for x in reversed(xs[:-1]):  # one step's graph at a time
            x = x.detach().requires_grad_(True)
            (g,) = torch.autograd.grad(P.step(x, dt), x, g)
        return xs[-1], g
    with torch.no_grad():
        if call == "residual":
            return P.residual(Q, dt)
        for _ in range(case["steps"]):
            Q = P.implicit(Q, dt) if call == "implicit" else P.step(Q, P.max_dt(Q, f["cfl"]) if call == "adaptive" else dt)
        return (Q,)
