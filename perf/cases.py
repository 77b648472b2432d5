"""Measured workloads of the DG solver, through its public entry points.

A case is a plain dict; `prepare` builds what a user's program holds before the
call (mesh, material, solver, initial wavefield), `run` is one pass of that
program, `exact` the same pass in 64 bits by an independent torch
implementation of the scheme (no code of the library), `work` the bytes and
operations a pass cannot do without.

Kinds of pass:
  step      set_fields, `steps` LSRK45 steps (with receivers: one step and one
            receiver sample at a time, as a seismic run records its traces),
            get_fields
  rhs       one semi-discrete right-hand side of a given state
  energy    set_fields, the discrete energy
  gradient  forward run with stage records, then the adjoint sweep: traces and
            the gradient with respect to c^2 and rho
"""
from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

from paper_1607_03399_gb300 import inputs as I
from paper_1607_03399_gb300 import adjoint as ADJ
from paper_1607_03399_gb300.dg import Solver

DEFAULTS = dict(kind="step", mesh="layered", side=32, layers=16, tet_layers=0, order=3, precision="f32", ops="fp32",
                mass="stored", bc="rigid", flux="upwind", shots=1, receivers=0, steps=5, every=12)


def _case(name=None, **kw):
    c = dict(DEFAULTS, **kw)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # the plain method's accuracy case: 128 wavy wedges, FP64, rigid walls
        _case("cube128_n3_f64", mesh="cube", side=4, layers=4, precision="f64", steps=20),
        # a small FP32 mesh whose traces are recorded every step: launches and latency count
        _case("small_n2_traces", side=8, layers=4, order=2, receivers=16, steps=20),
        # the headline throughput workload: 524,288 layered wedges, N = 3
        _case("layered524k_n3", side=128, layers=16, steps=10),
        # the same mesh at N = 4
        _case("layered524k_n4", side=128, layers=16, order=4, steps=4),
        # the highest order, on a footprint whose column count is no multiple of the block
        _case("layered_n5", side=37, layers=11, order=5, steps=4),
        # wedges under tetrahedra, c drawn per element: 221,184 wedges + 221,184 tets
        _case("hybrid442k_n3", mesh="hybrid", side=96, layers=12, tet_layers=4, steps=6),
        # a shot batch with receivers, sampled every step
        _case("shots16_n3", side=32, layers=16, shots=16, receivers=64, steps=8),
        # many small meshes of uneven size merged into one solver, factors recomputed in the stage
        _case("merged16_n3_onthefly", mesh="merged", side=16, mass="onthefly", steps=8),
        # one right-hand side of a hybrid mesh in FP64 (time integrators of the caller's own)
        _case("rhs_hybrid_f64", kind="rhs", mesh="hybrid", side=24, layers=12, tet_layers=4, precision="f64"),
        # the energy of a large FP32 state, as an energy history asks for it
        _case("energy524k_n3", kind="energy", side=128, layers=16),
        # differentiation: 110,592 wedges, surface receivers, stage records
        _case("gradient110k_n3", kind="gradient", side=48, layers=24, receivers=256, steps=24, every=12),
        # BF16 tensor-core operator applies
        _case("layered131k_n3_bf16", side=64, layers=16, ops="bf16", steps=8),
    ]


def _count(c):
    """(wedges, tets) of one shot."""
    if c["mesh"] == "hybrid":
        return 2 * c["side"] ** 2 * c["layers"], 6 * c["side"] ** 2 * c["tet_layers"]
    if c["mesh"] == "tets":
        return 0, 6 * c["side"] ** 2 * c["layers"]
    if c["mesh"] == "merged":
        return sum(2 * s * s * l for s, l in _merged_sizes(c["side"])), 0
    return 2 * c["side"] ** 2 * c["layers"], 0


def _nodes(c):
    kw, kt = _count(c)
    n = c["order"]
    nt = (n + 1) * (n + 2) // 2
    return c["shots"] * (kw * nt * (n + 1) + kt * nt * (n + 3) // 3)


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    while True:
        kind = rng.choices(["step", "rhs", "energy", "gradient"], [6, 1, 1, 2])[0]
        c = dict(DEFAULTS, kind=kind)
        c["mesh"] = rng.choices(["layered", "hybrid", "merged", "tets", "cube"], [6, 3, 1, 1, 1])[0]
        c["side"] = logint(3, 128)
        c["layers"] = rng.randint(2, 32)
        c["tet_layers"] = rng.randint(1, 4) if c["mesh"] == "hybrid" else 0
        c["order"] = rng.choices([1, 2, 3, 4, 5], [1, 2, 5, 3, 1])[0]
        c["precision"] = rng.choices(["f32", "f64"], [4, 1])[0]
        c["mass"] = rng.choices(["stored", "onthefly"], [4, 1])[0]
        c["bc"] = rng.choices(["rigid", "dirichlet"], [4, 1])[0]
        c["flux"] = rng.choices(["upwind", "central"], [5, 1])[0]
        c["steps"] = rng.randint(2, 20)
        if kind == "step":
            if c["precision"] == "f32" and c["order"] <= 4:
                c["ops"] = rng.choices(["fp32", "bf16", "tf32", "tf32x3"], [6, 1, 1, 1])[0]
            c["shots"] = rng.choices([1, 2, 5, 16], [6, 1, 1, 1])[0]
            c["receivers"] = rng.choices([0, 16, 64], [3, 1, 1])[0]
        if kind == "gradient":
            c["precision"], c["flux"], c["mass"] = "f32", "upwind", "stored"
            c["mesh"] = rng.choice(["layered", "layered", "hybrid"])
            c["tet_layers"] = rng.randint(1, 4) if c["mesh"] == "hybrid" else 0
            c["receivers"], c["every"], c["shots"] = rng.choice([16, 64, 256]), rng.randint(3, 12), rng.choice([1, 1, 2])
            c["side"] = min(c["side"], 48)
        if c["mesh"] == "cube":
            c["side"], c["layers"] = rng.randint(2, 12), rng.randint(2, 12)
        elif c["mesh"] in ("hybrid", "tets"):
            c["side"] = min(c["side"], 48)
        elif c["mesh"] == "merged":
            c["side"] = rng.randint(3, 16)
        # no dearer than the largest listed passes: 4 N = 4 steps of 524,288 wedges in FP32
        budget = 1.5e8 if c["order"] < 5 else 4e7
        if c["precision"] == "f64":
            budget /= 20
        if kind == "gradient":
            budget /= 2
        if kind in ("rhs", "energy"):
            c["steps"] = 1
        if _nodes(c) * c["steps"] <= budget and _nodes(c) <= 4e7 and _nodes(c) >= 1000:
            return c


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------

def _merged_sizes(n):
    """Footprints 2x8x8 to 2x40x40 and 4 to 20 layers, spread over n meshes."""
    return [(8 + (32 * ((7 * i) % n)) // n, 4 + (16 * ((5 * i) % n)) // n) for i in range(n)]


@lru_cache(maxsize=None)
def _mesh_of(mesh, side, layers, tet_layers):
    if mesh == "cube":
        return I.cube_wavy_mesh(side, layers, 0.12 / layers)
    if mesh == "hybrid":
        return I.hybrid_mesh(side, layers, tet_layers)
    if mesh == "tets":
        return I.tet_box_mesh(side, layers)
    if mesh == "merged":
        return I.merge_meshes([I.bumpy_layered_mesh(s, l, seed0=100 * i) for i, (s, l) in enumerate(_merged_sizes(side))])
    return I.bumpy_layered_mesh(side, layers)


def _mesh(c):
    return _mesh_of(c["mesh"], c["side"], c["layers"], c["tet_layers"])


def _dev():
    return torch.device("cuda:0" if torch.cuda.is_available() else "cpu")


def _material(c, seed):
    """Per-element c^2 (layered by height, with a seeded variation) and rho."""
    m = _mesh(c)
    rng = np.random.default_rng(seed)
    z = m.VX[m.EToV[:, 0], 2]
    z = (z - z.min()) / max(float(np.ptp(z)), 1e-9)
    base = np.asarray([2.5, 2.0, 1.5, 1.0])[np.minimum((4 * z).astype(np.int64), 3)]
    cc = base * rng.uniform(0.9, 1.1, m.K)
    return cc * cc, rng.uniform(0.8, 1.2, m.K)


def _points(c, seed, n, top):
    """Seeded points inside the domain of the (first) mesh, near its top surface or anywhere in its upper half."""
    m = _mesh(c)
    V = m.VX if c["mesh"] != "merged" else I.bumpy_layered_mesh(*_merged_sizes(c["side"])[0], seed0=0).VX
    lo, hi = V.min(axis=0), V.max(axis=0)
    rng = np.random.default_rng(seed)
    xy = lo[:2] + (hi - lo)[:2] * rng.uniform(0.06, 0.94, (n, 2))
    fz = np.full(n, 0.99) if top else rng.uniform(0.55, 0.97, n)
    return [(float(x), float(y), float(lo[2] + (hi - lo)[2] * f)) for (x, y), f in zip(xy, fz)]


def _sources(c, seed):
    """(shot, x, y, z, f0, t0, amp), one Ricker source per shot, already ringing at t = 0."""
    if not c["receivers"]:
        return []
    return [(s, *p, 8.0, 0.01, 50.0) for s, p in enumerate(_points(c, seed + 1, c["shots"], False))]


def _wavefield(c, seed):
    """A smooth seeded state [shots][4][nodes]: Gaussian pulses in every field, and one per cent of noise."""
    dev = _dev()
    xyz = _coords(c)
    lo = xyz.amin(dim=1, keepdim=True)
    size = float((xyz - lo).amax())
    rng = np.random.default_rng(seed + 2)
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) + 3)
    real = torch.float64 if c["precision"] == "f64" else torch.float32
    q = torch.empty((c["shots"], 4, xyz.shape[1]), dtype=real, device=dev)
    for s in range(c["shots"]):
        for f in range(4):
            v = 0.01 * torch.randn(xyz.shape[1], dtype=real, device=dev, generator=gen)
            for _ in range(3):
                ctr = torch.tensor(rng.uniform(0.1, 0.9, 3), device=dev)[:, None] * (xyz.amax(dim=1, keepdim=True) - lo) + lo
                w = size * float(rng.uniform(0.1, 0.35))
                r2 = ((xyz - ctr) / w).square_().sum(dim=0)
                v += (float(rng.uniform(-1, 1)) * torch.exp(-r2)).to(real)
            q[s, f] = v
    return q if c["shots"] > 1 else q[0]


def _observed(c, seed):
    """Recorded traces [steps][shots][receivers] that the model's are compared with."""
    gen = torch.Generator(device=_dev())
    gen.manual_seed(int(seed) + 4)
    return 0.5 * torch.randn((c["steps"], c["shots"], c["receivers"]), device=_dev(), generator=gen)


def _inputs(c, seed):
    c2, rho = _material(c, seed)
    if c["kind"] == "gradient":  # the model parameters are held in 32 bits
        c2, rho = c2.astype(np.float32).astype(np.float64), rho.astype(np.float32).astype(np.float64)
    recs = _points(c, seed + 5, c["receivers"], True) if c["receivers"] else []
    return c2, rho, recs, _sources(c, seed)


def prepare(case, seed):
    c = dict(DEFAULTS, **case)
    m = _mesh(c)
    c2, rho, recs, srcs = _inputs(c, seed)
    st = {"case": c, "q": _wavefield(c, seed), "c2": c2, "rho": rho}
    if c["kind"] == "gradient":
        pb = ADJ.Problem(m.VX, m.EToV, m.etype, c["order"], 0.0, c["steps"], recs, srcs, c["shots"], bc=c["bc"],
                         flux=c["flux"], checkpoint_every=c["every"], stage_records=True)
        S = pb.solver(c2, rho)
        pb.dt = S.stable_dt(0.5)
        st.update(pb=pb, observed=_observed(c, seed))
    else:
        S = Solver(m.VX, m.EToV, m.etype, c["order"], c2, rho, bc=c["bc"], flux=c["flux"], precision=c["precision"],
                   mass=c["mass"], shots=c["shots"], shot_sources=srcs, receivers=recs, ops=c["ops"])
        st["dt"] = S.stable_dt(0.5)
    st["S"] = S
    return st


def run(st):
    c, S, q = st["case"], st["S"], st["q"]
    if c["kind"] == "rhs":
        return {"rhs": S.rhs(q)}
    if c["kind"] == "energy":
        S.set_fields(q)
        return {"energy": S.energy()}
    if c["kind"] == "gradient":
        pb = st["pb"]
        traces, ck = ADJ.forward(S, pb, q)
        gk, gr = ADJ.reverse(S, pb, traces, st["observed"], ck)
        g2, grho = ADJ.material_gradient(st["c2"], st["rho"], gk, gr)
        return {"traces": traces, "grad_c2": torch.as_tensor(g2, dtype=torch.float32),
                "grad_rho": torch.as_tensor(grho, dtype=torch.float32)}
    S.set_fields(q)
    out = {}
    if c["receivers"]:
        out["traces"] = torch.empty((c["steps"], c["shots"], c["receivers"]), dtype=S.dtype, device=S.device)
        for n in range(c["steps"]):
            S.step(st["dt"], 1)
            S.sample(out["traces"][n])
    else:
        S.step(st["dt"], c["steps"])
    out["fields"] = S.get_fields(device=True)
    return out


def work(case):
    """Per stage and field value: the state read and written and the low-storage residual likewise; per element about
    64 bytes of vertices, neighbours and material.  Operations: the method's, an FMA as two."""
    c = dict(DEFAULTS, **case)
    kw, kt = (c["shots"] * k for k in _count(c))
    n, rb = c["order"], 8 if c["precision"] == "f64" else 4
    nt, nq = (n + 1) * (n + 2) // 2, n + 1
    npt = nt * (n + 3) // 3
    dof = 4 * _nodes(c)
    f = kw * (nq * (8 * nt * nq + 24 * nt * nt + 60 * nt + 3 * (18 * nq + 8 * nq * nq)) + 30 * nt + 150)
    f += kt * (12 * npt * npt + 4 * nt * (30 + 4 * npt) + 40 * npt + 250)
    elem = 64 * (kw + kt)
    move = 2 * rb * dof  # one state in, one out
    if c["kind"] == "rhs":
        return {"bytes": move + elem, "flops": f}
    if c["kind"] == "energy":
        return {"bytes": rb * dof + elem, "flops": kw * 4 * (2 * nq * nt * nt + 2 * nq * nq * nt) + kt * 8 * npt * npt}
    stage = 2 * move + elem
    if c["kind"] == "gradient":
        # forward steps, and per reverse stage: x, mu, Q and r read, x and mu written
        return {"bytes": 5 * c["steps"] * (stage + 3 * move + elem), "flops": 5 * c["steps"] * 3 * f}
    return {"bytes": 5 * c["steps"] * stage + 2 * move, "flops": 5 * c["steps"] * f}


# ----------------------------------------------------------------------------
# the scheme in 64 bits: nodal DG for the acoustic system on vertically mapped
# wedges (weak t-derivatives and exact Jacobian-weighted mass) and affine tets
# ----------------------------------------------------------------------------

ALPHA = (0.0, 0.0, 0.0, 0.1002, 1.1332)  # warp & blend parameter of orders 1..5
RK_A = (0.0, -567301805773 / 1357537059087, -2404267990393 / 2016746695238, -3550918686646 / 2091501179385,
        -1275806237668 / 842570457699)
RK_B = (1432997174477 / 9575080441755, 5161836677717 / 13612068292357, 1720146321549 / 2090206949498,
        3134564353537 / 4481467310338, 2277821191437 / 14882151754819)
RK_C = (0.0, 1432997174477 / 9575080441755, 2526269341429 / 6820363962896, 2006345519317 / 3224310063776,
        2802321613138 / 2924317926251)


def _gll(n):
    p = np.polynomial.legendre.Legendre.basis(n)
    return np.concatenate([[-1.0], np.sort(p.deriv().roots().real), [1.0]])


def _lag1(nodes, x):
    """Values and derivatives of the Lagrange basis on `nodes` at x, by a Legendre Vandermonde matrix."""
    n = len(nodes) - 1
    leg = np.polynomial.legendre
    inv = np.linalg.inv(leg.legvander(nodes, n))
    dv = np.stack([leg.legval(x, leg.legder(np.eye(n + 1)[k])) if k else np.zeros_like(x) for k in range(n + 1)], 1)
    return leg.legvander(x, n) @ inv, dv @ inv


def _simplex_basis(dim, n, X):
    """Products of Legendre polynomials of total degree <= n at X and their derivatives along every axis."""
    leg = np.polynomial.legendre
    P = [leg.legvander(X[:, d], n) for d in range(dim)]
    D = [np.stack([leg.legval(X[:, d], leg.legder(np.eye(n + 1)[k])) if k else np.zeros(len(X)) for k in range(n + 1)], 1)
         for d in range(dim)]
    idx = [k for k in np.ndindex(*([n + 1] * dim)) if sum(k) <= n]

    def prod(der):
        return np.stack([np.prod([(D if d == der else P)[d][:, k[d]] for d in range(dim)], axis=0) for k in idx], 1)

    return prod(-1), [prod(d) for d in range(dim)]


def _warped(n, dim):
    """Barycentric coordinates of the warp & blend nodes of the triangle (dim 2: the tetrahedron's face) or the
    tetrahedron, first lattice index fastest."""
    alpha = ALPHA[n - 1]
    lat = np.array([k[::-1] for k in np.ndindex(*([n + 1] * dim)) if sum(k) <= n], dtype=np.float64)
    L = np.concatenate([(n - lat.sum(1))[:, None], lat], 1) / n
    equi = np.linspace(-1, 1, n + 1)
    disp = _gll(n) - equi

    def edge(a, b, c):
        """Displacement of L_b (and its negative of L_a) along edge (a, b) of a triangle with third vertex c."""
        x = L[:, b] - L[:, a]
        w = _lag1(equi, x)[0] @ disp
        inner = np.abs(x) < 1 - 1e-10
        w = np.where(inner, w / np.where(inner, 1 - x * x, 1.0), 0.0)
        return 2 * L[:, a] * L[:, b] * w * (1 + (alpha * L[:, c]) ** 2)

    def face(v):
        d = np.zeros_like(L)
        for a, b, c in (v, (v[1], v[2], v[0]), (v[2], v[0], v[1])):
            w = edge(a, b, c)
            d[:, b] += w
            d[:, a] -= w
        return d

    if dim == 2:
        return L + face((0, 1, 2))
    shift = np.zeros_like(L)
    for opp in range(4):
        v = tuple(i for i in range(4) if i != opp)
        tri = L[:, v[0]] * L[:, v[1]] * L[:, v[2]]
        den = np.prod([L[:, i] + 0.5 * L[:, opp] for i in v], axis=0)
        ok = den > 1e-10
        blend = np.where(ok, tri * (1 + (alpha * L[:, opp]) ** 2) / np.where(ok, den, 1.0), tri)
        shift += blend[:, None] * face(v)
    # on an edge the face blends degenerate: the plain edge displacement
    on_edge = (L < 1e-12).sum(1) >= 2
    for opp in range(4):
        v = tuple(i for i in range(4) if i != opp)
        at = on_edge & (L[:, opp] < 1e-12)
        shift[at] = face(v)[at]
    return L + shift


@lru_cache(maxsize=None)
def _ref(n):
    """Reference operators (numpy, 64 bits)."""
    gx, gw = np.polynomial.legendre.leggauss(n + 4)
    R = {"t": _gll(n)}
    E, _ = _lag1(R["t"], gx)
    R["D1"] = _lag1(R["t"], R["t"])[1]
    R["M1"] = E.T @ (gw[:, None] * E)
    R["Ma"] = E.T @ ((gw * (1 - gx) / 2)[:, None] * E)
    R["Mb"] = E.T @ ((gw * (1 + gx) / 2)[:, None] * E)
    inv1 = np.linalg.inv(R["M1"])
    R["ell"] = inv1[:, [0, n]]
    # triangle
    R["triL"] = lam = _warped(n, 2)
    xy = lam @ np.array([[-1.0, -1], [1, -1], [-1, 1]])
    V, dV = _simplex_basis(2, n, xy)
    R["triV"] = inv = np.linalg.inv(V)
    R["Dr"], R["Ds"] = dV[0] @ inv, dV[1] @ inv
    a, b = (g.ravel() for g in np.meshgrid(gx, gx, indexing="ij"))
    w2 = (gw[:, None] * gw[None, :]).ravel() * (1 - b) / 2
    pts = np.stack([(1 + a) * (1 - b) / 2 - 1, b], 1)
    B = _simplex_basis(2, n, pts)[0] @ inv
    bary = np.stack([-(pts[:, 0] + pts[:, 1]) / 2, (1 + pts[:, 0]) / 2, (1 + pts[:, 1]) / 2], 1)
    R["Mtri_a"] = np.stack([B.T @ ((w2 * bary[:, k])[:, None] * B) for k in range(3)])
    R["Mtri"] = B.T @ (w2[:, None] * B)
    # tetrahedron
    R["tetL"] = lam3 = _warped(n, 3)
    xyz = lam3 @ np.array([[-1.0, -1, -1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]])
    V3, dV3 = _simplex_basis(3, n, xyz)
    R["tetV"] = inv3 = np.linalg.inv(V3)
    R["tD"] = [d @ inv3 for d in dV3]
    a, b, c = (g.ravel() for g in np.meshgrid(gx, gx, gx, indexing="ij"))
    w3 = (gw[:, None, None] * gw[None, :, None] * gw[None, None, :]).ravel() * (1 - b) * (1 - c) ** 2 / 8
    p3 = np.stack([(1 + a) * (1 - b) * (1 - c) / 4 - 1, (1 + b) * (1 - c) / 2 - 1, c], 1)
    B3 = _simplex_basis(3, n, p3)[0] @ inv3
    R["tM"] = B3.T @ (w3[:, None] * B3)
    # face nodes: wedge bottom, top, the three vertical faces; tet faces by their vertices
    nt, nq = len(lam), n + 1
    edges = [[i for _, i in sorted((lam[i, k2], i) for i in range(nt) if abs(lam[i, k3]) < 1e-9)]
             for k2, k3 in ((1, 2), (2, 0), (0, 1))]
    R["edges"] = edges
    R["wf"] = [list(range(nt)), [n * nt + i for i in range(nt)]] + [[j * nt + i for j in range(nq) for i in e] for e in edges]
    R["tf"] = [[i for i in range(len(lam3)) if abs(lam3[i, o]) < 1e-9] for o in (3, 2, 0, 1)]
    return R


WF = ((0, 1, 2), (3, 4, 5), (0, 1, 4, 3), (1, 2, 5, 4), (2, 0, 3, 5))
TF = ((0, 1, 2), (0, 1, 3), (1, 2, 3), (0, 2, 3))


def _t(x, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=dtype, device=_dev())


def _split(m):
    kw = int((m.etype == I.WEDGE).sum())
    if not (m.etype[:kw] == I.WEDGE).all():
        raise ValueError("wedges come first")
    return kw, m.K - kw


def _coords(c):
    """Node coordinates [3][nodes], element by element."""
    m, R = _mesh(c), _ref(c["order"])
    kw, kt = _split(m)
    V, out = _t(m.VX), []
    if kw:
        P = V[_t(m.EToV[:kw], torch.int64)]
        lam, t = _t(R["triL"]), _t(R["t"])
        bot = torch.einsum("ia,kad->dki", lam, P[:, :3])
        top = torch.einsum("ia,kad->dki", lam, P[:, 3:])
        x = torch.einsum("j,dki->dkji", (1 - t) / 2, bot) + torch.einsum("j,dki->dkji", (1 + t) / 2, top)
        out.append(x.reshape(3, -1))
    if kt:
        P = V[_t(m.EToV[kw:, :4], torch.int64)]
        out.append(torch.einsum("ia,kad->dki", _t(R["tetL"]), P).reshape(3, -1))
    return torch.cat(out, 1)


def _face_pairs(m, kw, kt):
    """(element, face) of both sides of every interior face."""
    nv = m.VX.shape[0]
    keys, elem, face = [], [], []
    for faces, lo, hi in ((WF, 0, kw), (TF, kw, kw + kt)):
        E = _t(m.EToV[lo:hi], torch.int64)
        for f, v in enumerate(faces):
            if hi > lo:
                s = E[:, list(v)].sort(dim=1).values[:, :3]
                keys.append((s[:, 0] * nv + s[:, 1]) * nv + s[:, 2])
                elem.append(torch.arange(lo, hi, device=_dev()))
                face.append(torch.full((hi - lo,), f, device=_dev()))
    keys, elem, face = torch.cat(keys), torch.cat(elem), torch.cat(face)
    keys, at = keys.sort()
    i = torch.nonzero(keys[1:] == keys[:-1])[:, 0]
    return elem[at[i]], face[at[i]], elem[at[i + 1]], face[at[i + 1]]


class _Exact:
    """Semi-discrete operator of one mesh; material as differentiable tensors."""

    def __init__(self, c):
        self.c, m, R = c, _mesh(c), _ref(c["order"])
        self.R, self.m = R, m
        n = self.n = c["order"]
        self.kw, self.kt = kw, kt = _split(m)
        self.nt, self.nq, self.npt = len(R["triL"]), n + 1, len(R["tetL"])
        self.npw = self.nt * self.nq
        V = _t(m.VX)
        self._connect(m, R)
        if kw:
            P = V[_t(m.EToV[:kw], torch.int64)]
            x, y, z = P[:, :3, 0], P[:, :3, 1], P[:, :, 2]
            xr, xs, yr, ys = ((q[:, i] - q[:, 0]) / 2 for q in (x, y) for i in (1, 2))
            A = self.A = xr * ys - xs * yr
            h = z[:, 3:] - z[:, :3]
            self.met = ys / A, -xs / A, -yr / A, xr / A  # r_x, r_y, s_x, s_y
            t = _t(R["t"])
            zt = ((1 - t) / 2)[None, :, None] * z[:, None, :3] + ((1 + t) / 2)[None, :, None] * z[:, None, 3:]
            zr, zs = (zt[..., 1] - zt[..., 0]) / 2, (zt[..., 2] - zt[..., 0]) / 2
            self.tx = (yr[:, None] * zs - zr * ys[:, None])[..., None]
            self.ty = (zr * xs[:, None] - xr[:, None] * zs)[..., None]
            Mk = torch.einsum("ka,aij->kij", A[:, None] * h / 2, _t(R["Mtri_a"]))
            self.Mk = Mk
            self.Mkinv = torch.linalg.inv(Mk) if c["kind"] != "energy" else None
            self.nrm, self.jf = [], []
            for v, s in ((P[:, :3], -1.0), (P[:, 3:], 1.0)):
                cr = s * torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
                ln = cr.norm(dim=1)
                self.nrm.append(cr / ln[:, None])
                self.jf.append(ln / 4)
            self.edge_w = []
            for a, b in ((0, 1), (1, 2), (2, 0)):
                dx, dy = x[:, b] - x[:, a], y[:, b] - y[:, a]
                le = (dx * dx + dy * dy).sqrt()
                self.nrm.append(torch.stack([dy / le, -dx / le, torch.zeros_like(le)], 1))
                self.edge_w.append((le * h[:, a] / 4, le * h[:, b] / 4))
        if kt:
            P = V[_t(m.EToV[kw:, :4], torch.int64)]
            G = torch.stack([P[:, i] - P[:, 0] for i in (1, 2, 3)], 2) / 2  # d x_d / d r_m
            self.tJ = torch.linalg.det(G)
            self.tG = torch.linalg.inv(G)
            cen = P.mean(dim=1)
            self.tn, self.ts = [], []
            inv = np.linalg.inv(R["tM"])
            self.lift = []
            for f, v in enumerate(TF):
                cr = torch.linalg.cross(P[:, v[1]] - P[:, v[0]], P[:, v[2]] - P[:, v[0]])
                cr = cr * torch.sign(((P[:, v[0]] - cen) * cr).sum(1))[:, None]
                ln = cr.norm(dim=1)
                self.tn.append(cr / ln[:, None])
                self.ts.append(ln / 4 / self.tJ)
                # the face's own mass in the order of its nodes in the element
                lam = R["tetL"][R["tf"][f]][:, list(v)]
                B = _simplex_basis(2, n, lam @ np.array([[-1.0, -1], [1, -1], [-1, 1]]))[0] @ R["triV"]
                Bi = np.linalg.inv(B)
                self.lift.append(_t(inv[:, R["tf"][f]] @ (Bi.T @ R["Mtri"] @ Bi)))

    def _connect(self, m, R):
        """Per face type: local nodes, neighbour node (own node on a boundary), neighbour element."""
        kw, kt, dev = self.kw, self.kt, _dev()
        wf, tf = R["wf"], R["tf"]
        self.off = torch.cat([torch.arange(kw, device=dev) * self.npw, kw * self.npw + torch.arange(kt, device=dev) * self.npt])
        self.total = kw * self.npw + kt * self.npt
        if self.c["kind"] == "energy":
            return
        xyz = _coords(self.c)
        e1, f1, e2, f2 = _face_pairs(m, kw, kt)
        self.idm, self.idp, self.nbr = [], [], []
        for faces, lo, k in ((wf, 0, kw), (tf, kw, kt)):
            for f in faces:
                own = self.off[lo:lo + k, None] + torch.tensor(f, device=dev)[None, :]
                self.idm.append(own)
                self.idp.append(own.clone())
                self.nbr.append(torch.full((k,), -1, device=dev))

        def table(e, f):
            return torch.where(e < kw, f, f + 5)

        for ea, fa, eb, fb in ((e1, f1, e2, f2), (e2, f2, e1, f1)):
            ta, tb = table(ea, fa), table(eb, fb)
            for i in range(9):
                for j in range(9):
                    sel = torch.nonzero((ta == i) & (tb == j))[:, 0]
                    for part in sel.split(200000):
                        la = ea[part] - (kw if i >= 5 else 0)
                        lb = eb[part] - (kw if j >= 5 else 0)
                        a, b = self.idm[i][la], self.idm[j][lb]
                        d = sum((xyz[k][a][:, :, None] - xyz[k][b][:, None, :]) ** 2 for k in range(3))
                        self.idp[i][la] = torch.gather(b, 1, d.argmin(dim=2))
                        self.nbr[i][la] = eb[part]

    def jumps(self, q, i, elems, nrm, z):
        """Penalty fluxes (F_p, F_u) on the nodes of face table i."""
        qm, qp = q[:, self.idm[i]], q[:, self.idp[i]]
        nb = self.nbr[i]
        bnd = (nb < 0)[:, None]
        zm = z[elems]
        za = 0.5 * (zm + torch.where(nb < 0, zm, z[nb.clamp(min=0)]))[:, None]
        un = sum(nrm[:, d, None] * qm[1 + d] for d in range(3))
        up = sum(nrm[:, d, None] * qp[1 + d] for d in range(3))
        rigid = self.c["bc"] == "rigid"
        dp = torch.where(bnd, torch.zeros_like(un) if rigid else -2 * qm[0], qp[0] - qm[0])
        du = torch.where(bnd, -2 * un if rigid else torch.zeros_like(un), up - un)
        if self.c["flux"] == "upwind":
            return 0.5 * (dp / za - du), 0.5 * (za * du - dp)
        return -0.5 * du, -0.5 * dp

    def rhs(self, q, kappa, rho, src=()):
        """[4][total] -> d/dt; src: (element, vector over its nodes, amplitude)."""
        R, kw, kt = self.R, self.kw, self.kt
        z = (kappa * rho).sqrt()
        out = []
        if kw:
            Q = q[:, :kw * self.npw].reshape(4, kw, self.nq, self.nt)
            W = torch.zeros_like(Q)  # weak form, before the mass solve
            D1, Mt = _t(R["D1"]), _t(R["Mtri"])
            dt = torch.einsum("jm,fkmi->fkji", D1, Q)
            A = self.A[:, None, None]
            T = -torch.stack([self.tx * dt[1] + self.ty * dt[2] + A * dt[3], self.tx * dt[0], self.ty * dt[0], A * dt[0]])
            elems = torch.arange(kw, device=_dev())
            for f in (0, 1):
                Fp, Fu = self.jumps(q, f, elems, self.nrm[f], z)
                F = torch.stack([Fp] + [self.nrm[f][:, d, None] * Fu for d in range(3)]) * self.jf[f][:, None]
                T = T + _t(R["ell"][:, f])[None, None, :, None] * F[:, :, None, :]
            W = T @ Mt
            for e in range(3):
                Fp, Fu = (v.reshape(kw, self.nq, self.nq) for v in self.jumps(q, 2 + e, elems, self.nrm[2 + e], z))
                F = torch.stack([Fp] + [self.nrm[2 + e][:, d, None, None] * Fu for d in range(2)])
                ca, cb = (v[:, None, None] for v in self.edge_w[e])
                W[:3, :, :, R["edges"][e]] += ca * (F @ _t(R["Ma"])) + cb * (F @ _t(R["Mb"]))
            X = torch.einsum("fkji,kil->fkjl", W, self.Mkinv)
            rx, ry, sx, sy = (v[:, None, None] for v in self.met)
            Dr, Ds = _t(R["Dr"]).T, _t(R["Ds"]).T
            div = (rx * Q[1] + ry * Q[2]) @ Dr + (sx * Q[1] + sy * Q[2]) @ Ds
            pr, ps = Q[0] @ Dr, Q[0] @ Ds
            k, ir = kappa[:kw, None, None], 1 / rho[:kw, None, None]
            out.append(torch.stack([k * (X[0] - div), ir * (X[1] - rx * pr - sx * ps), ir * (X[2] - ry * pr - sy * ps),
                                    ir * X[3]]).reshape(4, -1))
        if kt:
            Q = q[:, kw * self.npw:].reshape(4, kt, self.npt)
            D = [_t(d).T for d in R["tD"]]
            gr = [[Q[f] @ d for d in D] for f in range(4)]

            def ddx(f, d):
                return sum(self.tG[:, r, d, None] * gr[f][r] for r in range(3))

            X = -torch.stack([ddx(1, 0) + ddx(2, 1) + ddx(3, 2), ddx(0, 0), ddx(0, 1), ddx(0, 2)])
            elems = torch.arange(kw, kw + kt, device=_dev())
            for f in range(4):
                Fp, Fu = self.jumps(q, 5 + f, elems, self.tn[f], z)
                F = torch.stack([Fp] + [self.tn[f][:, d, None] * Fu for d in range(3)]) * self.ts[f][:, None]
                X = X + F @ self.lift[f].T
            sc = torch.stack([kappa[kw:], 1 / rho[kw:], 1 / rho[kw:], 1 / rho[kw:]])[:, :, None]
            out.append((sc * X).reshape(4, -1))
        r = torch.cat(out, 1)
        for e, g, amp in src:
            o = int(self.off[e])
            add = torch.zeros_like(r)
            add[0, o:o + len(g)] = kappa[e] * amp * g
            r = r + add
        return r

    def locate(self, p):
        """(element, basis values, inverse mass times them) at a point; the lowest element on ties."""
        m, R, n, kw = self.m, self.R, self.n, self.kw
        best = None
        if kw:
            P = m.VX[m.EToV[:kw]]
            a, b = P[:, 1, :2] - P[:, 0, :2], P[:, 2, :2] - P[:, 0, :2]
            d = np.asarray(p[:2]) - P[:, 0, :2]
            det = a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]
            l1, l2 = (d[:, 0] * b[:, 1] - d[:, 1] * b[:, 0]) / det, (a[:, 0] * d[:, 1] - a[:, 1] * d[:, 0]) / det
            L = np.stack([1 - l1 - l2, l1, l2], 1)
            zb, zt = (L * P[:, :3, 2]).sum(1), (L * P[:, 3:, 2]).sum(1)
            t = (2 * p[2] - zb - zt) / (zt - zb)
            at = np.nonzero((L.min(1) >= -1e-12) & (np.abs(t) <= 1 + 1e-12))[0]
            if len(at):
                e = int(at[0])
                xy = (L[e] @ np.array([[-1.0, -1], [1, -1], [-1, 1]]))[None]
                lt = (_simplex_basis(2, n, xy)[0] @ R["triV"])[0]
                l1d = _lag1(R["t"], np.array([t[e]]))[0][0]
                g = np.outer(np.linalg.inv(R["M1"]) @ l1d, np.linalg.solve(self.Mk[e].cpu().numpy(), lt)).ravel()
                best = e, np.outer(l1d, lt).ravel(), g
        if best is None and self.kt:
            P = m.VX[m.EToV[kw:, :4]]
            L = np.linalg.solve(np.stack([P[:, i] - P[:, 0] for i in (1, 2, 3)], 2), (np.asarray(p) - P[:, 0])[:, :, None])[:, :, 0]
            L = np.concatenate([1 - L.sum(1, keepdims=True), L], 1)
            e = int(np.nonzero(L.min(1) >= -1e-12)[0][0])
            x = (L[e] @ np.array([[-1.0, -1, -1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]]))[None]
            lt = (_simplex_basis(3, n, x)[0] @ R["tetV"])[0]
            best = kw + e, lt, np.linalg.solve(R["tM"], lt) / float(self.tJ[e])
        return best[0], _t(best[1]), _t(best[2])

    def step(self, q, t, dt, kappa, rho, sources):
        res = torch.zeros_like(q)
        for a, b, cs in zip(RK_A, RK_B, RK_C):
            src = []
            for e, g, (f0, t0, amp) in sources:
                x = (math.pi * f0 * (t + cs * dt - t0)) ** 2
                src.append((e, g, amp * (1 - 2 * x) * math.exp(-x)))
            res = a * res + dt * self.rhs(q, kappa, rho, src)
            q = q + b * res
        return q

    def stable_dt(self, c2):
        """CFL 0.5: 1 / (c (N + 1)^2 (largest face area / volume)), the smallest over the elements."""
        ratio = []
        if self.kw:
            area = torch.stack([2 * j for j in self.jf] + [2 * (a + b) for a, b in self.edge_w], 1).amax(1)
            ratio.append(area / self.Mk.sum((1, 2)) / 2)  # the line's length is 2
        if self.kt:
            ratio.append(1.5 * torch.stack(self.ts, 1).amax(1))
        return 0.5 / float((c2.sqrt() * (self.n + 1) ** 2 * torch.cat(ratio)).max())

    def energy(self, q, kappa, rho):
        e = 0.0
        w = torch.stack([1 / kappa, rho, rho, rho])
        kw = self.kw
        if kw:
            Q = q[:, :kw * self.npw].reshape(4, kw, self.nq, self.nt)
            X = torch.einsum("jm,fkmi->fkji", _t(self.R["M1"]), torch.einsum("fkji,kil->fkjl", Q, self.Mk))
            e += 0.5 * float(((Q * X).sum((2, 3)) * w[:, :kw]).sum())
        if self.kt:
            Q = q[:, kw * self.npw:].reshape(4, self.kt, self.npt)
            e += 0.5 * float(((Q * (Q @ _t(self.R["tM"]))).sum(2) * self.tJ * w[:, kw:]).sum())
        return e


def exact(case, seed):
    c = dict(DEFAULTS, **case)
    if _nodes(c) * c["steps"] > 3.2e8:
        return None
    c2, rho, recs, srcs = _inputs(c, seed)
    q0 = _wavefield(c, seed).double().reshape(c["shots"], 4, -1)
    X = _Exact(c)
    c2, rho = _t(c2), _t(rho)
    if c["kind"] == "energy":
        return {"energy": X.energy(q0[0], rho * c2, rho)}
    if c["kind"] == "rhs":
        return {"rhs": X.rhs(q0[0], rho * c2, rho)}
    dt = X.stable_dt(c2)
    rec = [X.locate(p) for p in recs]
    at = [[(e, g, s[4:]) for s in srcs if s[0] == shot for e, _, g in [X.locate(s[1:4])]] for shot in range(c["shots"])]

    def sample(q):
        return torch.stack([(l * q[0, int(X.off[e]):int(X.off[e]) + len(l)]).sum() for e, l, _ in rec])

    if c["kind"] != "gradient":
        traces, fields = [], []
        for shot in range(c["shots"]):
            q, tr = q0[shot], []
            for n in range(c["steps"]):
                q = X.step(q, n * dt, dt, rho * c2, rho, at[shot])
                if rec:
                    tr.append(sample(q))
            fields.append(q)
            traces.append(tr)
        out = {"traces": torch.stack([torch.stack(t) for t in traces], 1)} if rec else {}
        out["fields"] = torch.stack(fields) if c["shots"] > 1 else fields[0]
        return out
    # reverse-mode differentiation of the steps, one step's graph at a time
    obs = _observed(c, seed).double()
    g2, grho = torch.zeros_like(c2), torch.zeros_like(rho)
    traces = torch.zeros_like(obs)
    for shot in range(c["shots"]):
        states = [q0[shot]]
        with torch.no_grad():
            for n in range(c["steps"]):
                states.append(X.step(states[-1], n * dt, dt, rho * c2, rho, at[shot]))
                traces[n, shot] = sample(states[-1])
        lam = torch.zeros_like(states[0])
        for n in reversed(range(c["steps"])):
            q = states[n + 1]
            for (e, l, _), r in zip(rec, traces[n, shot] - obs[n, shot]):
                lam[0, int(X.off[e]):int(X.off[e]) + len(l)] += r * l
            del q
            a, b, v = c2.clone().requires_grad_(), rho.clone().requires_grad_(), states[n].clone().requires_grad_()
            y = X.step(v, n * dt, dt, b * a, b, at[shot])
            lam, da, db = torch.autograd.grad(y, (v, a, b), lam)
            lam = lam.clone()
            g2 += da
            grho += db
    return {"traces": traces, "grad_c2": g2, "grad_rho": grho}
