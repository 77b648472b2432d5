"""The wedge stage with a CTA per block, in both of its triangle-request forms.

Meshes below the small-mesh limit run the stage with a CTA per block and slice,
so these are sized just above it (the limit is read from the dispatch rule).
Listed column by column, 8 layers to a column, every triangle-face neighbour
lies in its element's 32-element block; listed layer by layer, or under
tetrahedra, they do not, and the stage requests them from global memory.

Tolerances (relative L2, as everywhere in this suite): FP64 1e-12, FP32 1e-5
for a right-hand side and for two steps; gradients 1e-9 and 1e-5; the adjoint
identity 1e-12."""
import functools
import os
import re

import numpy as np
import pytest

from oracle import adjoint as OA
from oracle import reference as ORef
from oracle.dg import Solver as Oracle
from paper_1607_03399_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA not available", allow_module_level=True)

from paper_1607_03399_gb300 import adjoint as AD  # noqa: E402
from paper_1607_03399_gb300 import dg  # noqa: E402
from paper_1607_03399_gb300.dg import HostMesh, Solver  # noqa: E402

LAYERS = 8
TOL = {"f64": 1e-12, "f32": 1e-5}
ORDERS = [1, 2, 3, 4, 5]


def _limit(N):
    """CTAs up to which the small-mesh stage runs at order N."""
    src = os.path.join(os.path.dirname(os.path.abspath(dg.__file__)), "csrc", "kernels.cuh")
    with open(src) as f:
        low, high = re.search(r"constexpr int kWideCtas = N <= 3 \? (\d+) : (\d+);", f.read()).groups()
    return int(low if N <= 3 else high)


def _side(N):
    """Smallest footprint whose LAYERS-layer mesh has more CTAs than the limit."""
    side = 2
    while -(-2 * side * side * LAYERS // 32) * (N + 1) <= _limit(N):
        side += 1
    return side


@functools.lru_cache(maxsize=None)
def _column_mesh(N):
    m = I.bumpy_layered_mesh(_side(N), LAYERS)
    return m, I.random_material(m.K, 5, 1.0, 3.0, 0.8, 1.3)


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a, dtype=np.float64) - b) / np.linalg.norm(b))


def _triangle_neighbours_in_block(m, N):
    """Whether every bottom and top neighbour lies in the element's block."""
    nt, nq = (N + 1) * (N + 2) // 2, N + 1
    nb = np.asarray(HostMesh(m.VX, m.EToV, m.etype, N).face_neighbors()).reshape(m.K, 2 * nt + 3 * nq * nq)
    tri = nb[:, [0, nt]] // (nt * nq)
    own = np.arange(m.K)[:, None] // 32
    return bool(((nb[:, [0, nt]] < 0) | (tri // 32 == own)).all())


@functools.lru_cache(maxsize=None)
def _oracle(N, bc, flux):
    """State (32-bit values), its right-hand side and the state two steps on."""
    m, (c2, rho) = _column_mesh(N)
    O = Oracle(m.VX, m.EToV, m.etype, N, c2, rho, bc=bc, flux=flux)
    q = I.random_fields(O.conn.total_nodes, 11).astype(np.float32).astype(np.float64)
    dt = O.stable_dt(0.4)
    return q, dt, O.rhs(q), O.step(q, dt, 2) if bc == "rigid" else None


@pytest.mark.parametrize("N", ORDERS)
def test_meshes_are_of_the_two_forms(N):
    m, _ = _column_mesh(N)
    assert -(-m.K // 32) * (N + 1) > _limit(N)
    assert _triangle_neighbours_in_block(m, N)
    assert not _triangle_neighbours_in_block(I.layer_major(m, LAYERS)[0], N)


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("listed,mass", [("columns", "stored"), ("layers", "stored"), ("columns", "onthefly")])
@pytest.mark.parametrize("bc,flux", [("rigid", "upwind"), ("dirichlet", "central")])
@pytest.mark.parametrize("N", ORDERS)
def test_against_the_oracle(precision, listed, mass, bc, flux, N):
    m, (c2, rho) = _column_mesh(N)
    q, dt, rhs, stepped = _oracle(N, bc, flux)
    npw = (N + 1) * (N + 1) * (N + 2) // 2
    idx = np.arange(q.shape[1])
    if listed == "layers":
        m, perm = I.layer_major(m, LAYERS)
        c2, rho = c2[perm], rho[perm]
        idx = (perm[:, None] * npw + np.arange(npw)).ravel()
    S = Solver(m.VX, m.EToV, m.etype, N, c2, rho, bc=bc, flux=flux, precision=precision, mass=mass)
    qs = np.ascontiguousarray(q[:, idx]).astype(S.np_dtype)
    err = _rel(S.rhs(qs).cpu().numpy(), rhs[:, idx])
    assert err <= TOL[precision], err
    if stepped is not None:
        S.set_fields(qs)
        S.step(dt, 2)
        err = _rel(S.get_fields(), stepped[:, idx])
        assert err <= TOL[precision], err
    S.close()


@pytest.mark.parametrize("N", ORDERS)
def test_hybrid_against_the_oracle(N):
    m = I.hybrid_mesh(_side(N), LAYERS, 1)
    c2, rho = I.random_material(m.K, 7, 1.0, 3.0, 0.8, 1.3)
    O = Oracle(m.VX, m.EToV, m.etype, N, c2, rho)
    q = I.random_fields(O.conn.total_nodes, 12).astype(np.float32)
    ref = O.rhs(q.astype(np.float64))
    for precision in ("f32", "f64"):
        S = Solver(m.VX, m.EToV, m.etype, N, c2, rho, precision=precision)
        err = _rel(S.rhs(q.astype(S.np_dtype)).cpu().numpy(), ref)
        S.close()
        assert err <= TOL[precision], err


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("N", ORDERS)
def test_both_request_forms_give_the_same_bits(precision, N):
    """The column order and the layer order of one mesh, element by element,
    after three steps with a point source."""
    m, (c2, rho) = _column_mesh(N)
    ml, perm = I.layer_major(m, LAYERS)
    src = (0.413, 0.371, 0.523, 6.0, 0.05, 1.0)
    A = Solver(m.VX, m.EToV, m.etype, N, c2, rho, precision=precision, sources=[src])
    B = Solver(ml.VX, ml.EToV, ml.etype, N, c2[perm], rho[perm], precision=precision, sources=[src])
    npw = A.total_nodes // m.K
    idx = (perm[:, None] * npw + np.arange(npw)).ravel()
    q = I.random_fields(A.total_nodes, 7, A.np_dtype)
    dt = A.stable_dt(0.4)
    out = []
    for S, state in ((A, q), (B, np.ascontiguousarray(q[:, idx]))):
        S.set_fields(state)
        S.step(dt, 3)
        out.append(S.get_fields())
        S.close()
    assert np.array_equal(out[0][:, idx], out[1])


@pytest.mark.parametrize("precision,N", [("f32", n) for n in ORDERS] + [("f64", n) for n in ORDERS[:-1]])
def test_small_mesh_stage_gives_the_bits_of_the_slab_form(precision, N):
    """256 wedges solved alone (8 blocks: the small-mesh stage) and as the first
    part of a mesh above the limit, all of whose triangle neighbours lie in
    their blocks.  (FP64 at N = 5 has one form for all sizes.)"""
    part = I.bumpy_layered_mesh(4, LAYERS)
    whole = I.merge_meshes([part, _column_mesh(N)[0]], shift=(4.0, 0.0, 0.0))
    assert part.K // 32 * (N + 1) <= _limit(N) and _triangle_neighbours_in_block(whole, N)
    c2, rho = I.random_material(whole.K, 9, 1.0, 3.0, 0.5, 2.0)
    src = [(0.413, 0.371, 0.523, 6.0, 0.05, 2.0)]
    B = Solver(whole.VX, whole.EToV, whole.etype, N, c2, rho, precision=precision, sources=src)
    A = Solver(part.VX, part.EToV, part.etype, N, c2[:part.K], rho[:part.K], precision=precision, sources=src)
    q = I.random_fields(B.total_nodes, 3, B.np_dtype)
    dt = B.stable_dt(0.4)
    out = []
    for S in (A, B):
        S.set_fields(np.ascontiguousarray(q[:, :S.total_nodes]))
        S.step(dt, 3)
        out.append(S.get_fields())
        S.close()
    assert np.array_equal(out[0], out[1][:, :out[0].shape[1]])


@pytest.mark.parametrize("listed", ["columns", "layers"])
@pytest.mark.parametrize("N", [2, 3, 4])
def test_adjoint_step_is_the_transpose(listed, N):
    """<Phi v, W P mu_n> = <v, W P mu_{n-1}> in the oracle's energy weights W."""
    m, (c2, rho) = _column_mesh(N)
    if listed == "layers":
        m, perm = I.layer_major(m, LAYERS)
        c2, rho = c2[perm], rho[perm]
    S = Solver(m.VX, m.EToV, m.etype, N, c2, rho, precision="f64")
    O = Oracle(m.VX, m.EToV, m.etype, N, c2, rho)
    n = S.total_nodes
    rng = np.random.default_rng(5)
    v, mu = rng.standard_normal((4, n)), rng.standard_normal((4, n))
    dt = O.stable_dt(0.4)
    S.set_fields(v)
    S.step(dt, 1)
    phiv = S.get_fields()
    S.adjoint_bind()
    S.adjoint_set(mu, ORef.LSRK45_B[4] * mu)
    S.set_fields(v)
    S.adjoint_step(dt)
    mu0 = S.adjoint_get()
    S.close()
    Ms = O.element_mass_method()
    M = np.stack([Ms[k] for k in range(m.K)])
    scale = np.stack([1.0 / O.kappa] + [-np.asarray(O.rho)] * 3)  # W P per field and element

    def product(a, b):
        a, b = (x.reshape(4, m.K, -1) for x in (a, b))
        return float((scale * np.einsum("fki,fki->fk", a, (M @ b.transpose(1, 2, 0)).transpose(2, 0, 1))).sum())

    lhs, rhs = product(phiv, mu), product(v, mu0)
    # (rounding is relative to the terms: the norms of the two factors bound their sum)
    P = np.array([1, -1, -1, -1])[:, None]
    size = np.sqrt(product(P * phiv, phiv) * product(P * mu, mu))
    assert abs(lhs - rhs) <= 1e-12 * max(abs(lhs), size), (lhs, rhs, size)


@pytest.mark.parametrize("precision,tol", [("f64", 1e-9), ("f32", 1e-5)])
def test_gradient_against_the_oracle(precision, tol):
    """The oracle's reverse-mode gradient of 8 wedges, which here are a part of
    a mesh above the limit; the rest, which no wave reaches, has none."""
    part = I.cube_wavy_mesh(2, 1, 0.05)
    m = I.merge_meshes([part, _column_mesh(1)[0]], shift=(4.0, 0.0, 0.0))
    assert -(-m.K // 32) * 2 > _limit(1)
    rng = np.random.default_rng(0)
    kap, rho = rng.uniform(1, 2, m.K), rng.uniform(0.8, 1.3, m.K)
    src, recs = (0.4, 0.6, 0.5, 3.0, 0.2, 1.0), [(0.7, 0.3, 0.6), (0.2, 0.2, 0.3)]
    st = OA.Setup(part, 1, kap[:part.K], rho[:part.K], [src], recs, 0.02, 12)
    data = OA.traces(st) * 0.9 + 0.01
    pb = AD.Problem(m.VX, m.EToV, m.etype, 1, 0.02, 12, recs, shot_sources=[(0, *src)], precision=precision,
                    checkpoint_every=5)
    S = pb.solver(kap / rho, rho)
    d = torch.as_tensor(data[:, None, :], dtype=S.dtype, device=S.device)
    traces, ckp = AD.forward(S, pb)
    gk, gr = AD.reverse(S, pb, traces, d, ckp)
    S.close()
    g = np.concatenate([gk[:part.K], gr[:part.K]])
    ref = np.concatenate(OA.gradient_reverse(st, data))
    assert np.linalg.norm(g - ref) <= tol * np.linalg.norm(ref)
    assert not gk[part.K:].any() and not gr[part.K:].any()
