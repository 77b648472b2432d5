"""The energy and receiver kernels over every order, precision and element
type, on meshes whose last 32-element block is partly filled.

Tolerances.  Energy, FP64: a block sums about Nq (Nt^2 / 2 + Nt) products per
field and element and the blocks are added in a tree, so the relative rounding
error stays below a few hundred unit roundoffs of 1.1e-16: 1e-12 leaves a
decade.  FP32 operators and vertices are rounded to 6e-8 each (the state is
passed to the oracle as rounded, sums are in double): 1e-6.  Samples are dot
products of Np entries: (Np + 2) unit roundoffs of the products' absolute sum."""
import numpy as np
import pytest

from oracle.adjoint import receiver_vector
from oracle.dg import Solver as Oracle
from paper_1607_03399_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA not available", allow_module_level=True)

from paper_1607_03399_gb300.dg import Solver  # noqa: E402

MESHES = {
    "wedges150": lambda: I.perturbed_layered_mesh(5, 3, 0.2, 1),  # 4 blocks and 22 elements
    "hybrid": lambda: I.hybrid_mesh(3, 2, 1),                     # 36 wedges, 54 tets
    "tets": lambda: I.tet_box_mesh(2, 2),                         # 48 tets
    "single": lambda: I.cube_wavy_mesh(1, 1, 0.0),                # 2 wedges
}


@pytest.mark.parametrize("meshname", list(MESHES))
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("precision,tol", [("f64", 1e-12), ("f32", 1e-6)])
def test_energy_every_order(meshname, N, precision, tol):
    m = MESHES[meshname]()
    c2, rho = I.random_material(m.K, 5, 1.0, 3.0, 0.5, 2.0)
    S = Solver(m.VX, m.EToV, m.etype, N, c2, rho, precision=precision)
    q = I.random_fields(S.total_nodes, N).astype(S.np_dtype)
    S.set_fields(q)
    E = S.energy()
    S.close()
    ref = Oracle(m.VX, m.EToV, m.etype, N, c2, rho).energy(q.astype(np.float64))
    assert abs(E - ref) <= tol * ref, (E, ref)


@pytest.mark.parametrize("meshname", ["wedges150", "hybrid", "tets"])
@pytest.mark.parametrize("N", [1, 3, 5])
@pytest.mark.parametrize("precision,u", [("f64", 2.0 ** -53), ("f32", 2.0 ** -24)])
def test_samples_every_order(meshname, N, precision, u):
    """Five receivers, two of them in one element, and two shots: a sample is the
    receiver's weights (themselves sampled, from states that are 1 at one node
    of every element) times the pressures of its element, in double."""
    m = MESHES[meshname]()
    lo, hi = m.VX.min(axis=0), m.VX.max(axis=0)
    pts = [tuple(lo + (hi - lo) * f) for f in ((0.21, 0.13, 0.17), (0.22, 0.13, 0.17), (0.71, 0.33, 0.84), (0.43, 0.92, 0.55),
                                              (0.11, 0.57, 0.95))]
    S = Solver(m.VX, m.EToV, m.etype, N, precision=precision, shots=2, receivers=pts)
    out = torch.empty((2, 5), dtype=S.dtype, device=S.device)

    def sample(q):
        S.set_fields(q)
        S.sample(out)
        S.sync()
        return out.cpu().numpy().astype(np.float64)

    O = Oracle(m.VX, m.EToV, m.etype, N)
    off = np.asarray(O.conn.offset)
    np_max = int(np.diff(off).max())
    ell = np.zeros((5, np_max))
    for n in range(np_max):
        q = np.zeros((2, 4, S.total_nodes), dtype=S.np_dtype)
        q[:, 0, (off[:-1] + n)[off[:-1] + n < off[1:]]] = 1
        got = sample(q)
        assert np.array_equal(got[0], got[1])
        ell[:, n] = got[0]
    q = np.stack([I.random_fields(S.total_nodes, s) for s in (1, 2)]).astype(S.np_dtype)
    got = sample(q)
    S.close()
    for r, x in enumerate(pts):
        k = receiver_vector(O, x)[0]
        p = q[:, 0, off[k]:off[k + 1]].astype(np.float64)
        w = ell[r, :p.shape[1]]
        assert abs(w.sum() - 1) < 1e-5  # the basis is a partition of unity
        bound = (len(w) + 2) * u * (np.abs(w) * np.abs(p)).sum(axis=1)
        assert (np.abs(got[:, r] - p @ w) <= bound).all(), (r, got[:, r], p @ w)
