"""Samples at receivers against the oracle's basis functions.

Bounds.  A sample is the dot product of the receiver's weights and the Np
pressures of its element: (Np + 3) unit roundoffs of the sum of |weight
pressure|, one of them the weight's own rounding.  The weights themselves come
from the receiver's reference coordinates, which library and oracle find by
iterations of their own to about 1e-12; a weight's slope in them is below 100
up to N = 5, so 1e-10 of the sum of |pressure|, in both precisions.  A receiver
taken at a wrong point is off by several per cent."""
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
    "wedges150": lambda: I.perturbed_layered_mesh(5, 3, 0.2, 1),
    "hybrid": lambda: I.hybrid_mesh(3, 2, 1),
    "tets": lambda: I.tet_box_mesh(2, 2),
}
FRACTIONS = ((0.21, 0.13, 0.17), (0.22, 0.13, 0.17), (0.71, 0.33, 0.84), (0.43, 0.92, 0.55), (0.11, 0.57, 0.95))


@pytest.mark.parametrize("meshname", list(MESHES))
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("precision,u", [("f64", 2.0 ** -53), ("f32", 2.0 ** -24)])
def test_samples_against_the_oracle(meshname, N, precision, u):
    m = MESHES[meshname]()
    lo, hi = m.VX.min(axis=0), m.VX.max(axis=0)
    pts = [tuple(lo + (hi - lo) * np.asarray(f)) for f in FRACTIONS]
    S = Solver(m.VX, m.EToV, m.etype, N, precision=precision, receivers=pts)
    q = I.random_fields(S.total_nodes, 4, S.np_dtype)
    out = torch.empty((1, len(pts)), dtype=S.dtype, device=S.device)
    S.set_fields(q)
    S.sample(out)
    S.sync()
    got = out.cpu().numpy().astype(np.float64)[0]
    S.close()
    O = Oracle(m.VX, m.EToV, m.etype, N)
    off = np.asarray(O.conn.offset)
    for r, x in enumerate(pts):
        k, ell = receiver_vector(O, x)
        p = q[0, off[k]:off[k + 1]].astype(np.float64)
        bound = (len(p) + 3) * u * float(np.abs(ell * p).sum()) + 1e-10 * float(np.abs(p).sum())
        assert abs(got[r] - ell @ p) <= bound, (r, got[r], ell @ p, bound)
