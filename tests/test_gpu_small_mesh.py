"""The small-mesh stage (a CTA per block and slice) against the large-mesh one.

A mesh solved alone (few enough blocks for the small-mesh stage at every
order) and the same elements inside a merged mesh large enough for the other
take different kernels; both accumulate every result in the same order with
explicit multiply-adds, so the states agree bit for bit.  The pieces have a
partly filled last block, triangle neighbours in another block and in tets,
and each its own point source."""
import numpy as np
import pytest

from paper_1607_03399_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA not available", allow_module_level=True)

from paper_1607_03399_gb300.dg import Solver  # noqa: E402


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("bc,flux,mass", [("rigid", "upwind", "stored"), ("dirichlet", "central", "stored"),
                                          ("rigid", "upwind", "onthefly")])
def test_small_mesh_stage_gives_the_same_bits(precision, N, bc, flux, mass):
    parts = [I.perturbed_layered_mesh(5, 3, 0.2, 1), I.hybrid_mesh(3, 2, 1), I.cube_wavy_mesh(24, 6, 0.01)]
    m = I.merge_meshes(parts, shift=(4.0, 0.0, 0.0))
    c2, rho = I.random_material(m.K, 9, 1.0, 3.0, 0.5, 2.0)
    src = [(4.0 * i + 0.15, 0.1, 0.3, 6.0, 0.05, 2.0) for i in (0, 1)]
    kw = dict(bc=bc, flux=flux, precision=precision, mass=mass)
    B = Solver(m.VX, m.EToV, m.etype, N, c2, rho, sources=src, **kw)
    q = np.random.default_rng(3).uniform(-1, 1, (4, B.total_nodes)).astype(B.np_dtype)
    B.set_fields(q)
    dt = B.stable_dt(0.4)
    B.step(dt, 3)
    whole = B.get_fields()
    B.close()
    node0 = 0
    for i, p in enumerate(parts[:2]):
        o = m.meta["offsets"][i]
        A = Solver(p.VX + np.array([4.0 * i, 0.0, 0.0]), p.EToV, p.etype, N, c2[o:o + p.K], rho[o:o + p.K],
                   sources=[src[i]], **kw)
        n = A.total_nodes
        A.set_fields(q[:, node0:node0 + n])
        A.step(dt, 3)
        got = A.get_fields()
        A.close()
        assert np.array_equal(got, whole[:, node0:node0 + n]), i
        node0 += n
