"""Stages launched as programmatic dependents against ordinary launches.

dg_step's captured steps launch the stages of small wedge meshes as
programmatic dependents; dg_step_record_chain makes the same stages one
ordinary launch after another.  The kernels are the same, so the states agree
bit for bit.  Sizes: a few blocks and about one wave (a CTA per block and
slice), and, where the form with a CTA per block takes over below 76 blocks,
a mesh of that form."""
import numpy as np
import pytest

from paper_1607_03399_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA not available", allow_module_level=True)

from paper_1607_03399_gb300.dg import Solver  # noqa: E402

# (side, layers): 2 side^2 layers wedges, listed column by column
SIZES = [(4, 4), (7, 8), (12, 8), (9, 8), (10, 11)]


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("side,layers", SIZES)
@pytest.mark.parametrize("mass", ["stored", "onthefly"])
def test_captured_steps_give_the_bits_of_ordinary_launches(precision, N, side, layers, mass):
    m = I.bumpy_layered_mesh(side, layers)
    c2, rho = I.random_material(m.K, 5, 1.0, 3.0, 0.8, 1.3)
    src = (0.413, 0.371, 0.523, 6.0, 0.05, 1.0)
    S = Solver(m.VX, m.EToV, m.etype, N, c2, rho, precision=precision, sources=[src], mass=mass)
    q = I.random_fields(S.total_nodes, 7, S.np_dtype)
    dt = S.stable_dt(0.4)
    S.set_fields(q)
    recs = [S.new_record() for _ in range(6)]
    S.step_record_chain(dt, recs)
    ref = S.get_fields()
    for _ in range(3):
        S.set_fields(q)
        S.step(dt, 6)
        got = S.get_fields()
        assert np.array_equal(got, ref)
    S.close()
