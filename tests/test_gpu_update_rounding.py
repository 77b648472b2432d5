"""The fused Runge-Kutta update in FP32 carries no scale error of its own.

In a medium with one c^2 and one rho a factor kappa dt (or dt / rho) that is
rounded to FP32 once would scale the update of every node by the same error,
where roundings node by node average out.  The first stage of a step gives
q_1 = q_0 + b_1 dt r with the recorded right-hand side r; where q_0 is zero
(the velocities under a state of pressure alone, the pressure under one of
velocity alone) the common part of the error is the regression of q_1 on
b_1 dt r, less one.  dt is an FP32 number and the material is chosen so that
the rounding errors of both products exceed 4e-8.

Bound: what independent roundings leave in the regression.  The recorded r and
the products of the update (by the material, dt and b_1) are each rounded to
within 2^-24 of their size (standard deviation 2^-24 / sqrt 3): six standard
deviations of four such errors, which must be below a quarter of the error
looked for."""
import numpy as np
import pytest

from paper_1607_03399_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA not available", allow_module_level=True)

from paper_1607_03399_gb300.dg import Solver  # noqa: E402

B1 = float(np.float32(1432997174477 / 9575080441755))

# whole 32-element blocks of one type, so that the packed records have no padding
MESHES = {
    "wedges2304": lambda: I.bumpy_layered_mesh(12, 8),  # 72 blocks
    "wedges1024": lambda: I.bumpy_layered_mesh(8, 8),   # 32 blocks
    "tets1536": lambda: I.tet_box_mesh(8, 4),
}


def _product_error(v, dt):
    """Relative error of the FP32 product of two FP32 numbers."""
    return float(np.float32(v) * np.float32(dt)) / (float(np.float32(v)) * float(np.float32(dt))) - 1.0


def _material(dt):
    """(c^2, rho) whose kappa dt and dt / rho are both rounded by more than 4e-8."""
    for i in range(4000):
        rho = 0.9 + 1e-4 * i
        if abs(_product_error(1.0 / rho, dt)) < 4e-8:
            continue
        for j in range(4000):
            c2 = 1.5 + 1e-4 * j
            if abs(_product_error(rho * c2, dt)) > 4e-8:
                return c2, rho
    raise AssertionError("no material found")


@pytest.mark.parametrize("meshname", list(MESHES))
@pytest.mark.parametrize("N", [2, 3, 4])
def test_update_has_no_common_scale_error(meshname, N):
    m = MESHES[meshname]()
    assert m.K % 32 == 0
    S = Solver(m.VX, m.EToV, m.etype, N, np.full(m.K, 2.0), np.ones(m.K), precision="f32")
    dt = float(np.float32(0.4 * S.stable_dt(1.0)))
    S.close()
    c2, rho = _material(dt)
    S = Solver(m.VX, m.EToV, m.etype, N, np.full(m.K, c2), np.full(m.K, rho), precision="f32")
    rec = S.new_record()
    n, fb = 4 * S.total_nodes, S.field_bytes // 4
    fields = I.random_fields(S.total_nodes, 3, np.float32)
    for zero, scale in ((slice(0, 1), rho * c2), (slice(1, 4), 1.0 / rho)):
        q = fields.copy()
        q[zero] = 0
        S.set_fields(q)
        S.step_record(dt, rec)
        S.sync()
        v = rec.view(torch.float32).double()
        q0, q1, r = (v[k * fb:k * fb + n].reshape(-1, 4)[:, zero] for k in (0, 1, 5))
        assert float(q0.abs().max()) == 0
        d = B1 * dt * r
        dd = float((d * d).sum())
        slope = float((q1 * d).sum()) / dd - 1.0
        bound = 6 * 2.0 ** -24 / 3 ** 0.5 * 2 * float((d ** 4).sum()) ** 0.5 / dd
        assert bound < 0.25 * abs(_product_error(scale, dt)), bound
        assert abs(slope) <= bound, (slope, bound, _product_error(scale, dt))
    S.close()
