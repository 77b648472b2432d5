"""The wedge and the tet stage of a hybrid mesh run beside each other.

Bound: a step's stage pair may not take longer than its two stages one after
the other, with 15% for the launches and the joins (device times; FP64 meshes
whose stages take tens of microseconds each, so that the launches are a small
part).  Stages that do not share SMs queue behind each other and take about
1.4 to 1.7 times the sum on these meshes; sharing them they take 0.8 to 0.9."""
import pytest

from paper_1607_03399_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA not available", allow_module_level=True)

from paper_1607_03399_gb300.dg import Solver  # noqa: E402


@pytest.mark.parametrize("N", [1, 2, 3])
def test_stage_pair_takes_no_longer_than_its_stages(N):
    m = I.hybrid_mesh(20, 4, 2)  # 100 wedge blocks, 150 tet blocks
    S = Solver(m.VX, m.EToV, m.etype, N, precision="f64")
    S.set_fields(I.random_fields(S.total_nodes, 1))
    dt = S.stable_dt(0.4)
    S.stage_times(5)
    alone = min(sum(S.stage_times(40)) for _ in range(5))
    S.step(dt, 4)
    S.sync()
    pair = []
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(S.stream)
        S.step(dt, 8)
        e1.record(S.stream)
        e1.synchronize()
        pair.append(1e3 * e0.elapsed_time(e1) / 40)
    S.close()
    assert min(pair) <= 1.15 * alone, (min(pair), alone)


def _reverse_step_us(side, layers, N):
    """Device microseconds of a recorded reverse step, FP64."""
    m = I.bumpy_layered_mesh(side, layers)
    S = Solver(m.VX, m.EToV, m.etype, N, precision="f64")
    S.set_fields(I.random_fields(S.total_nodes, 1))
    dt = S.stable_dt(0.3)
    S.adjoint_bind()
    S.adjoint_reset()
    rec = S.new_record()
    S.step_record(dt, rec)
    times = []
    for _ in range(6):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(S.stream)
        for _ in range(4):
            S.adjoint_step_recorded(dt, rec)
        e1.record(S.stream)
        e1.synchronize()
        times.append(1e3 * e0.elapsed_time(e1) / 4)
    S.close()
    return min(times)


def test_reverse_stages_share_the_gpu_with_their_gradient_kernels():
    """A reverse step of 128 blocks takes no longer, per block, than one of 72:
    on neither mesh do the gradient kernels and the stages fill the GPU.  (Where
    they queue behind each other, the 128 blocks take 3 times as long as the 72
    instead of 1.2 times.)"""
    small, large = _reverse_step_us(12, 8, 2), _reverse_step_us(16, 8, 2)
    assert large <= small * 128 / 72, (small, large)
