"""The benchmark's accounting of a whole step and of the stage's arithmetic
(host only): a step of five stages moves 72 B per field-DOF in FP32, not 80,
since its first stage reads no residual and its last one stores none; the
operation count follows the stage kernel, which applies M^tri to two vectors
per slice and four per wedge."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


@pytest.mark.parametrize("N", [3, 4])
def test_step_bytes_per_dof(N):
    K = 524288
    nodes = K * (N + 1) ** 2 * (N + 2) // 2
    step = 5 * bench._mean_stage_bytes(bench._alg_bytes_per_stage(K, nodes), nodes)
    assert step == pytest.approx(72 * 4 * nodes + 5 * 64 * K, rel=1e-12)


def test_flops_of_the_n3_stage():
    # per slice of 10 nodes: D_t 320 and the divergence 50, M^tri 400 + 200,
    # lifts 250, quadrilateral faces 492, mass solve 760, strong part 60 + 704 + 90,
    # triangle fluxes 85, update 280
    per_slice = 320 + 50 + 600 + 250 + 492 + 760 + 854 + 85 + 280
    assert bench._flops_per_wedge(3) == pytest.approx(4 * per_slice + 150)
    assert bench._flops_per_wedge(3, "onthefly") - bench._flops_per_wedge(3) == pytest.approx(275 + 1000 / 3 + 150)
