"""What the benchmark derives from the launches of a call (no GPU)."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402
import paper_2512_18453_b200 as nv  # noqa: E402
from synth import point_set  # noqa: E402


@pytest.mark.parametrize("launches,separate,want", [
    (1, 3, (1, 1)),                                     # one kernel
    (3, 3, (1, 3)), (6, 6, (2, 3)),                     # three kernels, one and two chunks
    (2, 3, (1, 2)), (4, 6, (2, 2)), (6, 9, (3, 2))])    # product and output transform in one
def test_chunks_and_kernels_of_a_call(launches, separate, want):
    assert bench.chunks_and_kernels(launches, separate) == want


def test_kernel_classes_cover_the_measured_time_and_the_bytes_that_move():
    kms, x, v, m, y = [0.02, 0.05, 0.04], 50e6, 100e6, 200e6, 50e6
    classes = lambda per, kms, flops: bench.kernel_classes(per, kms, flops, x, v, m, y, 1700.0, 6500.0, "product", "input", "output")
    three = classes(3, kms, 30e9)
    assert [k[0] for k in three] == ["input", "product", "output"] and [k[1] for k in three] == kms
    assert three[2][3] == m + y
    two = classes(2, [0.02, 0.08, 0.0], 30e9)
    assert [k[0] for k in two] == ["input", "product_and_output"]
    assert two[1][1] == pytest.approx(0.08) and two[1][2:] == ("hbm", v + y)        # M does not move
    assert classes(2, kms, 300e9)[1][2:] == ("tensor", 300e9)
    assert classes(1, [0.0, 0.03, 0.0], 1e9) == [("one_kernel", 0.03, "hbm", x + y)]


def test_int8_launch_count_of_a_plan_without_a_device():
    plan = nv.Plan(4, point_set("dyadic", 4), nv.FP16_F32ACC, nv.COEF_FP32)
    # CUDA-core input transform (two passes and the scale between them, or the given scale and one), product, output
    assert plan.int8_launch_count(1, 20, 20, 32, 48, 0.0, nv.GEMM_TCGEN05) == 5
    assert plan.int8_launch_count(1, 20, 20, 32, 48, 0.02, nv.GEMM_TCGEN05) == 4
    assert plan.int8_launch_count(1, 20, 20, 24, 48) < 0                             # C % 16
    assert nv.Plan(4, point_set("nova", 4), nv.FP32).int8_launch_count(1, 20, 20, 32, 48) < 0
