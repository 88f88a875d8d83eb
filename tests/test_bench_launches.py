"""The benchmark counts and times the kernels that a plan's ffeq_equalize launches."""
import pytest

import bench
from paper_1808_04473_gb300 import build as fbuild
from paper_1808_04473_gb300 import ffeq


@pytest.mark.parametrize("precision,arch,shape,kind", [
    (ffeq.FP32, ffeq.FD, (0, 0), "formed"), (ffeq.FP32, ffeq.FD, (1, 1), None), (ffeq.FP32, ffeq.PD, (0, 0), None),
    (ffeq.BF16X3, ffeq.FD, (6, 2), "streamed"), (ffeq.BF16X3, ffeq.FD, (5, 2), None),
    (ffeq.BF16X3, ffeq.PD, (6, 0), "streamed"), (ffeq.BF16X3, ffeq.FD, (0, 0), None),
])
def test_fused_kernel_of_the_headline_plans(precision, arch, shape, kind):
    fbuild.build()
    plan = ffeq.ffeq_plan_create(256, 16, 8, 1200, 14, arch=arch, precision=precision, llr_bits=4)
    ffeq.ffeq_plan_set_tuning(plan, shape)
    assert bench.fused_kernel(ffeq, plan) == kind
