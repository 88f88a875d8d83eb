"""Which plans run ffeq_equalize as one kernel (host side): the default shape by its
rule, shape 6, and nothing else; setting a shape ends the default's kernel."""
import pytest

from paper_1808_04473_gb300 import build as fbuild
from paper_1808_04473_gb300 import ffeq


@pytest.fixture(scope="module", autouse=True)
def built():
    fbuild.build()
    return ffeq.lib()


FD = dict(B=64, U=8, C=4, n_sc=10, n_sym=3, arch=ffeq.FD)


@pytest.mark.parametrize("kw,single", [
    ({}, True), (dict(precision=ffeq.TF32X3), True), (dict(precision=ffeq.FP16X3), True),
    (dict(equalizer=ffeq.ZF), True), (dict(precision=ffeq.BF16X3), False), (dict(arch=ffeq.PD), False),
    (dict(C=1), False), (dict(equalizer=ffeq.MRC), False), (dict(refine=1), False),
])
def test_default_shape(kw, single):
    assert ffeq.ffeq_plan_single_launch(ffeq.ffeq_plan_create(**{**FD, **kw})) == single


def test_a_set_shape_runs():
    plan = ffeq.ffeq_plan_create(**FD)
    for shape, single in (((1, 0), False), ((0, 0), True), ((0, 1), False), ((1, 2), False), ((2, 0), False)):
        ffeq.ffeq_plan_set_tuning(plan, shape)
        assert ffeq.ffeq_plan_single_launch(plan) == single, shape
    plan = ffeq.ffeq_plan_create(**{**FD, "precision": ffeq.BF16X3})
    for shape, single in (((5, 0), False), ((6, 0), True), ((7, 0), False)):
        ffeq.ffeq_plan_set_tuning(plan, shape)
        assert ffeq.ffeq_plan_single_launch(plan) == single, shape


def test_arguments():
    plan = ffeq.ffeq_plan_create(**FD)
    assert ffeq.lib().ffeq_plan_single_launch(plan.handle, None) == 1
    assert ffeq.lib().ffeq_plan_single_launch(None, None) == 1
