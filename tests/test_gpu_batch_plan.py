"""GPU tests: a small batch's default plan (equal shares of all rows per CTA) can
be named, survives calls that change nothing, and is reported before its first step."""
import numpy as np
import pytest

from paper_2309_10292_gb300 import gs
from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu
LS = [32, 48, 64] * 4


def make():
    need_cuda()
    return gs.GrayScottBatch(LS, np.linspace(0.02, 0.05, len(LS)), np.linspace(0.05, 0.065, len(LS)), noise=0.0, seed=3)


def shape(b):
    return b.info["grid"], b.info["items"]


def test_default_plan_keeps_its_name():
    a = make()
    shares = shape(a)
    a.step(3)
    assert shape(a) == shares  # the same kernel before the first step as after it
    b = make()
    for change in (lambda: b.set_depth(1), lambda: gs.gs_batch_set_plan(b.handle, 32, 8), lambda: (b.set_depth(3), b.set_depth(1)),
                   lambda: (gs.gs_batch_set_plan(b.handle, 16, 8), gs.gs_batch_set_plan(b.handle, 32, 8))):
        change()
        b.step(1)
        assert shape(b) == shares
        a.step(1)
    gs.gs_batch_set_plan(b.handle, 16, 8)
    b.step(3)
    assert shape(b) != shares
    a.step(b.t - a.t)
    for i in range(len(LS)):
        for x, y in zip(a.read(i), b.read(i)):
            np.testing.assert_array_equal(x, y)
    a.close()
    b.close()


def test_tuned_plan_applies_to_another_batch():
    a, b = make(), make()
    plan = a.autotune(steps_per_trial=48)
    gs.gs_batch_set_plan(b.handle, plan["tile_z"], plan["stages"])
    b.set_depth(plan["depth"])
    for x in (a, b):
        x.step(9)
    assert shape(a) == shape(b)
    for i in range(len(LS)):
        for x, y in zip(a.read(i), b.read(i)):
            np.testing.assert_array_equal(x, y)
    a.close()
    b.close()
