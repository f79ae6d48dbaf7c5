"""GPU tests: a long call of a small grid is cut into launches that leave the GPU
to other streams now and then, and the cuts do not show in the fields."""
import numpy as np
import pytest

from paper_2309_10292_gb300 import gs
from tests.gpu_util import PAPER, need_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,dtype,arith,n", [(256, "f64", 0, 300), (128, "f64", gs.GS_ARITH_FXF, 1200), (201, "f32", 0, 2500)])
def test_no_launch_is_long(L, dtype, arith, n):
    torch = need_cuda()
    sim = gs.GrayScott(L, dtype=dtype, **dict(PAPER, noise=0.1, seed=3))
    if arith:
        sim.arith = arith
    sim.step(2)
    sim.sync()
    before = gs.gs_launch_count(sim.handle)
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    e[0].record()
    sim.step(n)
    e[1].record()
    sim.sync()
    launches = gs.gs_launch_count(sim.handle) - before
    assert 1 < launches < 50
    assert e[0].elapsed_time(e[1]) / launches < 100
    sim.close()


@pytest.mark.parametrize("arith", [gs.GS_ARITH_IEEE, gs.GS_ARITH_DS, gs.GS_ARITH_FX, gs.GS_ARITH_FXF])
def test_cut_calls_equal_the_plain_kernel(arith):
    # 573 = one launch of 572 steps and one of a single step (odd: the packed state changes buffers)
    need_cuda()
    sim, ref = (gs.GrayScott(128, dtype="f64", **dict(PAPER, noise=0.1, seed=4)) for _ in range(2))
    ref.set_plan(gs.GS_KERNEL_NAIVE)
    for s in (sim, ref):
        s.arith = arith
        s.step(573)
    for a, b in zip(sim.read(), ref.read()):
        np.testing.assert_array_equal(a, b)
