"""GPU tests of the grid barrier's bounded wait: with a wait budget of a
nanosecond some CTA gives up within a few hundred steps, the error is reported,
and the object works again afterwards."""
import numpy as np
import pytest

from paper_2309_10292_gb300 import gs
from tests.gpu_util import PAPER, need_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,dtype,arith,held", [(64, "f32", 0, False), (96, "f32", 0, True), (33, "f64", 0, False),
                                                (96, "f64", gs.GS_ARITH_FXF, False), (48, "f64", gs.GS_ARITH_DS, True)])
def test_grid_reports_and_recovers(L, dtype, arith, held):
    need_cuda()
    sim, ref = (gs.GrayScott(L, dtype=dtype, **dict(PAPER, noise=0.1, seed=6)) for _ in range(2))
    ref.set_plan(gs.GS_KERNEL_NAIVE)
    for s in (sim, ref):
        s.arith = arith
        if held:
            s.boundary = gs.GS_BOUNDARY_HELD
    gs.gs_set_fault(sim.handle, 0, 1)
    sim.step(2000)
    with pytest.raises(gs.GsError) as e:
        sim.sync()
    assert e.value.status == gs.GS_ETIMEOUT
    gs.gs_set_fault(sim.handle, 0, 2_000_000_000)
    for s in (sim, ref):
        s.init()
        s.step(7)
    for a, b in zip(sim.read(), ref.read()):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_batch_reports_and_recovers(dtype):
    need_cuda()
    Ls = [32, 48, 64]
    a, b = (gs.GrayScottBatch(Ls, [0.02] * 3, [0.05] * 3, noise=0.1, seed=6, dtype=dtype) for _ in range(2))
    gs.gs_batch_set_plan(b.handle, 8, 4)
    gs.gs_batch_set_fault(a.handle, 0, 1)
    a.step(2000)
    with pytest.raises(gs.GsError) as e:
        a.sync()
    assert e.value.status == gs.GS_ETIMEOUT
    gs.gs_batch_set_fault(a.handle, 0, 2_000_000_000)
    for x in (a, b):
        x.init()
        x.step(7)
    for i in range(3):
        for x, y in zip(a.read(i), b.read(i)):
            np.testing.assert_array_equal(x, y)
