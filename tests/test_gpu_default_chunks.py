"""The default z-march tile of the packed FP64 arithmetics cuts the grid into equal
z-chunks, and its steps equal the plain kernel's to the bit."""
import numpy as np
import pytest

from paper_2309_10292_gb300 import gs
from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu

ARITH = {"ds": gs.GS_ARITH_DS, "fx": gs.GS_ARITH_FX, "fxf": gs.GS_ARITH_FXF}


def sim(L, arith, held):
    s = gs.GrayScott(L, Du=0.2, Dv=0.1, F=0.02, k=0.048, dt=1.0, noise=0.1, seed=5, dtype="f64")
    s.arith = ARITH[arith]
    s.boundary = gs.GS_BOUNDARY_HELD if held else gs.GS_BOUNDARY_PERIODIC
    return s


@pytest.mark.parametrize("arith", ARITH)
@pytest.mark.parametrize("held", [False, True])
def test_no_short_last_chunk(arith, held):
    need_cuda()
    for L in (*range(162, 300, 4), 320, 354):
        s = sim(L, arith, held)
        tz = s.plan["tile_z"]
        assert 2 * (L - (L - 1) // tz * tz) >= tz, (L, tz)
        s.close()


@pytest.mark.parametrize("L,arith,held", [(162, "fx", False), (200, "fxf", True), (258, "fxf", False), (258, "ds", True)])
def test_steps_equal_the_plain_kernel(L, arith, held):
    need_cuda()
    got = []
    for plan in (gs.GS_KERNEL_AUTO, gs.GS_KERNEL_NAIVE):
        s = sim(L, arith, held)
        s.set_plan(plan)
        s.step(3)
        got.append(s.read())
        s.close()
    assert all(np.array_equal(a, b) for a, b in zip(*got))
