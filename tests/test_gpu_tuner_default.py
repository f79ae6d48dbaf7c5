"""GPU tests: the tuner tries the default plan of every grid, so the plan that it
keeps is no slower than an untouched grid's."""
import pytest

from paper_2309_10292_gb300 import gs
from tests.gpu_util import PAPER, need_cuda

pytestmark = pytest.mark.gpu
TILE = ("tile_x", "tile_y", "tile_z", "stages")


@pytest.mark.parametrize("L,dtype,arith,held", [(320, "f32", 0, False), (300, "f32", 0, True), (192, "f64", gs.GS_ARITH_FXF, False),
                                                (100, "f64", gs.GS_ARITH_DS, True), (264, "f64", 0, False), (512, "f32", 0, False)])
def test_default_tile_is_among_the_trials(L, dtype, arith, held):
    need_cuda()
    sim = gs.GrayScott(L, dtype=dtype, **dict(PAPER, noise=0.1, seed=3))
    if arith:
        sim.arith = arith
    if held:
        sim.boundary = gs.GS_BOUNDARY_HELD
    default = sim.plan
    assert default["kernel"] == gs.GS_KERNEL_ZMARCH
    best, trials = sim.autotune(steps_per_trial=12)
    same = [t for t in trials if t["kernel"] == gs.GS_KERNEL_ZMARCH and all(t[k] == default[k] for k in TILE)]
    assert len(same) == 1
    assert best["us_per_step"] <= same[0]["us_per_step"]
    sim.close()
