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


@pytest.mark.parametrize("L,dtype,named", [(64, "f32", True), (222, "f32", True), (300, "f32", True), (264, "f64", False)])
def test_cached_plan_of_a_tuner_without_the_default_plan_is_no_hit(tmp_path, L, dtype, named):
    # lines whose key does not name the default plan were tuned without it:
    # they count where it is one of the listed z-march plans only
    need_cuda()
    sims = [gs.GrayScott(L, dtype=dtype, **dict(PAPER, noise=0.1, seed=3)) for _ in range(2)]
    path = str(tmp_path / "plans.txt")
    sims[0].autotune_cached(path, steps_per_trial=1)
    key = open(path).read().split()[1]
    old = "/".join(key.split("/")[:7])
    assert old.endswith(f"/L{L}/{dtype}/ieee/periodic/noise") and (key != old) == named
    with open(path, "w") as f:
        f.write(f"gs-plan-v1 {old} {gs.GS_KERNEL_NAIVE} 0 0 0 1 0 99.0\n")
    best, hit = sims[1].autotune_cached(path, steps_per_trial=1)
    assert hit != named
    if not named:
        assert best["kernel"] == gs.GS_KERNEL_NAIVE
    best2, hit2 = sims[1].autotune_cached(path, steps_per_trial=1)
    assert hit2 and best2 == best
    for s in sims:
        s.close()
