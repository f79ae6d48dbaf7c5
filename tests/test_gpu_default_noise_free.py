"""The default z-march tile of large FP32 grids without noise: 128 x 8 x 64 cells
where 128-cell tiles waste little of a row, the evenly cut one elsewhere."""
import pytest

from paper_2309_10292_gb300 import gs
from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def sim(L, noise):
    return gs.GrayScott(L, Du=0.2, Dv=0.1, F=0.02, k=0.048, dt=1.0, noise=noise, seed=5)


@pytest.mark.parametrize("L,noise,tile", [(512, 0.0, (256, 6, 32, 6)), (600, 0.0, (200, 8, 32, 6)), (604, 0.0, (128, 8, 64, 4)),
                                          (604, 0.1, (204, 8, 32, 6)), (648, 0.0, (216, 7, 32, 6)), (768, 0.0, (128, 8, 64, 4))])
def test_tile(L, noise, tile):
    need_cuda()
    s = sim(L, noise)
    p = s.plan
    s.close()
    assert (p["tile_x"], p["tile_y"], p["tile_z"], p["stages"]) == tile


@pytest.mark.parametrize("held", [False, True])
def test_steps_equal_the_plain_kernel(held):
    torch = need_cuda()
    got = []
    for plan in (gs.GS_KERNEL_AUTO, gs.GS_KERNEL_NAIVE):
        s = sim(604, 0.0)
        s.boundary = gs.GS_BOUNDARY_HELD if held else gs.GS_BOUNDARY_PERIODIC
        s.set_plan(plan)
        s.step(2)
        got.append([t.clone() for t in s.tensors()])
        s.sync()
        s.close()
    assert all(torch.equal(a, b) for a, b in zip(*got))
