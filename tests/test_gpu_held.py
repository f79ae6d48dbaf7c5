"""GPU test of the held outer layer written by the z-march kernel itself.

The plain kernel (followed by a copy of the six faces) is the reference; the
fields must be equal bit for bit for tiles that divide the grid and ragged
ones, chunks that march up and down, and a single tile holding every face.
"""
import numpy as np
import pytest

from paper_2309_10292_gb300 import gs
from tests.gpu_util import PAPER, need_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("noise", [0.0, 0.1])
@pytest.mark.parametrize("L,tile", [(4, (4, 4, 4)), (8, (8, 3, 3)), (20, (16, 7, 6)), (48, (32, 5, 7)), (64, (64, 8, 32)),
                                    (264, (132, 12, 32))])
def test_zmarch_holds_the_outer_layer(L, tile, noise, dtype):
    need_cuda()
    rng = np.random.default_rng(L)
    u, v = rng.uniform(0, 1, (L, L, L)), rng.uniform(0, 0.5, (L, L, L))
    got = []
    for kernel, t in ((gs.GS_KERNEL_ZMARCH, tile), (gs.GS_KERNEL_NAIVE, (0, 0, 0))):
        sim = gs.GrayScott(L, dtype=dtype, **dict(PAPER, noise=noise, seed=6))
        sim.boundary = gs.GS_BOUNDARY_HELD
        sim.set_plan(kernel, *t)
        sim.write(u, v)
        before = gs.gs_launch_count(sim.handle)
        sim.step(5)
        assert gs.gs_launch_count(sim.handle) - before == (5 if kernel == gs.GS_KERNEL_ZMARCH else 10)
        got.append(sim.read())
        sim.close()
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
    for f, g in zip(got[0], (u, v)):
        for ax in range(3):
            for e in (0, L - 1):
                np.testing.assert_array_equal(f.take(e, ax), g.take(e, ax).astype(f.dtype))
