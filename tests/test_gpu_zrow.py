"""GPU tests of the whole-row z-march kernel: the default plan of FP32 grids
whose edge is no multiple of 4 and that are too large for the resident kernel.
"""
import numpy as np
import pytest

from paper_2309_10292_gb300 import gs
from tests.gpu_util import PAPER, need_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("held", [False, True])
@pytest.mark.parametrize("L,noise", [(203, 0.1), (205, 0.0), (222, 0.1), (226, 0.0), (255, 0.1), (301, 0.1), (302, 0.1),
                                     (418, 0.0), (529, 0.1)])
def test_rows_equal_the_plain_kernel(L, noise, held):
    # odd and even edges, an odd number of rows in the last tile, one and
    # several pairs of rows per tile, runs that end at the end of the field
    need_cuda()
    out = []
    for plain in (False, True):
        sim = gs.GrayScott(L, dtype="f32", **dict(PAPER, noise=noise, seed=2 ** 34 + 5))
        u, v = sim.tensors()
        u.copy_(_smooth(L, 1))
        v.copy_(_smooth(L, 2) * 0.4)
        if held:
            sim.boundary = gs.GS_BOUNDARY_HELD
        if plain:
            sim.set_plan(gs.GS_KERNEL_NAIVE)
        before = gs.gs_launch_count(sim.handle)
        sim.step(3)
        sim.step(2)
        assert gs.gs_launch_count(sim.handle) - before == (10 if plain and held else 5)
        out.append(sim.read())
        sim.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


def _smooth(L, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand((L, L, L), generator=g, device="cuda")


@pytest.mark.parametrize("L", [203, 222])
def test_rows_stay_inside_their_buffers(L):
    # the four buffers between guard bands of a NaN pattern: the bands keep
    # their bits, and nothing of them reaches a field
    torch = need_cuda()
    cells, band = L ** 3, 1024
    pitch = (cells + 63) // 64 * 64 + band
    mem = torch.full((4 * pitch + band,), float("nan"), device="cuda")
    mem.view(torch.int32).fill_(-1)
    bufs = [mem[band + i * pitch: band + i * pitch + cells] for i in range(4)]
    h = gs.gs_create_on(L, *(PAPER[k] for k in ("Du", "Dv", "F", "k", "dt")), 0.1, 3, "f32", *bufs,
                        stream=torch.cuda.current_stream())
    gs.gs_step(h, 3)
    gs.gs_sync(h)
    ref = gs.GrayScott(L, dtype="f32", **dict(PAPER, noise=0.1, seed=3))
    ref.set_plan(gs.GS_KERNEL_NAIVE)
    ref.step(3)
    got = np.empty((L, L, L), dtype=np.float32)
    for f, r in zip((gs.GS_U, gs.GS_V), ref.read()):
        np.testing.assert_array_equal(gs.gs_read(h, f, got), r)
    for i in range(4):
        bufs[i].view(torch.int32).fill_(-1)
    assert bool((mem.view(torch.int32) == -1).all())
    gs.gs_destroy(h)


def test_tuner_keeps_rows():
    L = 222
    need_cuda()
    sim = gs.GrayScott(L, dtype="f32", **dict(PAPER, noise=0.1, seed=3))
    best, trials = sim.autotune(steps_per_trial=12)
    assert best["kernel"] == gs.GS_KERNEL_AUTO and len(trials) == 2
    sim.close()
