"""GPU tests of the default plan at the ends of its rules: the tiles of every
edge, the largest whole-row edges, and many steps of the split between a brick's
shell and its inner rows."""
import numpy as np
import pytest

from paper_2309_10292_gb300 import gs
from tests.gpu_util import PAPER, need_cuda

pytestmark = pytest.mark.gpu


def test_every_default_tile_is_a_valid_one():
    # a tile that the z-march rejects would fall silently to the plain kernel
    torch = need_cuda()
    biggest = 1624
    buf = torch.empty(biggest ** 3, dtype=torch.float32, device="cuda")
    for L in range(260, biggest + 1, 4):
        h = gs.gs_create_on(L, 0.2, 0.1, 0.02, 0.048, 1.0, 0.1, 3, "f32", buf, buf, buf, buf, stream=torch.cuda.current_stream())
        for held in (gs.GS_BOUNDARY_PERIODIC, gs.GS_BOUNDARY_HELD):
            gs.gs_set_boundary(h, held)
            assert gs.gs_get_plan(h)["kernel"] == gs.GS_KERNEL_ZMARCH, L
        gs.gs_destroy(h)
    for L in list(range(82, 600, 2)) + list(range(600, 1280, 46)):
        h = gs.gs_create_on(L, 0.2, 0.1, 0.02, 0.048, 1.0, 0.1, 3, "f64", buf, buf, buf, buf, stream=torch.cuda.current_stream())
        for arith in (gs.GS_ARITH_IEEE, gs.GS_ARITH_DS, gs.GS_ARITH_FX, gs.GS_ARITH_FXF):
            gs.gs_set_arith(h, arith)
            for held in (gs.GS_BOUNDARY_PERIODIC, gs.GS_BOUNDARY_HELD):
                gs.gs_set_boundary(h, held)
                assert gs.gs_get_plan(h)["kernel"] == gs.GS_KERNEL_ZMARCH, (L, arith, held)
        gs.gs_destroy(h)
    torch.cuda.synchronize()
    del buf
    torch.cuda.empty_cache()


@pytest.mark.parametrize("L,held", [(834, False), (838, True), (1061, False)])
def test_rows_of_one_pair_per_tile(L, held):
    torch = need_cuda()
    out = []
    for plain in (False, True):
        sim = gs.GrayScott(L, dtype="f32", **dict(PAPER, noise=0.1, seed=2 ** 33 + 5))
        g = torch.Generator(device="cuda").manual_seed(L)
        for t, s in zip(sim.tensors(), (1.0, 0.4)):
            t.copy_(torch.rand((L, L, L), generator=g, device="cuda") * s)
        if held:
            sim.boundary = gs.GS_BOUNDARY_HELD
        if plain:
            sim.set_plan(gs.GS_KERNEL_NAIVE)
        sim.step(2)
        sim.sync()
        out.append([t.clone() for t in sim.tensors()])
        sim.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
    del out, a, b, t, sim
    torch.cuda.empty_cache()


@pytest.mark.parametrize("L,dtype,arith,held", [(72, "f64", gs.GS_ARITH_DS, False), (80, "f64", gs.GS_ARITH_FX, False),
                                                (96, "f64", gs.GS_ARITH_FXF, False), (140, "f64", gs.GS_ARITH_FXF, False),
                                                (80, "f64", gs.GS_ARITH_DS, True), (80, "f64", gs.GS_ARITH_FXF, True),
                                                (76, "f32", 0, True), (128, "f32", 0, True), (236, "f32", 0, True)])
def test_many_steps_of_shell_and_inner_rows(L, dtype, arith, held):
    need_cuda()
    sim, ref = (gs.GrayScott(L, dtype=dtype, **dict(PAPER, noise=0.1, seed=3)) for _ in range(2))
    ref.set_plan(gs.GS_KERNEL_NAIVE)
    for s in (sim, ref):
        s.arith = arith
        if held:
            s.boundary = gs.GS_BOUNDARY_HELD
        s.step(300)
    for a, b in zip(sim.read(), ref.read()):
        np.testing.assert_array_equal(a, b)
