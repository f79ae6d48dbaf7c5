"""GPU test of the default plan's z-march tile: every edge that the rule covers
gets a tile that launches (in every FP64 arithmetic) and gives the plain
kernel's fields bit for bit, whichever order arithmetic and boundary are set in.
"""
import numpy as np
import pytest

from paper_2309_10292_gb300 import gs
from tests.gpu_util import PAPER, need_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,dtype,arith,noise", [(260, "f32", 0, 0.1), (300, "f32", 0, 0.0), (512 + 4, "f32", 0, 0.1),
                                                 (162, "f64", 1, 0.1), (190, "f64", 1, 0.0), (194, "f64", 2, 0.1),
                                                 (222, "f64", 2, 0.0), (162, "f64", 3, 0.1), (254, "f64", 3, 0.0),
                                                 (258, "f64", 3, 0.1), (302, "f64", 1, 0.1)])
def test_default_tile_equals_the_plain_kernel(L, dtype, arith, noise):
    need_cuda()
    out = []
    for plain in (False, True):
        sim = gs.GrayScott(L, dtype=dtype, **dict(PAPER, noise=noise, seed=3))
        if arith:
            sim.arith = arith
        sim.boundary = gs.GS_BOUNDARY_HELD  # the default plan follows the boundary there and back
        sim.boundary = gs.GS_BOUNDARY_PERIODIC
        assert sim.plan["kernel"] == gs.GS_KERNEL_ZMARCH
        if plain:
            sim.set_plan(gs.GS_KERNEL_NAIVE)
        sim.step(3)
        sim.step(1)
        out.append(sim.read())
        sim.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("L,arith", [(82, 1), (128, 2), (140, 3), (142, 3), (190, 1), (258, 2)])
def test_default_tile_with_the_outer_layer_held(L, arith):
    need_cuda()
    out = []
    for plain in (False, True):
        sim = gs.GrayScott(L, dtype="f64", **dict(PAPER, noise=0.1, seed=3))
        sim.boundary = gs.GS_BOUNDARY_HELD
        sim.arith = arith
        if plain:
            sim.set_plan(gs.GS_KERNEL_NAIVE)
        sim.step(3)
        out.append(sim.read())
        sim.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


def test_every_default_tile_launches():
    need_cuda()
    for L in list(range(82, 262, 2)) + list(range(264, 520, 16)):
        for arith in (1, 2, 3):
            held = gs.GrayScott(L, dtype="f64", **dict(PAPER, noise=0.1 if L % 4 else 0.0, seed=3))
            held.boundary = gs.GS_BOUNDARY_HELD
            held.arith = arith
            held.step(1)
            held.sync()
            held.close()
            sim = gs.GrayScott(L, dtype="f64", **dict(PAPER, noise=0.1 if L % 4 else 0.0, seed=3))
            sim.arith = arith
            sim.step(1)
            sim.step(3)  # converting, packing, packed and unpacking kernels
            sim.sync()
            sim.close()
