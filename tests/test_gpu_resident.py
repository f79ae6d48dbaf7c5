"""GPU tests of the many-steps launch that the default plan of a small grid takes.

It must equal the one-thread-per-cell kernel bit for bit in every arithmetic, whatever the edge
(vector and scalar loads, one CTA to one per SM, runs of rows and bricks that
do not divide the grid), the boundary and the grouping of steps into calls.
"""
import numpy as np
import pytest

import oracle
from paper_2309_10292_gb300 import gs
from tests.gpu_util import PAPER, maxabs, need_cuda

pytestmark = pytest.mark.gpu


def make(L, dtype, held=False, **kw):
    need_cuda()
    sim = gs.GrayScott(L, dtype=dtype, **dict(PAPER, **kw))
    if held:
        sim.boundary = gs.GS_BOUNDARY_HELD
    return sim


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("noise,held", [(0.1, False), (0.0, False), (0.1, True), (0.0, True)])
@pytest.mark.parametrize("L", [1, 2, 3, 4, 5, 12, 17, 32, 50, 63, 72, 88, 100])
def test_small_grids_equal_the_plain_kernel(L, noise, held, dtype):
    rng = np.random.default_rng(L)
    u, v = rng.uniform(0, 1, (L, L, L)), rng.uniform(0, 0.5, (L, L, L))
    sim, ref = (make(L, dtype, held, noise=noise, seed=2 ** 35 + 7) for _ in range(2))
    ref.set_plan(gs.GS_KERNEL_NAIVE)
    for s in (sim, ref):
        s.write(u, v)
        s.t = 5
    for n in (1, 7, 0, 2):  # an odd and an even number of buffer swaps per call, one step without the barrier
        sim.step(n)
    ref.step(10)
    assert sim.t == 15
    for a, b in zip(sim.read(), ref.read()):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("L", [72, 76, 80, 92, 104, 128, 144, 224])
def test_inner_rows_under_the_barrier(L):
    # bricks whose shell is announced before their inner rows are stepped: many
    # steps in one call, where a CTA that runs ahead would read or overwrite
    # what another one still needs
    sim, ref = (make(L, "f32", noise=0.1, seed=3) for _ in range(2))
    ref.set_plan(gs.GS_KERNEL_NAIVE)
    sim.step(300)
    ref.step(300)
    for a, b in zip(sim.read(), ref.read()):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("L,dtype", [(180, "f32"), (184, "f32"), (256, "f32"), (255, "f32"), (256, "f64"), (145, "f64")])
def test_largest_grids_equal_the_plain_kernel(L, dtype):
    # both sides of the L2 footprint rule and the largest edge
    sim, ref = (make(L, dtype, noise=0.1, seed=3) for _ in range(2))
    ref.set_plan(gs.GS_KERNEL_NAIVE)
    sim.step(5)
    ref.step(5)
    for a, b in zip(sim.read(), ref.read()):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("arith", [gs.GS_ARITH_DS, gs.GS_ARITH_FX, gs.GS_ARITH_FXF])
@pytest.mark.parametrize("L,noise,dt", [(1, 0.1, 1.0), (2, 0.1, 1.0), (5, 0.1, 0.5), (12, 0.0, 1.0), (33, 0.1, 1.0),
                                        (64, 0.1, 0.5), (101, 0.1, 1.0), (160, 0.1, 1.0)])
def test_fp64_arithmetics_equal_the_plain_kernel(L, noise, dt, arith):
    # packed between the steps of a call, FP64 at its ends, like the plain kernel
    _fp64_against_plain(L, noise, dt, arith, False)


@pytest.mark.parametrize("arith", [gs.GS_ARITH_DS, gs.GS_ARITH_FX, gs.GS_ARITH_FXF])
@pytest.mark.parametrize("L,noise,dt", [(1, 0.1, 1.0), (3, 0.1, 1.0), (12, 0.0, 0.5), (33, 0.1, 1.0), (80, 0.1, 1.0),
                                        (119, 0.0, 1.0)])
def test_fp64_arithmetics_with_the_outer_layer_held(L, noise, dt, arith):
    # FP64 between the steps: the outer layer keeps its values to the bit
    _fp64_against_plain(L, noise, dt, arith, True)


def _fp64_against_plain(L, noise, dt, arith, held):
    rng = np.random.default_rng(L)
    u, v = rng.uniform(0, 1, (L, L, L)), rng.uniform(0, 0.5, (L, L, L))
    sim, ref = (make(L, "f64", held, noise=noise, dt=dt, seed=11) for _ in range(2))
    ref.set_plan(gs.GS_KERNEL_NAIVE)
    for s in (sim, ref):
        s.arith = arith
        s.write(u, v)
        for n in (1, 6, 2, 0):
            s.step(n)
    assert gs.gs_launch_count(ref.handle) - gs.gs_launch_count(sim.handle) == (18 if held else 9) - 3
    for a, b in zip(sim.read(), ref.read()):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("held", [False, True])
@pytest.mark.parametrize("arith,bad", [(gs.GS_ARITH_FX, 1500.0), (gs.GS_ARITH_FXF, 5.0)])
def test_fp64_range_is_reported(arith, bad, held):
    L = 16
    u, v = np.ones((L, L, L)), np.zeros((L, L, L))
    u[3, 4, 5] = bad
    sim = make(L, "f64", held, noise=0.0)
    sim.arith = arith
    sim.write(u, v)
    sim.step(2)
    with pytest.raises(gs.GsError) as e:
        sim.sync()
    assert e.value.status == gs.GS_EINVAL
    sim.init()
    sim.step(2)
    sim.sync()


def test_fp64_call_of_several_launches_stays_packed():
    L, n = 6, 4096 + 5
    sim, ref = (make(L, "f64", noise=0.1, seed=3) for _ in range(2))
    ref.set_plan(gs.GS_KERNEL_NAIVE)
    for s in (sim, ref):
        s.arith = gs.GS_ARITH_FXF
        s.step(n)
    for a, b in zip(sim.read(), ref.read()):
        np.testing.assert_array_equal(a, b)


def test_more_steps_than_one_launch_holds():
    L, n = 8, 4096 + 3
    sim, ref = (make(L, "f32", noise=0.1, seed=3) for _ in range(2))
    ref.set_plan(gs.GS_KERNEL_NAIVE)
    before = gs.gs_launch_count(sim.handle)
    sim.step(n)
    assert gs.gs_launch_count(sim.handle) == before + 2
    ref.step(n)
    for a, b in zip(sim.read(), ref.read()):
        np.testing.assert_array_equal(a, b)


def test_captured_call_replays():
    # a captured call advances from the state it was captured at, every time
    import torch
    L, n = 24, 6
    st = torch.cuda.Stream()
    sim = make(L, "f32", noise=0.1, seed=4, stream=st)
    sim.step(2)
    start = [t.clone() for t in sim.tensors()]
    src = sim.tensors()
    st.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        sim.step(n)
    got = []
    for _ in range(2):
        with torch.cuda.stream(st):
            for a, b in zip(src, start):
                a.copy_(b)
            g.replay()
        got.append(sim.read())
    u0, v0 = oracle.init(L)
    uo, vo = oracle.step(u0, v0, 2 + n, **dict(PAPER, noise=0.1, seed=4))
    for (u, v) in got:
        assert maxabs(u, uo) <= 1e-4 and maxabs(v, vo) <= 1e-4
        np.testing.assert_array_equal(u, got[0][0])
        np.testing.assert_array_equal(v, got[0][1])


def test_grids_on_two_streams():
    import torch
    sims = [make(48, "f32", noise=0.1, seed=5 + i, stream=torch.cuda.Stream()) for i in range(2)]
    for _ in range(20):
        for s in sims:
            s.step(9)
    for i, s in enumerate(sims):
        ref = make(48, "f32", noise=0.1, seed=5 + i)
        ref.set_plan(gs.GS_KERNEL_NAIVE)
        ref.step(180)
        for a, b in zip(s.read(), ref.read()):
            np.testing.assert_array_equal(a, b)


def test_tuner_keeps_it_and_the_cache_remembers(tmp_path):
    path = str(tmp_path / "plans.txt")
    a = make(64, "f32", noise=0.1, seed=1)
    best, hit = a.autotune_cached(path, steps_per_trial=48)
    assert not hit and best["kernel"] == gs.GS_KERNEL_AUTO and a.plan == best
    b = make(64, "f32", noise=0.1, seed=1)
    best2, hit2 = b.autotune_cached(path, steps_per_trial=48)
    assert hit2 and best2 == best and b.plan == best
    before = gs.gs_launch_count(b.handle)
    b.step(30)
    assert gs.gs_launch_count(b.handle) == before + 1
    b.set_plan(gs.GS_KERNEL_ZMARCH)
    b.step(3)
    assert gs.gs_launch_count(b.handle) == before + 4


# ---------------------------------------------------------------------------
# Small batches (equal shares of all instances' rows per CTA)
# ---------------------------------------------------------------------------
def batch_pair(Ls, dtype, noise):
    need_cuda()
    F, k = np.linspace(0.02, 0.05, len(Ls)), np.linspace(0.05, 0.065, len(Ls))
    return [gs.GrayScottBatch(Ls, F, k, noise=noise, seed=2 ** 33 + 1, dtype=dtype) for _ in range(2)]


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("Ls,noise", [([4], 0.1), ([4, 8, 12, 100], 0.1), ([64, 20, 36] * 5, 0.0), ([32] * 40, 0.1),
                                      ([160, 4, 4], 0.1)])
def test_small_batches_equal_marched_items(Ls, noise, dtype):
    a, b = batch_pair(Ls, dtype, noise)
    gs.gs_batch_set_plan(b.handle, 8, 4)
    for n in (1, 6, 1, 3):
        a.step(n)
    assert a.info["grid"] <= 152 and a.t == 11
    b.step(11)
    for i in range(len(Ls)):
        for x, y in zip(a.read(i), b.read(i)):
            np.testing.assert_array_equal(x, y)
    # per-instance launches and a new step index continue from its state
    for x in (a, b):
        x.step_sequential(2)
        x.t = 40
        x.step(5)
    for x, y in zip(a.read(0), b.read(0)):
        np.testing.assert_array_equal(x, y)


def test_batch_of_many_tiny_grids_keeps_marched_items():
    # more segments than a CTA of the row-sharing kernel holds
    a, b = batch_pair([4] * 300 + [128], "f32", 0.1)
    gs.gs_batch_set_plan(b.handle, 32, 8)
    for x in (a, b):
        x.step(4)
    assert a.info["grid"] == b.info["grid"] > 152  # two CTAs per SM, as many items as there are
    for i in (0, 150, 299, 300):
        for x, y in zip(a.read(i), b.read(i)):
            np.testing.assert_array_equal(x, y)


def test_batch_tuner_keeps_row_shares():
    a, b = batch_pair([32, 48, 64] * 4, "f32", 0.0)
    plan = a.autotune(steps_per_trial=48)
    assert (plan["tile_z"], plan["stages"], plan["depth"]) == (32, 8, 1)
    assert a.info["grid"] == 152 and a.t == 0
    a.step(9)
    gs.gs_batch_set_plan(b.handle, 32, 8)
    b.step(9)
    for i in (0, 5, 11):
        for x, y in zip(a.read(i), b.read(i)):
            np.testing.assert_array_equal(x, y)
