"""GPU tests: a call of one step leaves the state it starts from as it is, in
every arithmetic and on both sides of the rules that choose its kernel, so a
captured call gives the same result at every replay."""
import numpy as np
import pytest

from paper_2309_10292_gb300 import gs
from tests.gpu_util import PAPER, need_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("arith", [gs.GS_ARITH_IEEE, gs.GS_ARITH_DS, gs.GS_ARITH_FX, gs.GS_ARITH_FXF])
@pytest.mark.parametrize("L,noise,held", [(2, 0.1, False), (16, 0.0, False), (33, 0.1, False), (48, 0.1, True), (64, 0.1, False),
                                          (80, 0.0, False), (82, 0.1, False), (101, 0.1, False), (140, 0.0, False),
                                          (160, 0.1, False)])
def test_replayed_one_step_call(L, noise, held, arith):
    torch = need_cuda()
    st = torch.cuda.Stream()
    prm = dict(PAPER, noise=noise, seed=21)
    rng = np.random.default_rng(L)
    u, v = rng.uniform(0, 1, (L, L, L)), rng.uniform(0, 0.5, (L, L, L))
    sim, ref = gs.GrayScott(L, dtype="f64", stream=st, **prm), gs.GrayScott(L, dtype="f64", **prm)
    ref.set_plan(gs.GS_KERNEL_NAIVE)
    for s in (sim, ref):
        s.arith = arith
        if held:
            s.boundary = gs.GS_BOUNDARY_HELD
        s.write(u, v)
    ref.step(1)
    want = ref.read()
    before = sim.tensors()
    st.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        sim.step(1)
    for _ in range(2):
        with torch.cuda.stream(st):
            g.replay()
        for a, b in zip(sim.read(), want):
            np.testing.assert_array_equal(a, b)
        for t, x in zip(before, (u, v)):
            np.testing.assert_array_equal(t.cpu().numpy(), x)

