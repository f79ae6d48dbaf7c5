"""GPU test of the mma.sync weight gradient where it has few units of work: N copies
of one grid have the gradients of one, whatever planes a unit holds."""
import numpy as np
import pytest

from paper_2309_10292_gb300 import gs, inputs
from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2, 4])
def test_gradients_of_copies(N):
    # units of 1 plane (one grid), 2 and 4; the loss is a mean and N a power of
    # two, so only the order of the FP32 sums differs
    torch = need_cuda()
    g = torch.Generator(device="cuda").manual_seed(2)
    f = [torch.rand((1, 16, 16, 16), generator=g, device="cuda") * s for s in (1.0, 0.5, 1.0, 0.5)]
    got = []
    for n in (8, N):
        net = gs.Surrogate(inputs.surrogate_init_params(seed=4, last_scale=1.0))
        u, v, tu, tv = (x.repeat(n, 1, 1, 1).contiguous() for x in f)
        loss = net.grad(u, v, [0.03] * n, [0.05] * n, tu, tv)
        got.append((loss, net.grads()))
        net.close()
    (la, ga), (lb, gb) = got
    assert abs(la - lb) <= 1e-5 * la
    for (wa, ba), (wb, bb) in zip(ga, gb):
        for a, b in ((wa, wb), (ba, bb)):
            assert np.abs(a - b).max() <= 1e-4 * np.abs(a).max()
