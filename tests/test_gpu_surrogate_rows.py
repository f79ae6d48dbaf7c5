"""GPU test of the mma.sync convolutions at every row length they are tiled for.

A field of period 16 (32) has the same network output and gradients on a
larger grid that the period divides, cell by cell: the larger grid's rows are
cut into other tiles and groups (the last one ragged for 48, 80 and 96), its
planes into other runs, and the sums of a cell run in the same order.
"""
import numpy as np
import pytest

from paper_2309_10292_gb300 import gs, inputs
from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def _tiled(torch, P, L, N, seed, scale):
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.rand((N, P, P, P), generator=g, device="cuda") * scale
    return f, f.repeat(1, L // P, L // P, L // P).contiguous()


def _net(seed):
    net = gs.Surrogate(inputs.surrogate_init_params(seed=seed, last_scale=1.0))
    gs.gs_surr_set_backend(net.handle, gs.GS_SURR_MMA)
    return net


@pytest.mark.parametrize("P,L,N", [(16, 32, 3), (16, 48, 2), (16, 64, 2), (16, 80, 1), (16, 96, 1), (16, 112, 1), (16, 128, 1),
                                   (128, 256, 1)])
def test_forward_of_a_periodic_field(P, L, N):
    torch = need_cuda()
    net = _net(L)
    (u, U), (v, V) = _tiled(torch, P, L, N, 1, 1.0), _tiled(torch, P, L, N, 2, 0.5)
    F, k = [0.02 + 0.01 * n for n in range(N)], [0.05] * N
    small, large = net.forward(u, v, F, k), net.forward(U, V, F, k)
    r = L // P
    for a, b in zip(small, large):
        np.testing.assert_array_equal(a.repeat(1, r, r, r).cpu().numpy(), b.cpu().numpy())
    assert float((small[0] - u).abs().max()) > 0
    net.close()


@pytest.mark.parametrize("P,L", [(32, 64), (16, 32), (16, 48), (16, 80), (16, 96), (16, 112), (16, 128)])
def test_gradients_of_a_periodic_field(P, L):
    # the loss is a mean, so the gradients are those of one period; dL/dout is
    # scaled by (P / L)^3: exactly where that is a power of two, else its bf16
    # values (and all that follow from them) round differently, by 2^-9 of each
    # at every layer
    torch = need_cuda()
    (u, U), (v, V) = _tiled(torch, P, L, 1, 3, 1.0), _tiled(torch, P, L, 1, 4, 0.5)
    (tu, TU), (tv, TV) = _tiled(torch, P, L, 1, 5, 1.0), _tiled(torch, P, L, 1, 6, 0.5)
    nets = [_net(7) for _ in range(2)]
    ls = nets[0].grad(u, v, [0.03], [0.05], tu, tv)
    ll = nets[1].grad(U, V, [0.03], [0.05], TU, TV)
    assert abs(ls - ll) <= 1e-5 * ls
    power_of_two = (L // P) & (L // P - 1) == 0
    for (ws, bs), (wl, bl) in zip(nets[0].grads(), nets[1].grads()):
        for a, b in ((ws, wl), (bs, bl)):
            # FP32 sums of the same products in another order, or six layers' bf16 roundings
            assert np.abs(a - b).max() <= (1e-4 if power_of_two else 6 * 2.0 ** -9) * np.abs(a).max()
    for n in nets:
        n.close()
