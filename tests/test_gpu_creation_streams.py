"""GPU tests: what creation fills is filled before creation returns, so an object
that is then given a non-blocking stream does not find it filled later."""
import numpy as np
import pytest

from paper_2309_10292_gb300 import gs, inputs
from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def busy_legacy_stream(torch):
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.default_stream()):
        torch.cuda._sleep(100_000_000)  # about 50 ms of work in front of what creation queues there


def test_surrogate_parameters_survive_creation():
    torch = need_cuda()
    params = inputs.surrogate_init_params(seed=3, last_scale=0.1)
    st = torch.cuda.Stream()
    busy_legacy_stream(torch)
    net = gs.Surrogate(params, stream=st)
    torch.cuda.synchronize()
    for (w, b), (w2, b2) in zip(params, net.params()):
        np.testing.assert_array_equal(np.asarray(w, dtype=np.float32).reshape(-1), w2.reshape(-1))
        np.testing.assert_array_equal(np.asarray(b, dtype=np.float32).reshape(-1), b2.reshape(-1))
    net.close()


def test_single_field_survives_creation():
    torch = need_cuda()
    f = np.random.default_rng(1).uniform(0, 1, (16, 16, 16)).astype(np.float32)
    with torch.cuda.stream(torch.cuda.Stream()):
        busy_legacy_stream(torch)
        one = gs.SingleField(16)
        one.write(f)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(one.read(), f)
        one.close()
