"""GPU test: in a context that may use part of the SMs a batch's launches are
sized by that part, and the many-steps launch of a single grid falls back.

The batch is not stepped there: a cooperative launch from a graph that does not
fit is not refused, it never ends.
"""
import subprocess
import sys

import pytest

from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes as C, sys
import numpy as np, torch
torch.zeros(1, device="cuda")
cu = C.CDLL("libcuda.so.1")
whole, part, rest, n = (C.c_ubyte * 1024)(), (C.c_ubyte * 1024)(), (C.c_ubyte * 1024)(), C.c_uint(1)
desc, green, ctx, st = C.c_void_p(), C.c_void_p(), C.c_void_p(), C.c_void_p()
if not hasattr(cu, "cuGreenCtxCreate"):
    sys.exit(77)
for rc in (cu.cuDeviceGetDevResource(0, whole, 1), cu.cuDevSmResourceSplitByCount(part, C.byref(n), whole, rest, 0, 64),
           cu.cuDevResourceGenerateDesc(C.byref(desc), part, 1), cu.cuGreenCtxCreate(C.byref(green), desc, 0, 1),
           cu.cuCtxFromGreenCtx(C.byref(ctx), green), cu.cuGreenCtxStreamCreate(C.byref(st), green, 1, 0)):
    if rc:
        sys.exit(77)
sms = int(np.frombuffer(bytes(part), dtype=np.uint32)[24])
from paper_2309_10292_gb300 import gs
def batch():
    b = gs.GrayScottBatch([64] * 3, [0.02] * 3, [0.05] * 3, noise=0.1, seed=3)
    grid = b.info["grid"]
    b.close()
    return grid
before = batch()
assert cu.cuCtxSetCurrent(ctx) == 0
assert batch() <= sms < before, (batch(), sms, before)
bufs = [torch.empty((128,) * 3, device="cuda") for _ in range(4)]
h = gs.gs_create_on(128, 0.2, 0.1, 0.02, 0.048, 1.0, 0.1, 3, "f32", *bufs, stream=type("S", (), {"cuda_stream": st.value}))
launches = gs.gs_launch_count(h)
gs.gs_step(h, 10)
gs.gs_sync(h)
assert gs.gs_launch_count(h) - launches == 10  # one per step: the many-steps launch does not fit
got = gs.gs_read(h, gs.GS_U, np.empty((128,) * 3, dtype=np.float32))
gs.gs_destroy(h)
ref = gs.GrayScott(128, Du=0.2, Dv=0.1, F=0.02, k=0.048, dt=1.0, noise=0.1, seed=3)
ref.set_plan(gs.GS_KERNEL_NAIVE)
ref.step(10)
assert np.array_equal(got, ref.read()[0])
"""


def test_part_of_the_sms():
    need_cuda()
    out = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, timeout=120)
    if out.returncode == 77:
        pytest.skip("no green contexts here")
    assert out.returncode == 0, out.stderr
