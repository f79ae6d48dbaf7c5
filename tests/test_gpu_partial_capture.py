"""GPU test: a call captured on a stream that may use part of the SMs records
one launch per step.

The many-steps launch does not fit there, which a capture does not report, and
a replay of it would never end; so the launches are counted before the replay.
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
if sys.argv[1] == "current":
    assert cu.cuCtxSetCurrent(ctx) == 0
from paper_2309_10292_gb300 import gs
L = 128
bufs = [torch.empty((L,) * 3, device="cuda") for _ in range(4)]
h = gs.gs_create_on(L, 0.2, 0.1, 0.02, 0.048, 1.0, 0.1, 3, "f32", *bufs, stream=type("S", (), {"cuda_stream": st.value}))
gs.gs_sync(h)
launches = gs.gs_launch_count(h)
graph, run = C.c_void_p(), C.c_void_p()
assert cu.cuStreamBeginCapture_v2(st, 1) == 0
gs.gs_step(h, 10)
assert cu.cuStreamEndCapture(st, C.byref(graph)) == 0
assert gs.gs_launch_count(h) - launches == 10, gs.gs_launch_count(h) - launches
assert cu.cuGraphInstantiateWithFlags(C.byref(run), graph, C.c_ulonglong(0)) == 0
assert cu.cuGraphLaunch(run, st) == 0
gs.gs_sync(h)
got = gs.gs_read(h, gs.GS_U, np.empty((L,) * 3, dtype=np.float32))
gs.gs_destroy(h)
ref = gs.GrayScott(L, Du=0.2, Dv=0.1, F=0.02, k=0.048, dt=1.0, noise=0.1, seed=3)
ref.set_plan(gs.GS_KERNEL_NAIVE)
ref.step(10)
assert np.array_equal(got, ref.read()[0])
"""


@pytest.mark.parametrize("context", ["current", "of_the_stream"])
def test_captured_on_part_of_the_sms(context):
    need_cuda()
    out = subprocess.run([sys.executable, "-c", CHILD, context], capture_output=True, text=True, timeout=120)
    if out.returncode == 77:
        pytest.skip("no green contexts here")
    assert out.returncode == 0, out.stderr
