"""bench.py on grids whose tuned plan is the default one (reported as GS_KERNEL_AUTO)."""
import json
import os
import subprocess
import sys

import pytest

from paper_2309_10292_gb300 import gs
from tests.gpu_util import need_cuda

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("plan,L,steps,launches,name,per,nbytes", [
    (dict(kernel=gs.GS_KERNEL_AUTO, depth=1), 64, 5000, 5, "resident", 1000, 16 * 64 ** 3 * 1000),
    (dict(kernel=gs.GS_KERNEL_AUTO, depth=1), 250, 5000, 5000, "zrow", 1, 16 * 250 ** 3),
    (dict(kernel=gs.GS_KERNEL_ZMARCH, depth=1), 512, 5000, 5000, "zmarch", 1, 16 * 512 ** 3),
    (dict(kernel=gs.GS_KERNEL_TBLOCK, depth=3), 512, 999, 333, "tblock", 3, 16 * 512 ** 3),
    (dict(kernel=gs.GS_KERNEL_NAIVE, depth=1), 16, 10, 10, "naive", 1, 16 * 16 ** 3)])
def test_launch_summary(plan, L, steps, launches, name, per, nbytes):
    sys.path.insert(0, ROOT)
    import bench
    kernel, got, bound, b = bench.launch_summary(plan, L, steps, launches)
    assert name in kernel and got == per and b == nbytes and bound


@pytest.mark.gpu
@pytest.mark.parametrize("L", [64, 250])
def test_bench_runs_on_a_small_grid(L):
    need_cuda()
    off = [f"--no-{x}" for x in ("cpu", "fp64", "batch", "large", "surrogate", "snapshot", "variants")]
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--L", str(L), "--time-steps", "50", "--steps", "2",
                          "--warmup", "3", *off], capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert out.returncode == 0, out.stderr
    line = json.loads(out.stdout.strip().splitlines()[-1])
    r = line["roofline"]
    assert line["value"] > 0 and line["config"]["plan"]["kernel"] == gs.GS_KERNEL_AUTO
    assert r["steps_per_launch"] == (50 if L == 64 else 1) and r["algorithmic_bytes_per_launch"] == 16 * L ** 3 * r["steps_per_launch"]
