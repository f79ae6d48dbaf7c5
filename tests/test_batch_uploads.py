"""The batch's device tables are copied on the batch's own stream.

A blocking cudaMemcpy from pageable memory runs on the legacy stream and may
return before its last part has landed; a launch on a non-blocking stream does
not wait for it and could read instance and row numbers that are not there yet.
"""
import os
import re

import numpy as np
import pytest

from paper_2309_10292_gb300 import gs
from tests.gpu_util import need_cuda

SRC = os.path.join(os.path.dirname(gs.__file__), "csrc", "gs_batch.cu")


def test_no_copy_on_the_legacy_stream():
    assert not re.search(r"\bcudaMemcpy\(", open(SRC).read())


@pytest.mark.gpu
@pytest.mark.parametrize("Ls", [[32, 48, 64] * 4, [4] * 300 + [128]])  # row shares, marched items
def test_first_step_on_a_non_blocking_stream(Ls):
    # tables built at creation (on the legacy stream) and by plan changes on
    # the new stream, each read by the next launch
    import torch
    need_cuda()
    F, k = np.linspace(0.02, 0.05, len(Ls)), np.linspace(0.05, 0.065, len(Ls))
    a, b = (gs.GrayScottBatch(Ls, F, k, noise=0.1, seed=9) for _ in range(2))
    st = torch.cuda.Stream()
    gs.gs_batch_set_stream(a.handle, st)
    a.step(3)
    gs.gs_batch_set_plan(a.handle, 8, 4)
    a.step(2)
    gs.gs_batch_set_plan(a.handle, 16, 8)
    a.step(2)
    b.step(7)
    for i in (0, len(Ls) // 2, len(Ls) - 1):
        for x, y in zip(a.read(i), b.read(i)):
            np.testing.assert_array_equal(x, y)
    for x in (a, b):
        x.close()
