"""The stencil timing command line on the default plan."""
import json

import pytest

from tests.gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def test_timing_cli_default_plan(capsys):
    need_cuda()
    from paper_2309_10292_gb300 import gs, timing
    timing.main(["--L", "32", "--steps", "3", "--plan", "auto"])
    out = json.loads(capsys.readouterr().out.strip().splitlines()[-1])
    sim = gs.GrayScott(32)
    assert out["plan"] == sim.plan and out["gcups"] > 0
    sim.close()
