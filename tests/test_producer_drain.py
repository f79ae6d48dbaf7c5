"""A copy producer waits for its copies on every way out of the kernel.

Consumers that give up on a plane (their wait ran out) leave at once; if the
producer has issued its last copies by then and leaves too, the CTA ends with
copies in flight into shared memory that the next CTA owns.
"""
import os
import re

import pytest

from paper_2309_10292_gb300 import gs

CSRC = os.path.join(os.path.dirname(gs.__file__), "csrc")
DRAIN = "for (uint32_t q = (seq > (uint32_t)S ? seq - S : 0); q < seq; ++q)"


@pytest.mark.parametrize("name", ["gs_stencil.cu", "gs_variants.cu", "gs_zrow.cu"])
def test_no_way_past_the_drain(name):
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    issue, after = src.split(DRAIN)
    tail = issue[max(issue.rfind(f) for f in ("gs_tma_load_3d(", "gs_bulk_load(")):]
    assert "return" not in tail and not re.search(r"if \([^)]*\)\s*$", tail)
    assert "gs_mbar_wait(&full[q % S]" in after[:120]
