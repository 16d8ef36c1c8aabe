"""The barriers and bounded waits of the kernels, read from their sources (what
they guard against must not be provoked on a GPU)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_07298_gb300", "csrc")


def _function(file, name):
    """The text of the function `name` from its parameter list to its closing brace."""
    src = open(os.path.join(CSRC, file)).read()
    at = re.search(r"^(?:__device__|\s+fw).*\b%s\(" % name, src, flags=re.M).start()
    return src[at:src.index("\n}", at)]


# What one CTA runs several times over the same shared memory.
@pytest.mark.parametrize("file,name", [("fw_single.cu", "piece_f32"), ("fw_f64.cu", "piece64"),
                                       ("phases_f32.cuh", "minplus_half_f32")])
def test_repeated_pieces_invalidate_their_barriers(file, name):
    """mbarrier.init on a word that still holds a live barrier is undefined: each
    use ends with mbarrier.inval, after the last wait."""
    body = _function(file, name)
    assert body.index("mbar_init(") < body.rindex("mbar_wait(") < body.rindex("mbar_inval(")
