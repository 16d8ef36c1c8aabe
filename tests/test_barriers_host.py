"""The barriers and bounded waits of the kernels, read from their sources (what
they guard against must not be provoked on a GPU)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_07298_gb300", "csrc")


def _function(file, name):
    """The text of the function `name` from its parameter list to its closing brace."""
    src = open(os.path.join(CSRC, file)).read()
    at = re.search(r"^(?:__device__.*\b|\s+)%s\(" % name, src, flags=re.M).start()
    return src[at:src.index("\n}", at)]


# What one CTA runs several times over the same shared memory.
@pytest.mark.parametrize("file,name", [("fw_single.cu", "piece_f32"), ("fw_f64.cu", "piece64"),
                                       ("phases_f32.cuh", "minplus_half_f32")])
def test_repeated_pieces_invalidate_their_barriers(file, name):
    """mbarrier.init on a word that still holds a live barrier is undefined: each
    use ends with mbarrier.inval, after the last wait."""
    body = _function(file, name)
    assert body.index("mbar_init(") < body.rindex("mbar_wait(") < body.rindex("mbar_inval(")


@pytest.mark.parametrize("file,kernel,piece", [("fw_single.cu", "fw_phase3_listed_f32", "piece_f32"),
                                               ("fw_f64.cu", "fw64_listed", "piece64")])
def test_listed_kernels_stop_where_a_wait_ran_out(file, kernel, piece):
    """A copy that arrived late would complete the next piece's phase with the wrong operands."""
    assert re.search(r"if \(!%s\b[^;]*\) return;" % piece, _function(file, kernel))
    assert re.search(r"give_up\([^;]*;\s*return false;", _function(file, piece))


def test_ctas_whose_wait_ran_out_wait_for_their_copies():
    """Nothing of a CTA may still land in its shared memory after it has left."""
    for file in ("fw_single.cu", "fw_f64.cu", "screen.cuh", "phases_f32.cuh"):
        src = open(os.path.join(CSRC, file)).read()
        for m in re.finditer(r"report_wait_timeout\(\);", src):  # phase 1, a cluster: at its end
            end = src[m.end():src.index("\n}", m.end())]
            assert "drain_ring(sm.bar, nquad, WARPS, cta)" in end, file
        assert "give_up(&sm.bar" in src, file


def test_default_wait_is_the_short_one():
    """A poll that suspends the thread takes about 3 us: 2^18 of them, not 2^22 (13 s)."""
    src = open(os.path.join(CSRC, "bulk.cuh")).read()
    assert re.search(r"kPollLimit = 1u << 18;", src)
    assert re.search(r"bool mbar_wait\(uint64_t \*bar, uint32_t parity, uint32_t limit = kPollLimit\)", src)
