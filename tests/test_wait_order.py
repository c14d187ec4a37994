"""Waits that a warp shares, read from the kernels' source (CPU only)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_25332_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


@pytest.mark.parametrize("path", SOURCES, ids=[os.path.basename(p) for p in SOURCES])
def test_a_lanes_wait_is_shared_behind_a_warp_barrier(path):
    """Lane 0 waits on an mbarrier and the other lanes take the result by shuffle: what they
    do next (a load into the stage that was waited for) is ordered after the wait by
    __syncwarp(), which the shuffle is not stated to do."""
    code = _code(path)
    for m in re.finditer(r"if \((?:lane|\(threadIdx\.x & 31\)) == 0\) (\w+) = [^;]*\bmbar_wait\w*\([^;]*;", code):
        after = code[m.end():]
        share = re.search(r"__shfl_sync\([^;]*\b" + m.group(1) + r"\b", after)
        assert share, m.group(0)
        assert "__syncwarp();" in after[:share.start()], f"{os.path.basename(path)}: {m.group(0)}"


def test_a_wait_of_every_lane_is_voted_on():
    """The streaming head scores' workers poll with every lane and treat the outcome as the
    warp's: where one lane gives up, no lane may go on waiting at the next chunk."""
    code = _code(os.path.join(CSRC, "head_scores_stream.cu"))
    waits = list(re.finditer(r"if \(!failed\) failed = !mbar_wait\([^;]*;", code))
    assert len(waits) == 1
    rest = code[waits[0].end():].lstrip()
    assert rest.startswith("failed = __any_sync(0xffffffffu, failed);")
