"""The event kernels hand data from lane to lane through a warp's shared memory.  CUDA's vote functions
guarantee no memory ordering, so a vote between the writes and the reads of it has to stand beside a
__syncwarp().  A missing one shows in no result for certain, so the sources themselves are read: in the
functions that work on a warp's buffer, every vote kept in a variable (those close a phase) is
followed at once by a __syncwarp()."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2312_02756_gb300", "csrc")


def _function(src, name):
    """The bodies of the definitions of the function `name`."""
    for start in re.finditer(r"__device__ [^;{]*\b%s\(" % name, src):
        i = src.index("{", start.end())
        depth, j = 1, i + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(src[j], 0)
            j += 1
        yield src[i:j]


@pytest.mark.parametrize("file,name,phases", [("select.cu", "warp_tile", 1), ("jagged.cu", "warp_batch", 1),
                                              ("jagged_bwd.cu", "warp_batch", 2)])
def test_votes_that_close_a_phase_are_barriers(file, name, phases):
    with open(os.path.join(CSRC, file)) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    votes = [body[m.end():] for body in _function(src, name)
             for m in re.finditer(r"\w+ = __any_sync\(kAll, \w+\);", body)]
    assert len(votes) == phases
    for rest in votes:
        assert re.match(r"\s*__syncwarp\(\);", rest), rest[:80]


def test_selection_reads_its_key_before_the_next_round():
    """offer(): the keys read against the round's minimum, then a barrier, then the next round's minimum."""
    with open(os.path.join(CSRC, "select.cu")) as f:
        body = next(_function(re.sub(r"//[^\n]*", "", f.read()), "offer"))
    assert re.search(r"key == W\.key\[e\];\s*__syncwarp\(\);", body)
