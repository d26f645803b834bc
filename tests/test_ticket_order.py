"""The ticket by which the last warp of several finds out that it is the last orders memory for
all lanes of the warp: lane 0's fences are extended to the others by warp barriers before the
fence of the arrival and after the one that follows it.  Shuffles order no memory."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_10257_gb300", "csrc")


def test_every_lane_is_ordered_by_the_ticket():
    text = re.sub(r"//.*", "", open(os.path.join(CSRC, "lbfs_internal.cuh")).read())
    body = text[text.index("bool last_of("):]
    body = body[:body.index("\n}")]
    steps = re.findall(r"__syncwarp|__threadfence|atomicAdd|__shfl_sync", body)
    assert steps == ["__syncwarp", "__threadfence", "atomicAdd", "__threadfence", "__syncwarp", "__shfl_sync"]
