"""A wait that gives up ends its kernel: no barrier without a limit stands where a warp whose wait gave up does not come.

mbarrier waits have a limit (csrc/tc_common.cuh); named barriers have none, so that one warp that left keeps the others for good.
The kernels that use one bring every warp to it whatever its waits returned; this list is the places that were looked at."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_06419_b200", "csrc")
NAMED = {"fused_rgran.cu": 1,      # quarter_sync: no warp leaves before the end, a failure only skips the work
         "fused_tc2.cu": 1,        # merge of the two warpgroups: reached with `ok` false too, whose sum is then NaN
         "fused_tc3.cu": 2,        # two warps of a row: they vote on the failure at the barrier and leave together
         "fused_tf32.cu": 2}       # merge of the two streams: as in fused_tc2.cu


def code(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", f.read(), flags=re.S))


@pytest.mark.parametrize("name", sorted(os.path.basename(p) for p in glob.glob(os.path.join(CSRC, "*.cu*"))))
def test_named_barriers(name):
    text = code(os.path.join(CSRC, name))
    assert len(re.findall(r"\b(?:bar|barrier)\.(?:cta\.)?(?:sync|red)|__barrier_sync|named_barrier", text)) == NAMED.get(name, 0)
