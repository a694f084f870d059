"""Counters of finished blocks that outlive a launch return to zero with the launch's last increment.

sum_mode0_kernel and finish_max keep such a counter in the mesh.  With atomicAdd and a reset by the last
block, two calls that overlap on one mesh could leave a remainder behind, and no later call would find its
last block; atomicInc wraps after the launch's own number of increments, whatever the order."""
import glob
import os
import re

from paper_2601_16911_gb300 import build as B
from tests.test_dependent_launch_sources import strip_comments


def test_block_counters_wrap_by_themselves():
    found = 0
    for f in sorted(glob.glob(os.path.join(B.CSRC, "*.cu*"))):
        with open(f) as h:
            text = strip_comments(h.read())
        found += len(re.findall(r"atomicInc\s*\(", text))
        # an increment compared with a block count is the last block's test
        assert not re.search(r"atomicAdd\s*\([^;{}]*\bdone\b[^;{}]*\)\s*==", text), os.path.basename(f)
        assert not re.search(r"\*\s*(\w+\.)?done\s*=\s*0", text), os.path.basename(f)
    assert found == 2
