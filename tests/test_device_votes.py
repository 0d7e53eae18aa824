"""Warp votes and shuffles name their lanes by a mask that the code has voted for: the lanes that __activemask() reports need not be
together at the next instruction, so a vote on them may wait for lanes that never come."""
import glob
import os
import re

from paper_2002_04353_gb300 import build


def test_no_mask_from_the_lanes_that_happen_to_run():
    for path in sorted(glob.glob(os.path.join(build.CSRC, "*.cu*")) + glob.glob(os.path.join(build.CSRC, "*.h"))):
        code = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        assert "__activemask" not in code, os.path.basename(path)
