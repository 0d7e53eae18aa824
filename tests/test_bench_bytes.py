"""The bench's byte count of the step follows the launch: where one kernel takes the propagation and the moments, the moments' second
reading of the populations is not counted."""
import os
import re

import bench
from paper_2002_04353_gb300 import build, inputs as I


def test_the_rule_is_the_launchs():
    src = open(os.path.join(build.CSRC, "kernels.cuh")).read()
    assert int(re.search(r"FAST_G_NODES = (\d+)", src).group(1)) == bench.FUSED_NODES
    n = bench.FUSED_NODES
    assert bench.moments_fused(True, I.MOTION_PITCH, n) and bench.moments_fused(True, I.MOTION_BLENDED_PITCH, n)
    assert not any((bench.moments_fused(True, I.MOTION_PITCH, n - 1), bench.moments_fused(True, I.MOTION_PLUNGE, n),
                    bench.moments_fused(True, I.MOTION_NONE, n), bench.moments_fused(False, I.MOTION_PITCH, n)))


def test_fused_bytes():
    n, e, w = 600320, 298560, 60000
    plain, fused = (sum(bench.kernel_bytes(k, n, e, w, fused=f) for k in bench.STEP_KERNELS) for f in (False, True))
    assert plain - fused == 72 * n - w * (4 + 72 + 12 + 4)  # the pairs read again, but for the listed nodes'
