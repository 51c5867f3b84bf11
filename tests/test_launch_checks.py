"""CPU check of the sources: every kernel launch is followed by its
BGL_LAUNCH_CHECK, which reports a launch that failed where it happened and
counts it (bgl_launch_count), before the next launch; the two sides of a
choice share one."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_03504_gb300", "csrc")


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))), ids=os.path.basename)
def test_every_launch_is_checked(path):
    src = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
    open_launch = None
    for m in re.finditer(r"<<<|cudaLaunchKernelEx\b|BGL_LAUNCH_CHECK\(\)|\belse\b|if \(!launched\)", src):
        if m.group() in ("<<<", "cudaLaunchKernelEx"):
            assert open_launch is None, src[open_launch - 60:open_launch + 20]
            open_launch = m.start()
        else:
            open_launch = None
    assert open_launch is None
