"""Rules of the kernels' sources that no result can show."""

import glob
import os
import re

from paper_2607_24062_gb300 import build


def _sources():
    return {p: open(p).read() for p in sorted(glob.glob(os.path.join(build.CSRC, "*.cu*")))}


def test_aligned_cluster_barriers_follow_a_warp_sync():
    """barrier.cluster's .aligned form is undefined for a warp whose lanes come apart, and every kernel that uses it
    has blocks that one lane takes before it."""
    found = 0
    for path, text in _sources().items():
        for m in re.finditer(r"barrier\.cluster\.arrive[.a-z]*\.aligned", text):
            found += 1
            before = text[:m.start()].rstrip()
            assert re.search(r"__syncwarp\(\);\s*asm volatile\(\s*\"$", before), (path, before[-120:])
    assert found >= 1
