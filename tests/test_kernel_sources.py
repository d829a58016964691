"""The hash that ties the committed profile to the step kernel covers every file that the
kernel is compiled from: what step_impl.cuh includes, and what that includes."""
import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

CSRC = os.path.join(ROOT, "paper_1508_03452_gb300", "csrc")


def test_kernel_hash_covers_every_included_header():
    seen, todo = set(), ["step_impl.cuh"]
    while todo:
        name = todo.pop()
        if name not in seen:
            seen.add(name)
            todo += re.findall(r'^\s*#\s*include\s+"([^"]+)"', open(os.path.join(CSRC, name)).read(), re.M)
    assert seen == set(bench.KERNEL_SOURCES)
