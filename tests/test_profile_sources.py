"""Every summary of a step kernel's capture names the sources it was taken on, and these are
the committed ones: a summary of an earlier kernel is no evidence for this one."""
import glob
import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_step_summaries_are_of_the_committed_sources():
    files = sorted(glob.glob(os.path.join(ROOT, "profiles", "step_*.md")))
    assert len(files) >= 5
    for path in files:
        sha = re.findall(r"kernel_sources_sha: ([0-9a-f]+)", open(path).read())
        assert sha and set(sha) == {bench.kernel_sha()}, os.path.basename(path)
