"""Launch rules take the number of multiprocessors from the device: a grid of "one wave" or a
rule on idle SMs written for one chip is wrong on a smaller part or a slice of it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1508_03452_gb300", "csrc")


def test_no_sm_count_in_the_code():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
        code = re.sub(r"//.*", "", src)
        assert not re.search(r"\b(148|152|160)\b", code), os.path.basename(path)
