"""The bounded waits of the learned seed's network. A wait that runs out is reported as
what it is (not as a tile copy whose update was skipped: the update goes on from the
previous velocity), and the block waits again, with a limit, for its copy and its products
before it gives its memory back."""
import os
import re
import time

import pytest

import device_checks as D

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _src(name):
    return open(os.path.join(ROOT, "paper_1508_03452_gb300", "csrc", name)).read()


def test_a_late_seed_has_its_own_status():
    step, api = _src("step_impl.cuh"), _src("api.cu")
    late = step[step.index("if (!tc_run("):]
    assert re.search(r"atomicOr\(A\.status, (STATUS_\w+)\)", late).group(1) == "STATUS_SEED_TIMEOUT"
    bits = dict(re.findall(r"constexpr int (STATUS_\w+) = (\d+);", _src("common.cuh")))
    assert sorted(bits.values()) == ["1", "2", "4"] and bits["STATUS_SEED_TIMEOUT"] == "4"
    for name in bits:
        assert re.search(r"if \(status & lb::%s\)\s*return fail\(h, LBRMHD_ERR_TIMEOUT" % name, api), name


def test_a_late_block_waits_for_what_it_has_in_flight():
    body = _src("mlp_tc.cuh")
    body = body[body.index("bool tc_run("):]
    drain = body[body.index("if (!got)"):body.index("tc_dealloc(")]
    assert drain.count("mbar_wait_bounded(") == 2  # the weights' copy and the products


@pytest.mark.gpu
def test_the_waits_give_up():
    """Weights that never arrive (nothing is in flight): every thread of the block is told
    within the two wait limits of 0.5 s, and tensor memory and the context stay usable."""
    lib = D.load()
    for _ in range(5):  # (five blocks' columns: one more than an SM has, were they kept)
        t0 = time.perf_counter()
        assert lib.check_late_seed() == 128
        assert time.perf_counter() - t0 < 4.0
