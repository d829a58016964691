"""The kernels that may be launched while their predecessor drains (they call
grid_wait) live while other kernels write the state that they read, so nothing on
their way may take the read-only load path, whose terms are that nobody writes the
data while the kernel lives. Checked on the sources: a wrong load there is a race
that no run has to show."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1508_03452_gb300", "csrc")
READ_ONLY = re.compile(r"__ldg\s*\(|__restrict__|\.nc\b|mlp_ld<true>")


def _code(name):
    src = re.sub(r"/\*.*?\*/", "", open(os.path.join(CSRC, name)).read(), flags=re.S)
    return re.sub(r"//.*", "", src)


def _body(src, name):
    """The function `name` (its first definition), from its name to the closing brace."""
    i = src.index("{", re.search(r"\b%s\s*\(" % name, src).start())
    depth, j = 1, i + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        j += 1
    return src[src.rindex(name, 0, i):j]


def test_state_loads_are_ordinary():
    assert not READ_ONLY.findall(_code("common.cuh"))
    step = _code("step_impl.cuh")
    # the argument records and tile lists of the batched and persistent launches are
    # constant while those kernels live
    for kernel in ("step_batch_kernel", "step_persistent_kernel"):
        step = step.replace(_body(step, kernel), "").replace("__restrict__ args", "args").replace("__restrict__ tiles", "tiles")
    assert "step_kernel" in step and "step_cell" in step
    assert not READ_ONLY.findall(step)
    assert "grid_wait();" in _body(_code("aux.cu"), "bfix_kernel")
    assert not READ_ONLY.findall(_body(_code("aux.cu"), "bfix_kernel"))
    assert not READ_ONLY.findall(_body(_code("aux.cu"), "load_prim"))


def test_training_kernels_read_what_the_chain_writes_through_l2():
    """The samples are constant over a call; parameters, moments and partial sums are
    written by the launch before: no read-only promise on them."""
    src = _code("mlp.cu")
    for kernel, constant in (("mlp_grad_kernel", {"data"}), ("mlp_reduce_kernel", set())):
        params = re.search(r"\b%s\s*\(([^)]*)\)" % kernel, src).group(1)
        assert set(re.findall(r"__restrict__\s+(\w+)", params)) <= constant, kernel
        assert "grid_wait();" in _body(src, kernel)
