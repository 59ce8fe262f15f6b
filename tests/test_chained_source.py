"""Rules of the kernels that start under their predecessor which a run on a GPU must not be made to break: the order of their wait, their
TMEM allocation and the start of their successor.  Checked on the source text (no GPU)."""
import os
import re

import pytest

import paper_2603_15965_b200 as M

CSRC = os.path.join(os.path.dirname(M.__file__), "csrc")


def body(name, kernel):
    """Text of one kernel, without comments."""
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    start = re.search(r"__global__ void[^;{]*\b" + kernel + r"\(", text).end()
    return text[start:text.index("\n}\n", start)]


def test_every_kernel_that_allocates_tmem_is_looked_at():
    users = {f for f in os.listdir(CSRC) if f.endswith(".cu") and "tmem_alloc(" in open(os.path.join(CSRC, f)).read()}
    assert users == {"apply_umma.cu", "route_mlp.cu", "route_gate_umma.cu"}


@pytest.mark.parametrize("name,kernel", [("apply_umma.cu", "apply_umma_kernel"), ("route_mlp.cu", "route_mlp_umma_kernel")])
def test_tmem_is_allocated_after_the_wait_and_before_the_successor_may_start(name, kernel):
    """The allocation has no limit: a CTA that held its columns while it waited for its predecessor could keep them from a CTA of that
    predecessor on the same SM, and one that let its successor start before it had columns could find them taken by it."""
    code = body(name, kernel)
    wait, alloc = code.index("grid_dependency_wait()"), code.index("tmem_alloc(")
    barrier = code.index("__syncthreads()", alloc)
    first = min(m.start() for m in re.finditer(r"grid_dependency_(trigger|sync)\(\)", code))
    assert wait < alloc < barrier < first


def test_gate_allocates_before_its_successor_may_start():
    """It is chained to its own preparation launch only, which uses no TMEM, so it may allocate before the wait."""
    code = body("route_gate_umma.cu", "route_gate_umma_kernel")
    assert code.index("tmem_alloc(") < code.index("__syncthreads()") < code.index("grid_dependency_sync()")
    with open(os.path.join(CSRC, "route_gate_umma.cu")) as f:
        assert "image == kImageBuildAndUse) ? 2 : 1" in f.read()


def test_shrink_of_the_pair_is_an_ordinary_launch():
    """The expand loads tables, y and B before it waits for the shrink."""
    with open(os.path.join(CSRC, "apply_twophase.cu")) as f:
        text = f.read()
    assert re.search(r"launch_kernel\(shrink_kernel<R, GROUP>,[^;]*\bs, 1, false, prm, su\)", text)
    expand = body("apply_twophase.cu", "expand_kernel")
    assert expand.index("request(item)") < expand.index("grid_dependency_sync()")
