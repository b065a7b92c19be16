"""What the kernels that begin before the launch ahead of them has ended must keep to, checked in their source on the CPU."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2307_14995_b200", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"/\*.*?\*/|//[^\n]*", "", text, flags=re.S)


@pytest.mark.parametrize("name,unless_known", [
    ("la_tc_state.cuh", ""),                                                   # may be the first launch of a call
    ("la_tc_walk.cuh", "if (EARLY && args.follows == FOLLOWS_ANY) "),           # the others follow this library's kernels
    ("la_tc_walk64.cuh", "if (args.follows == FOLLOWS_ANY) ")])
def test_tensor_memory_is_taken_behind_the_wait(name, unless_known):
    """The kernel ahead may belong to another library and let this one begin before it has all its tensor memory.  Columns taken
    before it is complete are given back only after it: neither would go on."""
    text = source(name)
    allocs = [m.start() for m in re.finditer(r"\btmem_alloc\(", text)]
    assert len(allocs) == 1
    before = " ".join(text[:allocs[0]].split())
    assert before.endswith("if (warp == 1) { " + unless_known + "grid_dep_wait();")


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_loads_take_no_path_for_memory_that_nobody_writes(name):
    """A kernel that begins early runs while the launch ahead still writes what it will read: ld.global.nc (__ldg, or the compiler's
    choice for const __restrict__ parameters) is for memory that is read-only from the kernel's beginning on, and the other load
    intrinsics may be moved ahead of the wait."""
    assert re.findall(r"__ldg|__ldc[gsav]|__ldlu|ld\.global\.nc|__restrict__", source(name)) == []
