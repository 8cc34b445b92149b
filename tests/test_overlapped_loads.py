"""Loads behind griddepcontrol.wait, read from the kernels' source (no GPU).

A kernel launched with programmatic stream serialization starts while the kernel in front
of it still writes.  What that kernel writes is not read-only for the whole life of the
one that waits, so its loads may take neither the non-coherent path (__ldg, or a pointer
that is both const and __restrict__) nor move in front of the wait: they go through a
volatile load with a memory clobber.  Whether the compiler does move one cannot be tested
by running, so the rule is held where it is written."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2104_06311_gb300", "csrc")


def _kernel(path, name):
    """Parameters and body of a kernel, comments removed."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, path)).read())
    m = re.search(r"__global__[^{;]*\b" + name + r"\s*\(([^{;]*)\)\s*\{", text)
    assert m, name
    depth, end = 1, m.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        end += 1
    return m.group(1), text[m.end():end]


# kernel, what it reads that the kernel in front of it writes: pointer, and how it is loaded
CASES = [("kk.cu", "kk_filter_kernel", "E", r"kk_load_behind_wait\(src \+"),
         ("cnn.cu", "edge_in_kernel", "a.in", r"tc_load_behind_wait\([^;]*a\.in \+")]


@pytest.mark.parametrize("path,name,pointer,load", CASES)
def test_reads_of_the_kernel_in_front(path, name, pointer, load):
    params, body = _kernel(path, name)
    for p in params.split(","):
        if re.search(r"\b" + pointer + r"\s*$", p):
            assert "__restrict__" not in p, p
    assert not re.search(r"__ldg\([^;]*\b" + re.escape(pointer), body)
    wait = re.search(r"griddepcontrol\.wait|tc_grid_wait\(\)", body).end()
    assert re.search(load, body[wait:]) and not re.search(load, body[:wait])


@pytest.mark.parametrize("path,helper", [("kk.cu", "kk_load_behind_wait"), ("cnn.cu", "tc_load_behind_wait")])
def test_the_load_is_volatile_and_clobbers_memory(path, helper):
    text = open(os.path.join(CSRC, path)).read()
    m = re.search(helper + r"\([^)]*\)\s*\{(.*?)\n\}", text, flags=re.S)
    assert re.search(r'asm volatile\("ld\.global\.v2[^;]*;[^;]*:\s*"memory"\)', m.group(1), flags=re.S), m.group(1)
