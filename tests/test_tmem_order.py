"""Tensor memory and dependent launch, read from the kernel sources: a blocking
allocation before griddepcontrol.wait, or a launch_dependents before the barrier
behind the allocation, can leave two kernels of a stream waiting for each other."""
import glob
import os
import re

import pytest

from paper_2603_27569_gb300 import build

ALLOC = re.compile(r"tcgen05\.alloc|tmem_alloc_warp\s*\(|\.allocate\(\)")
BARRIER = re.compile(r"__syncthreads\(\)|\.publish\(\)")
SOURCES = sorted(glob.glob(os.path.join(build.CSRC, "*.cu")) +
                 glob.glob(os.path.join(build.CSRC, "*.cuh")))


def strip_comments(text):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def block(text, start):
    """The braces' content from the first brace after `start`."""
    at = i = text.index("{", start)
    depth = 0
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
        if depth == 0:
            return text[at:i]


def kernels():
    for path in SOURCES:
        text = strip_comments(open(path).read())
        for m in re.finditer(r"__global__", text):
            brace, semi = text.find("{", m.end()), text.find(";", m.end())
            if brace < 0 or (0 <= semi < brace):
                continue  # a declaration
            name = re.findall(r"(\w+)\s*\(", text[m.end():brace])[-1]
            body = block(text, m.end())
            # objects built in the kernel: their constructors run in place
            for cls in set(re.findall(r"\b([A-Z]\w+)<[^;{}]*>\s+\w+\(", body)):
                for c in re.finditer(rf"__forceinline__\s+{cls}\(", text):
                    body = re.sub(rf"\b{cls}<[^;{{}}]*>\s+\w+\(", block(text, c.end()) + "(", body, count=1)
            yield os.path.basename(path), name, body


ALLOCATING = [k for k in kernels() if ALLOC.search(k[2])]


def test_every_allocating_kernel_is_seen():
    assert {n for _, n, _ in ALLOCATING} >= {"filter_fwd_kernel", "filter_bwd_kernel",
                                             "filter_step_kernel", "tc_kernel", "tmem2_kernel"}


@pytest.mark.parametrize("path,name,body", ALLOCATING, ids=[k[1] for k in ALLOCATING])
def test_wait_then_allocate_then_barrier_then_trigger(path, name, body):
    wait = body.index("griddepcontrol.wait")
    allocs = list(ALLOC.finditer(body))
    assert wait < allocs[0].start(), "allocates before the kernel before it has finished"
    barrier = BARRIER.search(body, allocs[-1].end())
    trigger = body.find("griddepcontrol.launch_dependents")
    assert barrier and (trigger < 0 or barrier.end() < trigger), "releases dependents too early"


def test_publish_is_a_barrier():
    text = strip_comments(open(os.path.join(build.CSRC, "filter_fused.cu")).read())
    body = block(text, text.index("void publish()"))
    assert "__syncthreads()" in body
