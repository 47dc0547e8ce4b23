"""What can be checked on the source of a kernel alone: a wrong order of these
steps hangs a GPU, so no test may run into it there."""

import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_2506_03781_gb300", "csrc", "*.cu*")))


def kernels(path):
    """The bodies of the __global__ functions of a file, without comments."""
    txt = re.sub(r"/\*.*?\*/|//[^\n]*", "", open(path).read(), flags=re.S)
    for m in re.finditer(r"__global__\b", txt):
        start = txt.index("{", re.compile(r"\)\s*\{").search(txt, m.end()).start())
        depth, i = 1, start + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(txt[i], 0)
            i += 1
        yield txt[start:i]


ALLOCATING = [(os.path.basename(p), body) for p in SOURCES for body in kernels(p) if "tc::alloc(" in body]


def test_the_kernels_with_tensor_memory_are_found():
    assert [name for name, _ in ALLOCATING] == ["uq_bcq_tc.cu"]


@pytest.mark.parametrize("name,body", ALLOCATING, ids=[name for name, _ in ALLOCATING])
def test_tensor_memory_is_taken_after_the_grid_wait_and_before_dependents_start(name, body):
    """A block must not hold tensor memory while it waits for a kernel whose
    blocks may still need some on the same SM, nor let a kernel start that may
    take some before this block has its own."""
    wait, alloc, start = (body.index(s) for s in ("inputs_ready();", "tc::alloc(", "dependents_may_start();"))
    assert wait < alloc < start
    assert "__syncthreads();" in body[alloc:start]         # one thread's signal counts for its block
    assert body.count("inputs_ready();") == body.count("dependents_may_start();") == 1
