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


@pytest.mark.parametrize("name,body", ALLOCATING, ids=[name for name, _ in ALLOCATING])
def test_after_a_timeout_exactly_what_was_started_is_waited_for(name, body):
    """The copies of the last stages, none that was never started, and the last
    product of each buffer, before tensor memory is given back.  Only an expired
    wait gets there, so it is read from the source."""
    txt = open(os.path.join(os.path.dirname(SOURCES[0]), name)).read()
    issuer = body[body.index("if (issuer) {"):body.index("!issuer; ++mt")]
    first = re.search(r"drain\(full, (.*), copies\)", txt).group(1)
    total = re.search(r"const int total = (.*?), copies = (.*?);", issuer)
    c = lambda e: re.sub(r"^(.*?) \? (.*) : (.*)$", r"(\2) if (\1) else (\3)", e).replace("copies", "made")  # noqa: E731
    # the loop starts one stage each time the last one of a slot has been read, as long as some are left
    assert "stage + kTcStages < my_tiles * spt) copy(wg, stage + kTcStages);" in issuer
    for stages in range(7):
        started = min(2, stages)
        for stage in range(stages + 1):
            made = eval(c(total.group(2)), {}, {"stage": stage, "kTcStages": 2, "total": stages})
            assert made == started
            assert list(range(eval(c(first), {}, {"made": made, "kTcStages": 2}), made)) == list(range(started))[-2:]
            started += stage + 2 < stages
    assert total.group(1) == "staged ? my_tiles * spt : 0"
    # a commit flips the parity bit of its buffer: the last one's phase has the other parity
    assert issuer.count("tc::commit(") == issuer.count("ph ^= 1u << b;") == 1
    assert "tma::bar_wait(tma::smem_addr(&done[k]), ((ph >> k) & 1u) ^ 1u)" in txt
    tail = body[body.index("!issuer; ++mt"):]
    assert re.search(r"__syncthreads\(\);\s+if \(dead && warp == 0 && lane < n_wg\) tc_drain\(", tail)
    assert tail.index("tc_drain(") < tail.rindex("__syncthreads();") < tail.index("tc::dealloc(")
