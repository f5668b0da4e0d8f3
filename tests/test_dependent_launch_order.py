"""Kernels that take tensor memory let the next kernel of the stream start only afterwards.

The next kernel may allocate tensor memory before it waits for its predecessor.  Were it started while a CTA of the
predecessor had none yet, it could take the columns first, and each would wait for the other: tcgen05.alloc has no limit.
Nothing else keeps them apart (whether both fit on an SM depends on registers and shared memory), and the case cannot be
tried on a GPU, so the order is read from the sources: the allocation, a barrier of the whole CTA, then the trigger."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_03700_gb300", "csrc")
ALLOC = re.compile(r"tcgen05\.alloc|\btmem_alloc\(")
TRIGGER = re.compile(r"\bpdl_launch_dependents\(\)|\bPDL_ENTRY\(\)|griddepcontrol\.launch_dependents")
BARRIER = re.compile(r"__syncthreads\(\)")


def kernels():
    """(file, kernel, body without comments) of every kernel that allocates tensor memory."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        for m in re.finditer(r"__global__", text):
            start = text.index("{", m.end())
            depth, end = 0, start
            while True:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
                if depth == 0:
                    break
            if ALLOC.search(text, start, end):
                name = re.findall(r"(\w+)\s*\(", text[m.end():start])
                out.append(pytest.param(text[start:end], id=os.path.basename(path) + ":" + name[-1]))
    return out


def test_every_tensor_memory_kernel_is_found():
    assert len(kernels()) == 4


@pytest.mark.parametrize("body", kernels())
def test_trigger_follows_the_allocation(body):
    alloc = max(m.end() for m in ALLOC.finditer(body))
    triggers = [m.start() for m in TRIGGER.finditer(body)]
    barrier = BARRIER.search(body, alloc)
    assert barrier and triggers and min(triggers) > barrier.end()
