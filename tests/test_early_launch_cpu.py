"""What keeps early launches of dependent kernels safe, read from the kernels' source.

A kernel launched with the programmatic attribute may start before its predecessor is done:
it has to wait (pdl_enter) on every path, because the kernels after it rely on that wait
for the work of all kernels before it.  A kernel that lets its successor start early while it
takes tensor memory has to own its columns by then: the successor's blocks may share its
SMs, take columns and wait for it to complete, and an allocation has no time limit.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_15668_gb300", "csrc")


def _source(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _block(text, at):
    """The braces' content that opens at or after `at`."""
    at = text.index("{", at)
    depth, k = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[at + 1:k]
        k += 1


def _at_top(body, statement):
    """Places of a statement that every thread of the kernel reaches: outside nested blocks."""
    plain = re.sub(r'"(?:\\.|[^"\\])*"', lambda m: re.sub(r"[{}]", " ", m.group(0)), body)
    depth, places = 0, []
    for k, c in enumerate(plain):
        depth += {"{": 1, "}": -1}.get(c, 0)
        if depth == 0 and plain.startswith(statement, k):
            places.append(k)
    return places


def _kernels():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = _source(path)
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\)\s*)?(\w+)\s*\(", text):
            # the parameter list holds no braces
            found.append(pytest.param(text, m.group(1), _block(text, m.end()), id=f"{os.path.basename(path)}-{m.group(1)}"))
    return found


KERNELS = _kernels()


def test_all_kernels_are_seen():
    n = sum(_source(p).count("__global__") for p in glob.glob(os.path.join(CSRC, "*.cu")))
    assert len(KERNELS) == n and n > 40


@pytest.mark.parametrize("text, name, body", KERNELS)
def test_dependent_launches_wait(text, name, body):
    if re.search(name + r"(?:<[^;{}]*>)?\s*<<<", text) or name == "batch_kernel":
        return   # ordinary launches (batch_kernel's is cooperative)
    assert _at_top(body, "pdl_enter();"), name


@pytest.mark.parametrize("text, name, body", KERNELS)
def test_tensor_memory_is_owned_before_the_successor_may_start(text, name, body):
    triggers = [m.start() for m in re.finditer(r"griddepcontrol\.launch_dependents", body)]
    if not triggers or "tcgen05.alloc" not in body:
        return
    alloc = body.rindex("tcgen05.alloc")
    for k in triggers:
        assert any(alloc < b < k for b in _at_top(body, "__syncthreads();")), name
