"""Read-only loads (__ldg) in the kernels that are launched as a chain (no GPU).

Such a kernel is resident before the one ahead of it has finished, so buffers
of the build itself (records, scratch rows, group totals) are not read-only
while it runs; only the caller's mesh is."""
import os
import re

import pytest

import paper_1604_04689_gb300 as pkg

CSRC = os.path.join(os.path.dirname(pkg.__file__), "csrc")
CHAINED = ("nn_device.cuh", "nn_bulk.cuh", "nn_emit.cu", "nn_bucket.cuh", "nn_compact.cu", "nn_batch.cu")
# what the arguments of a read-only load may name: connectivity, element types and ranges, and pointers into them
MESH = re.compile(r"\b(conn|elem_type|elem_ptr|c4|nd)\b|reinterpret_cast<const int4\*>\(src\)|\bsrc \+ q\b")


@pytest.mark.parametrize("name", CHAINED)
def test_read_only_loads_are_of_the_mesh(name):
    with open(os.path.join(CSRC, name)) as f:
        lines = [re.sub(r"//.*", "", line) for line in f]
    bad = [(i + 1, line.strip()) for i, line in enumerate(lines)
           if any(not MESH.search(arg) for arg in re.findall(r"__ldg\(((?:[^()]|\([^()]*\))*)\)", line))
           or re.search(r"__ld(cg|cs|lu|cv)\(|ld\.global\.nc", line)]
    assert not bad, bad


def test_there_are_read_only_loads_to_look_at():
    with open(os.path.join(CSRC, "nn_emit.cu")) as f:
        assert "__ldg(" in f.read()
