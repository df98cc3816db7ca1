"""Kernels that use tensor memory and are launched chained (programmatic serialisation): a block lets the next
kernel's blocks in only after its own allocation and a barrier of the block.  The next kernel's blocks hold their
columns while they wait, so the other order can leave both sides waiting for ever on an SM whose 512 columns are
taken.  Read from the sources: nothing here runs on a GPU."""
import glob
import os
import re

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_0903_3053_gb300", "csrc")
RELEASE = re.compile(r"\bchain_wait\(\s*(?!false\b)|\bchain_release\(\)|griddepcontrol\.launch_dependents")


def kernels():
    """(name, body) of every __global__ function, comments taken out."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        for m in re.finditer(r"__global__", text):
            depth, i = 0, text.index("{", m.end())
            name = re.findall(r"(k_\w+)\s*\(", text[m.end():i])[0]
            for j in range(i, len(text)):
                depth += {"{": 1, "}": -1}.get(text[j], 0)
                if depth == 0:
                    break
            out.append((name, text[i:j + 1]))
    return out


TENSOR = [(n, b) for n, b in kernels() if "tmem_alloc(" in b]


def test_the_tensor_memory_kernels_are_found():
    assert {n for n, _ in TENSOR} >= {"k_layer1_tc", "k_conv_runs", "k_dw32_tc"}


@pytest.mark.parametrize("name,body", TENSOR, ids=[n for n, _ in TENSOR])
def test_successors_come_in_after_the_allocation(name, body):
    alloc = [m.start() for m in re.finditer(r"tmem_alloc\(", body)]
    release = [m.start() for m in RELEASE.finditer(body)]
    assert len(alloc) == 1
    assert all(r > body.index("__syncthreads()", alloc[0]) for r in release), name
