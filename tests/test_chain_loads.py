"""Kernels that may start before their predecessor has ended read what it writes with coherent loads.

A read-only load (`__ldg`, or a `const T* __restrict__` kernel parameter, which the compiler turns into one) is defined only
for memory that nobody writes during the kernel's lifetime."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_05124_b200", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
# written once at context creation
TABLES = {"maps", "stage_ids", "tile_start", "order", "segs"}
# fixed from before the first launch of a chain to its end: token ids (copied in by the launch in front of the chain),
# biases (written by the update, a chain of its own), tables
FIXED = {"ids", "bias", "order", "tile_start"}


def _text(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


@pytest.mark.parametrize("name", SOURCES)
def test_kernel_parameters(name):
    text = _text(name)
    starts = [m.start() for m in re.finditer(r"__global__", text)]
    for a, b in zip(starts, starts[1:] + [len(text)]):
        kernel = text[a:b]
        if "pdl_wait()" not in kernel:
            continue
        head = kernel[:kernel.index("{")]
        for m in re.finditer(r"const [\w:]+\*\s*__restrict__ (\w+)", head):
            assert m.group(1) in TABLES, (name, m.group(0))


@pytest.mark.parametrize("name", SOURCES)
def test_read_only_loads(name):
    for m in re.finditer(r"__ldg\((?:reinterpret_cast<[^>]*>\()?(\w+)", _text(name)):
        assert m.group(1) in FIXED, (name, m.group(0))
