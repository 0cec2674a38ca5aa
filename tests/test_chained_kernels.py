"""Order of the steps of a chained kernel's set-up, read from the sources.

A kernel that allocates tensor memory lets the next kernel's CTAs be placed only once
its own allocation is held by the whole CTA: a dependent CTA that allocated first
would wait for the kernel whose allocation it keeps waiting, and neither wait ends."""

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_20692_gb300", "csrc")


def _kernels():
    """(file, name, body) of every __global__ function, comments removed."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void[^{;]*?(\w+_kernel)\s*\([^{;]*\{", src):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            yield os.path.basename(path), m.group(1), src[m.end():i]


ALLOCATING = [(f, n, b) for f, n, b in _kernels() if "tmem_alloc(" in b]


def test_the_sources_are_read():
    assert {n for _, n, _ in ALLOCATING} == {"moments_kernel", "dnf_conv_kernel", "dnf_wgrad_kernel"}


@pytest.mark.parametrize("name,body", [(n, b) for _, n, b in ALLOCATING], ids=[n for _, n, _ in ALLOCATING])
def test_dependents_are_let_in_after_the_allocation(name, body):
    allocated = body.index("tmem_alloc(")
    held = body.index("__syncthreads()", allocated)
    assert "dep_launch()" not in body[:held]
    assert body.index("dep_launch()") > held
