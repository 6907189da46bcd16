"""Bounded waits of the tensor-core kernels (CPU, the sources): a kernel's deadline starts after it holds its tensor memory and
after the kernels it was launched ahead of have ended, so that time spent behind other kernels is not counted as a wait of
its own that ran out."""

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2104_04547_gb300", "csrc")


def _kernels():
    """(file, kernel, body) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void[^;{]*?(\w+)\s*\((?:[^()]|\([^()]*\))*\)\s*\{", src):
            depth, at = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[at], 0)
                at += 1
            yield os.path.basename(path), m.group(1), src[m.end():at]


def _bounded():
    return [(f, k, b) for f, k, b in _kernels() if "globaltimer() + kWaitNs" in b]


def test_kernels_are_found():
    names = {k for _, k, _ in _bounded()}
    assert {"conv3d_tc_kernel", "conv3d_f32tc_kernel", "dense_f32tc_kernel"} <= names and len(names) >= 6, names


@pytest.mark.parametrize("file,kernel,body", _bounded(), ids=lambda v: v if isinstance(v, str) and len(v) < 40 else "")
def test_deadline_starts_after_the_waits_for_others(file, kernel, body):
    first = body.index("globaltimer() + kWaitNs")
    for waits in ("wait_prior()", "tmem_alloc("):
        if waits in body:
            assert body.index(waits) < first, (file, kernel, waits)
