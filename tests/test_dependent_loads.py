"""Kernels of this library may start while the kernel before them in the stream still runs, and
wait for it themselves.  What that kernel writes is then not read-only for their lifetime, so
none of them reads memory through the non-coherent path, whose contract that is: no __ldg, no
ld.global.nc, and no __restrict__ that would let the compiler choose it."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_05650_b200", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.h")) +
                 glob.glob(os.path.join(CSRC, "*.cuh")))


@pytest.mark.parametrize("path", SOURCES, ids=[os.path.basename(p) for p in SOURCES])
def test_no_non_coherent_loads(path):
    code = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
    assert not re.findall(r"__ldg\b|ld\.global[a-z0-9.]*\.nc\b|__restrict__", code)

