"""Kernels launched as programmatic dependents may be resident while the work before them still writes
their input, so nothing in them may claim that memory is constant for the kernel's lifetime: no
__restrict__ pointers, no read-only (non-coherent) loads."""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2002_05983_gb300", "csrc")


def _code(path):
    with open(path) as fh:
        s = fh.read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", s, flags=re.S)


DEPENDENT = sorted(p for p in glob.glob(os.path.join(CSRC, "*.cu*")) if "grid_dep_wait()" in _code(p))


def test_the_dependent_kernels_are_found():
    assert {os.path.basename(p) for p in DEPENDENT} >= {"pack.cu", "march_kernel.cuh", "sweep_kernel.cuh", "tile_kernel.cuh"}


@pytest.mark.parametrize("path", DEPENDENT, ids=os.path.basename)
def test_no_claim_of_constant_memory(path):
    assert not re.search(r"__restrict|__ldg\b|ld\.global\.nc", _code(path))
