"""Kernels that start under programmatic dependent launch, while the previous
launch may still be writing their input, must not promise the compiler that the
input is unchanged for the kernel's whole life (__restrict__ on const data,
__ldg, ld.global.nc): it could then be read through the read-only path, which
need not see those writes.  Checked in the sources, without their comments."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1603_01955_gb300", "csrc")


def code(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


CHAINED = sorted(p for p in glob.glob(os.path.join(CSRC, "*.cu")) if "griddepcontrol.wait" in code(p))


def test_the_chained_kernels_are_found():
    assert [os.path.basename(p) for p in CHAINED] == ["march.cu", "sweep.cu", "sweep_tma.cu", "tile.cu"]


@pytest.mark.parametrize("path", CHAINED + sorted(glob.glob(os.path.join(CSRC, "*.cuh"))), ids=os.path.basename)
def test_no_promise_of_unchanged_input(path):
    assert not re.search(r"const\s+\w+\s*\*\s*__restrict__|__ldg\b|ld\.global\.nc", code(path))
