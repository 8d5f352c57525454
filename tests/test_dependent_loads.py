"""Kernels that are resident while the kernel before them still writes their input (programmatic
dependent launch, the persistent ensemble) may not read it through the read-only path: no
ld.global.nc in their sources, by the intrinsic or by pointers declared __restrict__."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_00577_gb300", "csrc")


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_no_read_only_loads(name):
    with open(os.path.join(CSRC, name)) as fh:
        code = re.sub(r"//[^\n]*|/\*.*?\*/", "", fh.read(), flags=re.S)
    assert not re.search(r"__ldg\s*\(|ld\.global(\.\w+)*\.nc|__restrict__", code)
