"""Kernels that may start while the one before still runs (those that call pdl_wait),
and the device functions that load for them, take nothing through const __restrict__
that a kernel of the same step writes: such loads are non-coherent, and may find what
an earlier launch left in L1. The exceptions are tables written outside the steps (the
reservoirs' and walls' entries) and the kernels that are never launched so."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2201_05280_gb300", "csrc")
TABLES = {"ghost", "hw", "g"}
ORDINARY = {"k_init", "k_ghost", "k_moments", "k_diag", "k_diag_pair", "k_diag_final"}


@pytest.mark.parametrize("name", ["rpk_device.cuh", "rpk_pair.cuh", "rpk_collide.cuh", "rpk_kernels.cuh", "rpk_brick.cuh"])
def test_loads_of_overlapping_kernels(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    for m in re.finditer(r"const\s[\w:<> ]*\*\s*__restrict__\s+(\w+)", text):
        function = re.findall(r"(\w+)\s*\((?=[^()]*$)", text[:m.start()])[-1]
        assert m.group(1) in TABLES or function in ORDINARY, (function, m.group(1))
