"""Kernels that may become resident while the kernel before them still runs
(chain() of csrc/pmpm_impl.cuh) read what that kernel writes through plain
pointers: `const T* __restrict__` promises that nothing writes there while the
kernel lives, and lets the compiler load it early and through the read-only path.
Tables that are made once, before any step, may keep it."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_03931_gb300", "csrc")
MADE_ONCE = {"table", "tw", "twiddles", "E"}


def chained_kernels():
    found = []
    for unit in sorted(os.listdir(CSRC)):
        if not unit.endswith((".cu", ".cuh")):
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, unit)).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(k_\w+)\s*\(([^{]*)\)\s*\{", text):
            name, params, rest = m.group(1), m.group(2), text[m.end():]
            if re.match(r"\s*chain_(begin|wait)\(\);", rest):
                found.append((unit, name, params))
    return found


def test_the_chained_kernels_are_found():
    names = {name for _, name, _ in chained_kernels()}
    assert {"k_step_begin", "k_column", "k_tile", "k_scan_apply", "k_scatter", "k_coarse_z", "k_pk_z"} <= names


@pytest.mark.parametrize("unit,name,params", chained_kernels(), ids=lambda v: v if str(v).startswith("k_") else "")
def test_only_tables_are_read_only(unit, name, params):
    promised = re.findall(r"const\s+\w+(?:\s+\w+)*\s*\*\s*__restrict__\s+(\w+)", params)
    assert set(promised) <= MADE_ONCE, (unit, name)
