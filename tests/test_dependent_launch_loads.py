"""Kernels launched as programmatic dependents are alive while the kernels before them still write.  What they read of those
kernels' results must therefore not go through the read-only data path, which is defined only for data that does not change
while the kernel lives: no __ldg, no ld.global.nc, no `const ... __restrict__` input in a source file of such kernels."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_01831_b200", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _includes(name):
    return {i for i in re.findall(r'#include "([^"]+)"', _code(name)) if os.path.exists(os.path.join(CSRC, i))}


def _dependents():
    """Files with a kernel that waits for the grids before it, what they include and what includes them."""
    names = [n for n in sorted(os.listdir(CSRC)) if n.endswith((".cu", ".cuh"))]
    own = {n for n in names if n != "lynx_common.cuh" and re.search(r"\bpdl_(?:begin|wait)\(\)|griddepcontrol\.wait", _code(n))}
    units = own | {n for n in names if _includes(n) & own}
    return sorted(units.union(*(_includes(n) for n in units)))


def test_there_are_dependent_kernels():
    assert {"attention.cu", "attention_i8.cuh", "attention_f16.cuh", "lynx_common.cuh"} <= set(_dependents())


@pytest.mark.parametrize("name", _dependents())
def test_no_read_only_loads(name):
    code = _code(name)
    found = re.findall(r"__ldg\s*\(|ld\.global\.nc[\w.]*|\bconst\s+\w+\s*\*\s*__restrict__\s*\w+", code)
    assert not found, found
