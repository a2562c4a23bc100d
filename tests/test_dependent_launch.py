"""Kernels that are launched while the kernel before them still runs must not
load through the read-only path: that kernel may still write what they read, and
the read-only path is neither ordered by griddepcontrol.wait nor meant for data
written during the kernel's life."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1907_13088_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _dependent():
    """Files with a dependent launch of their own or through an included header."""
    files = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
    waits = {f for f in files if "griddepcontrol.wait" in _code(f)}
    uses = {f for f in files for h in re.findall(r'#include "(\w+\.cuh)"', _code(f)) if h in waits}
    return sorted(waits | uses)


def test_some_kernels_are_dependent():
    assert {"adjoint.cu", "tile2d.cu", "adj_tile2d.cu"} <= set(_dependent())


@pytest.mark.parametrize("name", _dependent())
def test_no_read_only_loads(name):
    code = _code(name)
    assert "__ldg" not in code and "ld.global.nc" not in code and "const float *__restrict__" not in code
    assert not re.search(r"const T \*\s*__restrict__", code)
