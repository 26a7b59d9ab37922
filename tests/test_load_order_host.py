"""Loads of what the previous time step wrote come after the wait for it.  The step kernels are
programmatic dependent launches: their blocks start while the previous step still writes, and
griddepcontrol.wait orders ordinary loads only.  A read-only load (__ldg, ld.global.nc) or an inline
load without `volatile` and a memory clobber may be issued above the wait, so the sources hold
neither for populations, temperature planes and the outflow history."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1611_03329_gb300", "csrc")
UNITS = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
# memory that no step writes: the porosity field, and a batch's map from blocks to lattices
CONSTANT = re.compile(r"__ldg\((p\.phi_field|blk_lat)\b")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


@pytest.mark.parametrize("name", UNITS)
def test_inline_loads_are_ordered(name):
    for stmt in re.findall(r"\basm\b[^;]*?\([^;]*?\bld\.global.*?\)\s*;", _code(name), flags=re.S):
        assert ".nc" not in stmt and "volatile" in stmt and '"memory"' in stmt, stmt


@pytest.mark.parametrize("name", UNITS)
def test_read_only_loads_are_of_constant_memory(name):
    for m in re.finditer(r"__ldg\(", _code(name)):
        assert CONSTANT.match(_code(name)[m.start():]), _code(name)[m.start():m.start() + 60]


def test_the_wait_is_ordered():
    code = _code("lbm_kernels.cu")
    assert re.search(r'asm volatile\("griddepcontrol\.wait;" ::: "memory"\);', code)
