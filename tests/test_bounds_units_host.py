"""Every translation unit that holds site kernels reports to lbm_bounds_report (no GPU): the kernels
are compiled into several units, each with a flag of its own for an index out of range."""
import ctypes
import os

import pytest

from paper_1611_03329_gb300 import build


def _holds_site_kernels(name):
    if name == "lbm_kernels.cu":
        return True
    lines = open(os.path.join(build.CSRC, name)).read().splitlines()
    inc = [ln.split('"')[1] for ln in lines if ln.startswith('#include "lbm_') and ln.endswith('.cu"')]
    return any(_holds_site_kernels(i) for i in inc)


@pytest.mark.parametrize("checked", [True, False])
def test_every_unit_with_site_kernels_reports(checked):
    units = [s for s in build.SOURCES if _holds_site_kernels(s)]
    assert "lbm_pair.cu" in units and "lbm_pair_first.cu" in units and "lbm_api.cu" not in units
    lib = ctypes.CDLL(build.build(checked=checked))
    assert lib.lbm_bounds_units() == (len(units) if checked else 0)
