"""lbm_macros_device into buffers of any 4-byte alignment, any of them absent: the fields are those that
lbm_macros returns, and nothing outside the buffers is written."""
import numpy as np
import pytest

from lbm_inputs import cavity_problem, channel_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import paper_1611_03329_gb300 as gb

    gb.build.build()
    gb.lib()
    return gb


CASES = {"even": dict(cavity_problem(24, Ra=1e4, Da=1e-2, phi=0.6), ny=9, nz=8),
         "odd": dict(cavity_problem(23, Ra=1e4, Da=1e-2, phi=0.6), ny=9, nz=7),
         "channel_fp16": dict(channel_problem(34, 10, 7, Da=1e-2), storage="fp16"),
         "q15": dict(cavity_problem(24, Ra=1e4, Da=1e-2, phi=0.6, q=15), ny=9, nz=8)}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("shift", [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 1), (1, None, 1), (None, 1, None)])
def test_fields_at_any_alignment(gb, name, shift):
    import torch

    pb = CASES[name]
    n = pb["nx"] * pb["ny"] * pb["nz"]
    lat = gb.Lattice(pb)
    lat.step(5)
    want = [a.ravel() for a in lat.macros()]
    bufs, ptrs = [], []
    for s, m in zip(shift, (n, 3 * n, n)):
        bufs.append(torch.full((m + 4,), -7.0, device="cuda"))
        ptrs.append(0 if s is None else bufs[-1].data_ptr() + 4 * s)
    torch.cuda.synchronize()
    lat.macros_device(*ptrs)
    lat.sync()
    for s, b, w in zip(shift, bufs, want):
        got = b.cpu().numpy()
        if s is None:
            assert (got == -7.0).all()
            continue
        assert np.array_equal(got[s:s + w.size], w)
        assert (got[:s] == -7.0).all() and (got[s + w.size:] == -7.0).all()
    lat.close()
