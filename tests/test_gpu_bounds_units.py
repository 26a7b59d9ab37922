"""The bounds-checked build over the kernels that lattices run by default: pairs in odd and even rows,
D3Q15, the enthalpy model, the L2-hinted step, AA, node walls, batches, the fields and the residual.  No
access leaves its buffer, and the checked build computes what the ordinary one does."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import json, sys
import numpy as np
sys.path.insert(0, ROOT)
import paper_1611_03329_gb300 as gb
from lbm_inputs import cavity_problem, channel_problem, porosity_field
def cavity(nx, ny, nz, **kw):
    return dict(cavity_problem(nx, Ra=1e4, Da=1e-2, phi=0.6, Pr=0.71), ny=ny, nz=nz, **kw)
def field(pb):
    return dict(pb, phi_field=porosity_field(pb["nx"], pb["ny"], pb["nz"], seed=3).astype(np.float32))
per = dict(mapping="lattice", nu_e=0.05, alpha_f=0.03, gbeta=2e-3, phi=0.5, K=2.0, F_phi=0.4)
cases = {}
for tag, kw in (("fp32", {}), ("fp16", dict(storage="fp16")), ("bf16", dict(storage="bf16")), ("q15", dict(q=15))):
    for nx in (33, 34, 1, 2):
        cases[f"cavity_{nx}_{tag}"] = cavity(nx, 9, 8, **kw)
        cases[f"periodic_{nx}_{tag}"] = dict(per, nx=nx, ny=5, nz=4, **kw)
    for nx in (23, 24):
        cases[f"channel_{nx}_{tag}"] = dict(channel_problem(nx, 10, 9, Da=1e-2), **kw)
        cases[f"field_{nx}_{tag}"] = field(cavity(nx, 10, 9, **kw))
for nx in (13, 14, 1, 2):
    cases[f"aa_{nx}"] = cavity(nx, 9, 8, scheme="aa")
    cases[f"aa_per_{nx}"] = dict(per, nx=nx, ny=5, nz=4, scheme="aa")
cases["aa_field"] = field(cavity(15, 9, 8, scheme="aa"))
for nx in (24, 25):
    cases[f"melt_{nx}"] = dict(cavity_problem(nx, Ra=1e5, Da=None, phi=1.0, Pr=0.71, enthalpy=True, T_m=0.5,
                                              St=1.0, T_init=0.0), ny=11, nz=9)
for q in (19, 15):
    cases[f"nodes_{q}"] = dict(cavity(13, 11, 14, q=q, L=12.0), flow_bc=[4] * 6, heat_bc=[4, 4, 5, 5, 5, 5])
for tag, kw, n in (("fp32", {}, (70, 65, 72)), ("fp16", dict(storage="fp16"), (90, 80, 84)),
                   ("q15", dict(q=15), (78, 70, 73)), ("odd", {}, (77, 65, 65))):
    cases["hinted_" + tag] = cavity(*n, **kw)
cases["hinted_channel"] = dict(channel_problem(90, 80, 84, Da=1e-2), storage="fp16")
cases["hinted_field"] = field(cavity(90, 80, 84, storage="bf16"))
out = {}
def keep(name, lat):
    f, g = lat.populations()
    rho, u, T = lat.macros()
    out[name] = np.concatenate([f.ravel(), g.ravel(), rho.ravel(), u.ravel(), T.ravel()])
for name, pb in cases.items():
    lat = gb.Lattice(pb)
    lat.step(3)
    lat.residual()
    lat.step(2)
    out[name + "_r"] = np.array(lat.residual())
    keep(name, lat)
    lat.close()
names = [k for k in cases if "hinted" not in k]
lats = [gb.Lattice(cases[k]) for k in names]
batch = gb.Batch(lats)
batch.step(5)
for k, l in zip(names, lats):
    keep("batch_" + k, l)
np.savez(sys.argv[1], **out)
try:
    print(json.dumps({"first_bad": gb.bounds_report()}))
except gb.LbmError:
    print(json.dumps({"first_bad": None}))
"""


def _run(lib, out):
    env = dict(os.environ, LBM_LIBRARY=lib)
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + SCRIPT, out],
                       capture_output=True, text=True, env=env, cwd=ROOT, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads(r.stdout.strip().splitlines()[-1])["first_bad"], np.load(out)


def test_default_kernels_stay_in_bounds(tmp_path):
    from paper_1611_03329_gb300 import build

    bad, got = _run(build.build(checked=True), str(tmp_path / "checked.npz"))
    assert bad == -1, f"out-of-range site index {bad}"
    none, ref = _run(build.build(), str(tmp_path / "plain.npz"))
    assert none is None
    assert sorted(got.files) == sorted(ref.files)
    for k in ref.files:
        assert np.isfinite(ref[k]).all(), k
        assert np.array_equal(got[k], ref[k]), k
