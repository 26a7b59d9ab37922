"""The kernels of lattices of more than ~82 M sites (one site per thread, a pointer per population plane),
chosen on small lattices by a test hook, against the paired kernels those run by default: single steps,
AA, batches, fields and residuals."""
import numpy as np
import pytest

from lbm_inputs import cavity_problem, channel_problem, porosity_field

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import paper_1611_03329_gb300 as gb

    gb.build.build()
    gb.lib()
    return gb


def _cavity(nx, ny, nz, **kw):
    return dict(cavity_problem(nx, Ra=1e5, Da=1e-2, phi=0.6, Pr=0.71), ny=ny, nz=nz, **kw)


def _periodic(nx, ny, nz, **kw):
    return dict(nx=nx, ny=ny, nz=nz, mapping="lattice", nu_e=0.05, alpha_f=0.03, gbeta=2e-3, phi=0.5,
                K=2.0, F_phi=0.4, sigma=1.7, accel=[2e-4, -1e-4, 5e-5], **kw)


def _lid(nx, ny, nz, **kw):
    return _cavity(nx, ny, nz, flow_bc=[2, 2, 1, 2, 1, 2],
                   face_u=[(0, .01, .01), (0, -.01, 0), (0, 0, 0), (.01, 0, .02), (0, 0, 0), (.01, .02, 0)], **kw)


def _field(pb):
    phi = porosity_field(pb["nx"], pb["ny"], pb["nz"], seed=5).astype(np.float32)
    return dict(pb, phi_field=phi, alpha_m=0.02)


CASES = {}
for tag, kw in (("fp32", {}), ("fp16", dict(storage="fp16")), ("bf16", dict(storage="bf16")), ("q15", dict(q=15))):
    CASES |= {f"cavity/{tag}": _cavity(34, 9, 8, **kw), f"cavity_odd/{tag}": _cavity(33, 11, 7, **kw),
              f"channel/{tag}": dict(channel_problem(41, 10, 9, Da=1e-2), **kw),
              f"lid/{tag}": _lid(20, 9, 8, **kw), f"periodic/{tag}": _periodic(38, 5, 3, **kw),
              f"field/{tag}": _field(_cavity(24, 9, 8, **kw)),
              f"field_channel/{tag}": _field(dict(channel_problem(24, 10, 9, Da=1e-2), **kw))}
CASES |= {"cavity/aa": _cavity(34, 9, 8, scheme="aa"), "cavity_odd/aa": _cavity(33, 11, 7, scheme="aa"),
          "lid/aa": _lid(20, 9, 8, scheme="aa"), "periodic/aa": _periodic(31, 5, 4, scheme="aa"),
          "field/aa": _field(_cavity(24, 9, 8, scheme="aa")),
          "melt": dict(cavity_problem(24, Ra=1e5, Da=None, phi=1.0, Pr=0.71, enthalpy=True, T_m=0.5, St=1.0,
                                      T_init=0.0), ny=11, nz=9),
          "nodes": dict(_cavity(13, 11, 14, L=12.0), flow_bc=[4] * 6, heat_bc=[4, 4, 5, 5, 5, 5])}


def _pair(gb, pb):
    """The lattice twice, the second with the wide kernels, from the same seeded fields."""
    rng = np.random.default_rng(3)
    T = 0.5 + 0.3 * rng.uniform(-1, 1, (pb["nz"], pb["ny"], pb["nx"]))
    u = 0.02 * rng.uniform(-1, 1, (3, pb["nz"], pb["ny"], pb["nx"]))
    lats = [gb.Lattice(pb), gb.Lattice(pb)]
    lats[1].test_wide_offsets()
    for lat in lats:
        lat.init_equilibrium(T_field=T, u_field=u)
    return lats


def _same(a, b):
    for x, y in zip(a, b):
        assert np.isfinite(x).all() and np.array_equal(x, y)


@pytest.mark.parametrize("name", sorted(CASES))
def test_wide_steps_fields_and_residuals(gb, name):
    pb = CASES[name]
    lats = _pair(gb, pb)
    want = ("aa_pull_kernel, aa_local_kernel" if pb.get("scheme") == "aa" else
            "step_nee_kernel" if name == "nodes" else "step_kernel")
    assert lats[1].step_kernel_name == want
    res = []
    for lat in lats:
        lat.step(3)
        assert lat.residual() == (np.inf, np.inf)
        lat.step(4)
        res.append(lat.residual())
    _same(lats[0].populations(), lats[1].populations())
    _same(lats[0].macros(), lats[1].macros())
    # FP64 sums of the same FP32 fields in another order (at most 1e4 terms of one sign)
    assert res[1] == pytest.approx(res[0], rel=1e-11)
    lats[1].test_wide_offsets(False)
    assert lats[1].step_kernel_name == lats[0].step_kernel_name
    for lat in lats:
        lat.step(2)
    _same(lats[0].populations(), lats[1].populations())
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("rows", [1, 3])
def test_wide_batches(gb, rows):
    """All of them in one batch, against the same lattices stepped alone by the default kernels."""
    pairs = [_pair(gb, pb) for pb in CASES.values()]
    batch = gb.Batch([p[1] for p in pairs])
    batch.set_block(64, rows)
    batch.step(5)
    for p in pairs:
        p[0].step(5)
        _same(p[0].populations(), p[1].populations())
    batch.close()
    for p in pairs:
        for lat in p:
            lat.close()
