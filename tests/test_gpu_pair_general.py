"""Steps of two sites per thread where the row length is odd, the flow lattice is D3Q15, the
enthalpy model runs or the scheme is AA: against the one-site kernel, bit for bit (both read the same stored values
and run the same explicitly rounded operations).  The sizes are those at which the pairing can
go wrong: a row of one site, rows that end in half a pair, rows shorter and longer than a warp,
a warp spanning several rows, every kind of face on the last site."""
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


def _melt(nx, ny, nz, **kw):
    return dict(cavity_problem(nx, Ra=1e5, Da=None, phi=1.0, Pr=0.71, enthalpy=True, T_m=0.5,
                               St=1.0, T_init=0.0), ny=ny, nz=nz, **kw)


def _periodic(nx, ny, nz):
    return dict(nx=nx, ny=ny, nz=nz, mapping="lattice", nu_e=0.05, alpha_f=0.03, gbeta=2e-3, phi=0.5,
                K=2.0, F_phi=0.4, sigma=1.7, accel=[2e-4, -1e-4, 5e-5])


def _lid(nx, ny, nz):
    return _cavity(nx, ny, nz, flow_bc=[2, 2, 1, 2, 1, 2],
                   face_u=[(0, .01, .01), (0, -.01, 0), (0, 0, 0), (.01, 0, .02), (0, 0, 0), (.01, .02, 0)])


def _field(pb):
    phi = porosity_field(pb["nx"], pb["ny"], pb["nz"], seed=5).astype(np.float32)
    return dict(pb, phi_field=phi, alpha_m=0.02)


ODD = {
    "cavity_33x21x19": _cavity(33, 21, 19), "cavity_63x5x4": _cavity(63, 5, 4),
    "cavity_1x9x9": _cavity(1, 9, 9), "cavity_3x17x4": _cavity(3, 17, 4),
    "channel_41x17x13": channel_problem(41, 17, 13, Da=1e-2),
    "channel_T_out_67x9x8": dict(channel_problem(67, 9, 8, Da=1e-2), heat_bc=[2, 3, 2, 2, 0, 0]),
    "channel_walls_23x9x8": dict(channel_problem(23, 9, 8, Da=1e-2), flow_bc=[2, 3, 1, 2, 1, 1],
                                 heat_bc=[2, 2, 2, 2, 1, 1],
                                 face_u=[(0.01, 0, 0)] + [(0, 0, 0)] * 2 + [(0.02, 0, 0)] + [(0, 0, 0)] * 2),
    "periodic_31x7x5": _periodic(31, 7, 5), "periodic_1x8x8": _periodic(1, 8, 8),
    "lid_21x11x12": _lid(21, 11, 12), "field_33x12x9": _field(_cavity(33, 12, 9)),
    "field_channel_23x10x9": _field(channel_problem(23, 10, 9, Da=1e-2)),
}
CASES = {f"{k}/{s}": dict(pb, storage=s) for k, pb in ODD.items() for s in ("fp32", "fp16", "bf16")}
CASES |= {f"{k}/q15": dict(pb, q=15) for k, pb in ODD.items()}
CASES |= {f"{k}/aa": dict(pb, scheme="aa") for k, pb in ODD.items() if "channel" not in k}
CASES |= {"aa_even/" + k: dict(pb, scheme="aa") for k, pb in
          {"cavity": _cavity(34, 9, 8), "periodic": _periodic(38, 5, 3), "lid": _lid(20, 9, 8),
           "pair": _periodic(2, 9, 8), "field": _field(_cavity(24, 9, 8))}.items()}
CASES |= {"q15_even/" + k: dict(pb, q=15) for k, pb in
          {"cavity": _cavity(34, 9, 8), "channel": channel_problem(40, 9, 8, Da=1e-2), "lid": _lid(20, 9, 8),
           "field": _field(_cavity(24, 9, 8))}.items()}
CASES |= {f"melt_{n}{tag}": _melt(n, 11, 9, **kw) for n in (24, 25)
          for tag, kw in (("", {}), ("_mushy", dict(T_s=0.4, T_l=0.6, alpha_ratio=1.7)),
                          ("_off", dict(flow_off=True)))}


@pytest.mark.parametrize("name", sorted(CASES))
def test_two_sites_per_thread_match_one(gb, name):
    pb = CASES[name]
    rng = np.random.default_rng(3)
    nx, ny, nz = pb["nx"], pb["ny"], pb["nz"]
    T = 0.5 + 0.3 * rng.uniform(-1, 1, (nz, ny, nx))
    u = 0.02 * rng.uniform(-1, 1, (3, nz, ny, nx))
    got = []
    for kernel in (None, "plain"):
        lat = gb.Lattice(pb if kernel is None else dict(pb, scheme="pingpong"))
        lat.init_equilibrium(T_field=T, u_field=u)
        if kernel:
            lat.set_step_kernel(kernel)
        lat.step(3)
        lat.step(4)
        got.append(lat.populations())
        lat.close()
    assert np.isfinite(got[0][0]).all()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("storage,field,shape,q", [
    ("fp32", False, (70, 65, 72), 19), ("fp32", True, (70, 65, 72), 19), ("fp16", False, (90, 80, 84), 19),
    ("bf16", True, (90, 80, 84), 19), ("fp32", False, (77, 65, 65), 19), ("fp32", False, (78, 70, 73), 15)])
def test_l2_hinted_step_matches_one_site(gb, storage, field, shape, q):
    """The paired step with loads that leave L2 first (one population copy of 33-36 MB, just above
    the size at which it is chosen) against the one-site kernel, bit for bit."""
    pb = _cavity(*shape, storage=storage, q=q)
    pb = _field(pb) if field else pb
    got = []
    for kernel in (None, "plain"):
        lat = gb.Lattice(pb)
        if kernel:
            lat.set_step_kernel(kernel)
        lat.step(5)
        got.append(lat.populations())
        lat.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("name", ["cavity_33x21x19/fp32", "channel_41x17x13/fp16", "field_33x12x9/aa", "melt_25",
                                  "cavity_1x9x9/fp32", "lid_21x11x12/q15"])
def test_residual_is_that_of_the_fields(gb, name):
    """lbm_residual against the FP64 norms of the fields lbm_macros returns (the same FP32 values;
    at most 1e5 terms summed in another order: 1e-11 relative is far above the rounding)."""
    pb = CASES[name]
    rng = np.random.default_rng(4)
    lat = gb.Lattice(pb)
    lat.init_equilibrium(T_field=0.5 + 0.3 * rng.uniform(-1, 1, (pb["nz"], pb["ny"], pb["nx"])))
    lat.step(3)
    assert lat.residual() == (np.inf, np.inf)
    _, u0, T0 = lat.macros()
    lat.step(2)
    _, u1, T1 = lat.macros()
    ru, rT = lat.residual()
    lat.close()
    for r, new, old in ((ru, u1, u0), (rT, T1, T0)):
        new, old = new.astype(np.float64), old.astype(np.float64)
        assert r == pytest.approx(np.sqrt(((new - old) ** 2).sum() / (new ** 2).sum()), rel=1e-11)


@pytest.mark.parametrize("scheme", ["pingpong", "aa"])
def test_step_graphs_match_launches(gb, scheme):
    """Calls long enough for the replayed step graphs (chosen after 500 steps in calls of 32 or
    more), from either parity and across a change of medium, against calls too short for them."""
    pb = _cavity(24, 10, 9, scheme=scheme)
    lats = [gb.Lattice(pb), gb.Lattice(pb)]
    for phi in (0.6, 0.7):
        for lat in lats:
            lat.set_medium(phi=phi, F_phi=-1.0)
        for chunk in (600, 64, 33, 64, 67):
            lats[0].step(chunk)
            for _ in range(chunk // 31):
                lats[1].step(31)
            lats[1].step(chunk % 31)
    assert lats[0].steps == lats[1].steps
    for a, b in zip(lats[0].populations(), lats[1].populations()):
        assert np.array_equal(a, b)
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("kind", ["nodes_all", "nodes_y", "nodes_x"])
def test_node_walls_in_their_own_blocks_match_the_batched_step(gb, kind):
    """The single-lattice node-wall step (wall sites in blocks of their own) against the batched
    one (wall and fluid sites in one block), which share nee_site: bit for bit."""
    n = 13
    pb = dict(cavity_problem(n, Ra=1e4, Da=1e-2, phi=0.6, L=n - 1.0), ny=n - 2, nz=n + 1)
    pb.update({"nodes_all": dict(flow_bc=[4] * 6, heat_bc=[4, 4, 5, 5, 5, 5]),
               "nodes_y": dict(flow_bc=[1, 1, 4, 4, 0, 0], heat_bc=[2, 2, 4, 5, 0, 0]),
               "nodes_x": dict(flow_bc=[4, 1, 1, 4, 1, 2], heat_bc=[4, 2, 1, 4, 1, 2],
                               face_u=[(0, 0, 0)] * 3 + [(.01, 0, .01), (0, 0, 0), (0, .01, 0)])}[kind])
    lats = [gb.Lattice(pb), gb.Lattice(pb)]
    lats[0].step(9)
    batch = gb.Batch(lats[1:])
    batch.step(9)
    for a, b in zip(lats[0].populations(), lats[1].populations()):
        assert np.array_equal(a, b)
    batch.close()
    for lat in lats:
        lat.close()
