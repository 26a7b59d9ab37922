"""lbm_step_kernel_name says which kernel steps a context, and lbm_reset_step_kernel brings back the
default choice that any selection ends (the two-site step of odd rows, D3Q15 and the enthalpy model)."""
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


def _cavity(nx, **kw):
    return dict(cavity_problem(nx, Ra=1e4, Da=1e-2, phi=0.6), ny=10, nz=9, **kw)


PAIR, AA = "step_pair_kernel", "aa_pair_pull_kernel, aa_pair_local_kernel"
MELT = dict(cavity_problem(9, Ra=1e5, Da=None, phi=1.0, Pr=0.71, enthalpy=True, T_m=0.5, St=1.0, T_init=0.0))
NODES = dict(cavity_problem(9, Ra=1e4, Da=1e-2, phi=0.6, L=8.0), flow_bc=[4] * 6, heat_bc=[4, 4, 5, 5, 5, 5])
CASES = {"even": (_cavity(8), "paired", PAIR), "odd": (_cavity(9), "plain", PAIR),
         "q15": (_cavity(8, q=15), "plain", PAIR), "melt": (MELT, "plain", PAIR),
         "aa": (_cavity(8, scheme="aa"), "plain", AA), "nodes": (NODES, "plain", "step_nee_kernel"),
         "channel": (channel_problem(34, 10, 7, Da=1e-2), "paired", PAIR)}


@pytest.mark.parametrize("name", sorted(CASES))
def test_name_of_the_kernel_that_runs(gb, name):
    pb, selected, runs = CASES[name]
    lat = gb.Lattice(pb)
    assert (lat.step_kernel, lat.step_kernel_name) == (selected, runs)
    lat.set_step_kernel("plain")
    one = {AA: AA, "step_nee_kernel": "step_nee_kernel"}.get(runs, "step_kernel")
    assert (lat.step_kernel, lat.step_kernel_name) == ("plain", one)
    lat.reset_step_kernel()
    assert (lat.step_kernel, lat.step_kernel_name) == (selected, runs)
    lat.close()


def test_name_of_the_tma_kernel_and_of_the_hinted_step(gb):
    lat = gb.Lattice(dict(channel_problem(64, 8, 6, Da=1e-2)))
    lat.set_step_kernel("tma")
    assert lat.step_kernel_name == "tma_step_kernel"
    lat.reset_step_kernel()
    assert lat.step_kernel_name == PAIR
    lat.close()
    lat = gb.Lattice(dict(_cavity(70), ny=65, nz=72))  # 34 MB a copy
    assert lat.step_kernel_name == PAIR + ", loads leave L2 first"
    lat.close()


def test_reset_steps_the_same_populations(gb):
    pb = _cavity(9)
    lats = [gb.Lattice(pb), gb.Lattice(pb)]
    lats[0].set_step_kernel(lats[0].step_kernel)
    for lat in lats:
        lat.step(3)
    lats[0].reset_step_kernel()
    for lat in lats:
        lat.step(4)
    for a, b in zip(lats[0].populations(), lats[1].populations()):
        assert np.array_equal(a, b)
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("nx", [70, 71])
def test_per_lattice_batch_takes_the_kernel_of_lbm_step(gb, nx):
    """A batch that steps its members by their own kernels, at a size that takes the hinted step."""
    pb = dict(_cavity(nx), ny=65, nz=72)
    lats = [gb.Lattice(pb) for _ in range(2)]
    batch = gb.Batch(lats[1:])
    batch.set_launch_mode("per_lattice")
    lats[0].step(7)
    batch.step(7)
    for a, b in zip(lats[0].populations(), lats[1].populations()):
        assert np.array_equal(a, b)
    batch.close()
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("storage,setup,hinted", [("bf16", "cavity", False), ("bf16", "field", True),
                                                  ("bf16", "channel", True), ("fp16", "cavity", True)])
def test_hinted_16_bit_steps(gb, storage, setup, hinted):
    """Which 16-bit steps take the L2 hint at a size whose copy fits L2 (35 MB), each against the
    one-site kernel, bit for bit."""
    pb = channel_problem(184, 60, 62, Da=1e-2) if setup == "channel" else dict(_cavity(90), ny=80, nz=94)
    pb = dict(pb, storage=storage)
    if setup == "field":
        pb["phi_field"] = np.linspace(0.4, 0.8, 90 * 80 * 94, dtype=np.float32)
    lats = [gb.Lattice(pb), gb.Lattice(pb)]
    assert lats[0].step_kernel_name == PAIR + (", loads leave L2 first" if hinted else "")
    lats[1].set_step_kernel("plain")
    for lat in lats:
        lat.step(5)
    for a, b in zip(lats[0].populations(), lats[1].populations()):
        assert np.array_equal(a, b)
    for lat in lats:
        lat.close()
