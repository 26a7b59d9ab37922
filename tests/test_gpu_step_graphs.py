"""The replayed step graphs (chosen after 500 steps in calls of 32 or more) beside a caller's own stream
captures: a capture of the context's stream records its steps as launches, and a capture of another
stream is left alone by the building of a graph."""
import numpy as np
import pytest

from lbm_inputs import cavity_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import paper_1611_03329_gb300 as gb

    gb.build.build()
    gb.lib()
    return gb


def _cavity(**kw):
    return dict(cavity_problem(20, Ra=1e5, Da=1e-2, phi=0.6, Pr=0.71), ny=10, nz=9, **kw)


def _launched(gb, pb, steps):
    """The populations after `steps` steps in calls too short for a graph."""
    lat = gb.Lattice(pb)
    for _ in range(steps // 31):
        lat.step(31)
    lat.step(steps % 31)
    out = lat.populations()
    lat.close()
    return out


def _same(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
@pytest.mark.parametrize("scheme", ["pingpong", "aa"])
def test_a_capture_of_another_stream_survives(gb, mode, scheme):
    import torch

    pb = _cavity(scheme=scheme)
    lat = gb.Lattice(pb)
    for chunk in (62,) * 8:  # one more call and the graph is due
        lat.step(chunk)
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode=mode):
        x += 1
        lat.step(64)  # builds the graph on the lattice's own stream
        lat.set_launch(128)  # drops it
        x += 1
    g.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [2.0] * 8
    got = lat.populations()
    lat.close()
    _same(got, _launched(gb, pb, 8 * 62 + 64))


def test_a_change_before_every_chunk_builds_no_graph(gb):
    """A graph is due again only 500 steps after the last change of what its launches hold."""
    lat = gb.Lattice(_cavity())
    lat.step(640)
    lat.step(64)
    built = lat.test_step_graphs()[0]
    assert built == 1
    for phi in np.linspace(0.5, 0.7, 10):
        lat.set_medium(phi=phi, F_phi=-1.0)
        lat.step(64)
        lat.set_launch(128)
        lat.step(64)
    assert lat.test_step_graphs()[0] == built
    lat.step(640)
    assert lat.test_step_graphs()[0] == built + 1
    lat.close()


CHANGES = {
    "none": lambda gb, lat: None,
    "block_threads": lambda gb, lat: lat.set_launch(128),
    "ordinary_launches": lambda gb, lat: lat.set_launch(0, 0),
    "one_site": lambda gb, lat: lat.set_step_kernel("plain"),
    "medium": lambda gb, lat: lat.set_medium(phi=0.7, F_phi=-1.0),
    "to_aa": lambda gb, lat: _to_aa(gb, lat),
}


def _to_aa(gb, lat):
    batch = gb.Batch([lat])
    batch.set_scheme("aa")
    batch.close()


@pytest.mark.parametrize("change", sorted(CHANGES))
def test_replayed_steps_match_launches_across_a_change(gb, change):
    """Steps from replayed graphs before and after a change of what a graph holds, against a second
    lattice stepped in calls too short for one."""
    lats = [gb.Lattice(_cavity()), gb.Lattice(_cavity())]
    for part in range(2):
        before = lats[0].test_step_graphs()[1]
        for chunk in (600, 33, 64, 67):
            lats[0].step(chunk)
            for _ in range(chunk // 31):
                lats[1].step(31)
            lats[1].step(chunk % 31)
        replayed = lats[0].test_step_graphs()[1] - before
        assert replayed == (0 if part and change == "ordinary_launches" else 18 + 1 + 2 + 2)
        assert lats[1].test_step_graphs() == (0, 0)
        if part == 0:
            for lat in lats:
                CHANGES[change](gb, lat)
    assert lats[0].steps == lats[1].steps
    _same(lats[0].populations(), lats[1].populations())
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("scheme", ["pingpong", "aa"])
def test_a_capture_of_its_own_stream_records_launches(gb, scheme):
    """lbm_step inside a capture of the context's stream, with the step graph built: the capture records
    the steps (an even number), and each replay takes them once more."""
    import torch

    pb = _cavity(scheme=scheme)
    stream = torch.cuda.Stream()
    lat = gb.Lattice(pb, stream=stream.cuda_stream)
    lat.step(640)
    counts = lat.test_step_graphs()
    assert counts[1] == 20
    lat.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        lat.step(64)  # recorded, not run
    assert lat.test_step_graphs() == counts
    with torch.cuda.stream(stream):
        g.replay()
        g.replay()
    lat.step(64)
    got = lat.populations()
    lat.close()
    del g
    _same(got, _launched(gb, pb, 640 + 64 + 64 + 64))
