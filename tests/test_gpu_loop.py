"""The step loop of small meshes (swe_loop.cuh: all steps of a call in one
cooperative launch) against the kernels launched step by step, bit for bit.
A mesh with nothing chosen about its launches takes the loop from 4 steps on;
graph_steps=-1 (no graphs) keeps it on single launches."""
import numpy as np
import pytest

from paper_2010_14416_gb300 import build as libbuild
from paper_2010_14416_gb300 import capi
from paper_2010_14416_gb300 import meshgen as mg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    libbuild.build()
    return capi.load()


def _mesh(mi, precision, **kw):
    m = capi.Mesh(mi.nodes, mi.tris, mi.z, mi.manning, precision=precision, **kw)
    for pairs, kind, value in mi.bcs:
        m.set_bc(pairs, kind, value)
    m.set_state(mi.h.astype(m.dtype), mi.hu.astype(m.dtype), mi.hv.astype(m.dtype))
    return m


def _equal(a, b):
    assert all(np.array_equal(x, y) for x, y in zip(a.get_state(), b.get_state()))
    ia, ib = a.info(), b.info()
    for k in ("t", "dt_next", "n_steps", "n_clamped", "n_active", "status"):
        assert ia[k] == ib[k], k


# one block, a block and a ragged one, whole blocks; the last sizes fill most of
# the resident grid (FP64 about 24,000 cells, FP32 about 116,000)
CASES = [("canal", 3, 1), ("canal", 17, 1), ("canal", 16, 4), ("canal", 65, 3), ("dam4k", 0, 0),
         ("river", 90, 13), ("river_wet", 60, 12), ("river", 300, 37)]


def _make(kind, nx, ny):
    if kind == "canal":
        return mg.canal(nx, ny, float(nx), float(ny), 0.2, seed=3, hL=2.0, hR=0.0, x_dam=nx / 2.0, manning=0.03)
    if kind == "dam4k":
        return mg.dam_break_4k()
    return mg.river(nx, ny, seed=4, n_bumps=20, fully_wet=kind == "river_wet")


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
@pytest.mark.parametrize("kind,nx,ny", CASES)
def test_loop_matches_single_launches_bitwise(kind, nx, ny, precision):
    mi = _make(kind, nx, ny)
    flux = capi.SWE_FLUX_HLL if (nx, ny) == (60, 12) else capi.SWE_FLUX_HLLC
    loop, single = _mesh(mi, precision, flux=flux), _mesh(mi, precision, flux=flux, graph_steps=-1)
    for steps in (4, 3, 50, 1, 61):   # the loop starts from every step index modulo 6
        assert loop.step(steps) == single.step(steps)
        _equal(loop, single)


def test_loop_takes_large_fp32_meshes_and_leaves_larger_ones():
    for nx, ny in ((500, 110), (700, 110)):   # 110,000 cells: the loop; 154,000: one launch a step
        mi = mg.river(nx, ny, seed=2, n_bumps=10)
        loop, single = _mesh(mi, capi.SWE_FP32), _mesh(mi, capi.SWE_FP32, graph_steps=-1)
        assert loop.step(40) == single.step(40)
        _equal(loop, single)


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
def test_loop_without_water_reports_it_and_keeps_the_state(precision):
    mi = mg.canal(20, 4, 20.0, 4.0, 0.2, seed=1, hL=0.0, hR=0.0, x_dam=10.0, manning=0.0)
    m = _mesh(mi, precision)
    with pytest.raises(capi.SWEError) as e:
        m.step(10)
    assert e.value.code == capi.SWE_EDRY
    assert all(np.array_equal(x, np.zeros_like(x)) for x in m.get_state())


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
def test_steps_under_stream_capture_are_single_launches(precision):
    # a mesh's first steps, captured by the caller: no cooperative launch, no
    # allocation, and the replayed graph gives the same states
    mi = mg.river(60, 12, seed=4, n_bumps=20)
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    captured, single = _mesh(mi, precision), _mesh(mi, precision, graph_steps=-1)
    captured.set_stream(stream)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        captured.step(6, sync=False)
    graph.replay()
    torch.cuda.synchronize()
    captured.set_stream(None)
    assert captured.info()["t"] == single.step(6)
    _equal(captured, single)


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
def test_a_wait_that_runs_out_is_reported_until_a_new_state(precision):
    # no polls: every block gives up at the first meeting and the kernel returns
    mi = mg.dam_break_4k()
    m, single = _mesh(mi, precision), _mesh(mi, precision, graph_steps=-1)
    m.debug_loop(max_polls=0)
    calls = [lambda: m.step(10), lambda: m.step(10), lambda: m.step(1), lambda: m.step_dt([1e-3, 1e-3]),
             lambda: m.run_to_steady(1e-9, check_every=5, max_steps=10), m.synchronize, lambda: capi.Ensemble([m])]
    if precision == capi.SWE_FP64:
        calls.append(lambda: m.adjoint(5, [1], [1.0]))
    for call in calls:
        with pytest.raises(capi.SWEError) as e:
            call()
        assert e.value.code == capi.SWE_ETIMEOUT
    assert m.info()["status"] == capi.SWE_ETIMEOUT
    m.debug_loop(max_polls=1 << 22)
    with pytest.raises(capi.SWEError) as e:      # no loop starts on what the other left
        m.step(10)
    assert e.value.code == capi.SWE_ETIMEOUT
    m.set_state(mi.h.astype(m.dtype), mi.hu.astype(m.dtype), mi.hv.astype(m.dtype))
    done = m.debug_loop()
    assert m.step(50) == single.step(50) and m.debug_loop() == done + 50
    _equal(m, single)


def test_the_loop_runs_where_it_should():
    mi = mg.river(90, 13, seed=4, n_bumps=20)
    for kw, steps in ((dict(), 50), (dict(graph_steps=48), 0), (dict(graph_steps=-1), 0), (dict(block_size=128), 0),
                      (dict(activity=1), 0), (dict(debug_checks=1), 0)):
        m = _mesh(mi, capi.SWE_FP32, **kw)
        m.step(50)
        m.step(3)
        assert m.debug_loop() == steps, kw


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
def test_a_refused_cooperative_launch_leaves_the_mesh_on_single_launches(precision):
    # more blocks than the device holds at once: the runtime refuses the launch
    mi = mg.river(700, 110, seed=2, n_bumps=10)
    m, single = _mesh(mi, precision), _mesh(mi, precision, graph_steps=-1)
    m.debug_loop(max_cells=1 << 20)
    for steps in (7, 60):
        assert m.step(steps) == single.step(steps)
        _equal(m, single)
    assert m.debug_loop() == 0


def test_long_calls_of_larger_fp32_meshes_replay_graphs():
    # 110,000 cells, past four blocks an SM: calls of a graph (48 steps) and more
    # replay it, shorter ones take the loop; 70,000 cells: the loop for both
    for nx, expect in ((500, 20 + 20), (318, 20 + 100 + 20)):
        mi = mg.river(nx, 110, seed=2, n_bumps=10)
        m, single = _mesh(mi, capi.SWE_FP32), _mesh(mi, capi.SWE_FP32, graph_steps=-1)
        for steps in (20, 100, 20):
            assert m.step(steps) == single.step(steps)
        assert m.debug_loop() == expect
        _equal(m, single)


@pytest.mark.parametrize("precision,nx,ny", [(capi.SWE_FP64, 60, 12), (capi.SWE_FP32, 60, 12), (capi.SWE_FP64, 400, 29),
                                             (capi.SWE_FP32, 500, 110)])
def test_the_autotuner_chooses_between_the_loop_and_its_shape(precision, nx, ny):
    mi = mg.river(nx, ny, seed=4, n_bumps=20)
    m, single = _mesh(mi, precision), _mesh(mi, precision, graph_steps=-1)
    shaped = _mesh(mi, precision, graph_steps=48)          # the tuned shape runs every step here
    for x in (m, single, shaped):
        x.step(37)
    done = m.debug_loop()
    for x in (m, shaped):
        x.autotune(trial_steps=2)
        _equal(x, single)                                  # the trials leave nothing behind
    assert m.debug_loop() == done and shaped.debug_loop() == 0
    for steps in (20, 101, 48, 5):
        ref = single.step(steps)
        for x in (m, shaped):
            before = x.debug_loop()
            assert x.step(steps) == ref
            assert x.debug_loop() - before in (0, steps)   # a call runs in one way
            _equal(x, single)
    assert shaped.debug_loop() == 0
    # on the smallest meshes the loop is the faster by a third and more
    if nx == 60:
        assert m.debug_loop() == done + 20 + 101 + 48 + 5


def test_no_loop_on_larger_meshes_nor_under_capture():
    large = _mesh(mg.river(700, 110, seed=2, n_bumps=10), capi.SWE_FP32)   # 154,000 cells
    large.step(20)
    assert large.debug_loop() == 0
    m = _mesh(mg.river(60, 12, seed=4, n_bumps=20), capi.SWE_FP64)
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    m.set_stream(stream)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        m.step(6, sync=False)
    assert m.debug_loop() == 0
    graph.replay()
    torch.cuda.synchronize()
    assert m.info()["status"] == 0
