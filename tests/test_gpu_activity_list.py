"""The two kernels of an FP32 mesh's activity steps -- through all cells, over a
list of the active ones -- against the kernel without activity bytes, bit for
bit, and the choice between them."""
import numpy as np
import pytest

from paper_2010_14416_gb300 import build as libbuild
from paper_2010_14416_gb300 import capi
from paper_2010_14416_gb300 import meshgen as mg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LIST, ALL = 0, 1 << 40


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    libbuild.build()
    return capi.load()


def _mesh(mi, **kw):
    m = capi.Mesh(mi.nodes, mi.tris, mi.z, mi.manning, precision=capi.SWE_FP32, **kw)
    for pairs, kind, value in mi.bcs:
        m.set_bc(pairs, kind, value)
    m.set_state(*(x.astype(np.float32) for x in (mi.h, mi.hu, mi.hv)))
    return m


def _equal(a, b, tag):
    assert all(np.array_equal(x, y) for x, y in zip(a.get_state(), b.get_state())), tag
    ia, ib = a.info(), b.info()
    for k in ("t", "dt_next", "n_active", "n_clamped", "status"):
        assert ia[k] == ib[k], (tag, k)


# every compiled (block_size, min_blocks, geometry_early, stages)
SHAPES = [(128, 8, 0, 3), (256, 4, 0, 3), (512, 2, 0, 3), (128, 8, 1, 3), (256, 4, 1, 3), (128, 8, 1, 4), (128, 8, 1, 5),
          (256, 4, 1, 4), (128, 8, 0, 4)]


@pytest.mark.parametrize("shape", SHAPES)
def test_both_activity_kernels_match_the_plain_one(shape):
    block, minb, geo, stages = shape
    for mi in (mg.river(101, 21, seed=8), mg.canal(401, 20, Lx=200.0, Ly=10.0, hR=0.0, seed=3, manning=0.03)):
        ref = _mesh(mi, graph_steps=-1)
        ref.step(131)
        for cells in (LIST, ALL):
            for grid in (0, 3):
                m = _mesh(mi, activity=1, block_size=block, min_blocks=minb, geometry_early=geo, stages=stages, grid=grid)
                m.debug_activity(list_cells=cells)
                m.step(7)
                assert m.debug_activity() == (cells == LIST)
                m.step(124)
                _equal(m, ref, (cells, grid))
                m.close()
        ref.close()


def test_changing_between_the_kernels_while_water_enters_dry_spans():
    # the list passes over spans of 4,096 cells whose flags are 0; in between, the
    # other kernel carries the front across several of them, and two of the
    # bytes' three buffers and both state buffers take turns at every length
    mi = mg.canal(600, 80, 600.0, 80.0, 0.2, seed=5, hL=6.0, hR=0.0, x_dam=30.0, manning=0.0)
    m, ref = _mesh(mi, activity=1), _mesh(mi, graph_steps=-1)
    for cells, steps in ((LIST, 13), (ALL, 2000), (LIST, 60), (ALL, 1), (LIST, 2), (ALL, 3), (LIST, 50)):
        m.debug_activity(list_cells=cells)
        assert m.step(steps) == ref.step(steps)
        assert m.debug_activity() == (cells == LIST)
        _equal(m, ref, (cells, steps))


def test_activity_steps_without_water_carry_over():
    mi = mg.canal(60, 20, 60.0, 20.0, 0.2, seed=1, hL=0.0, hR=0.0, x_dam=10.0, manning=0.0)
    for cells in (LIST, ALL):
        m = _mesh(mi, activity=1)
        m.debug_activity(list_cells=cells)
        with pytest.raises(capi.SWEError) as e:
            m.step(5)
        assert e.value.code == capi.SWE_EDRY
        assert all(np.array_equal(x, np.zeros_like(x)) for x in m.get_state())


def test_the_choice_follows_size_and_share_of_wet_cells():
    dry = mg.river(3000, 201, seed=2, n_bumps=10)          # 1.2M cells, 6 % wet
    m = _mesh(dry, activity=1)
    m.step(4)
    assert m.debug_activity()
    flood = np.maximum(dry.h, 0.5).astype(np.float32)      # a flooded state, then the first one again
    m.set_state(flood, 0 * flood, 0 * flood)
    m.step(4)
    assert not m.debug_activity()
    m.set_state(*(x.astype(np.float32) for x in (dry.h, dry.hu, dry.hv)))
    m.step(4)
    assert m.debug_activity()
    small = _mesh(mg.river(101, 21, seed=8), activity=1)
    small.step(4)
    assert not small.debug_activity()
    # an activity shape that the autotuner keeps stays on the list
    if small.autotune(trial_steps=2)["activity"]:
        small.step(4)
        assert small.debug_activity()
