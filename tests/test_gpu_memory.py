"""What a mesh reports as the device memory that it holds (swe_info.device_bytes)
and what it keeps between calls."""
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


def _mesh(mi, precision=capi.SWE_FP64, **kw):
    m = capi.Mesh(mi.nodes, mi.tris, mi.z, mi.manning, precision=precision, **kw)
    for pairs, kind, value in mi.bcs:
        m.set_bc(pairs, kind, value)
    m.set_state(*(x.astype(m.dtype) for x in (mi.h, mi.hu, mi.hv)))
    return m


def _held(m):
    return m.info()["device_bytes"]


def test_kept_buffers_are_reported():
    mi = mg.river(90, 13, seed=4, n_bumps=20)
    n = mi.n_cells
    m = _mesh(mi)
    base = _held(m)
    interior = (3 * n - sum(len(p) for p, _, _ in mi.bcs)) // 2
    m.step(10)                                        # the FP64 loop's edges: 96 slots of 24 B a block, 4 B a cell
    loop = -(-n // 32) * 96 * 24 + 4 * n + 4
    assert m.debug_loop() == 10 and _held(m) - base == loop
    m.diagnostics()
    diag = _held(m) - base - loop
    assert diag >= 1024 * 5 * 8                       # the blocks' partials and the boundary edges'
    m.adjoint(30, [5], [1.0])
    kept = _held(m) - base - loop - diag
    states, terms = 30 * n * 32, 30 * interior * 40   # of the one segment
    assert states < kept < 1.2 * (states + terms) + 12 * n * 32
    m.set_bc(mi.bcs[1][0], mg.BC_WALL)                # the boundary edges' groups change, not their number
    m.diagnostics()
    assert _held(m) - base == loop + diag + kept
    m.close()


def test_meshes_together_keep_a_bounded_adjoint_workspace():
    # six meshes whose workspaces take 48 steps of 32 B a cell and 40 B an edge,
    # 1.04 GiB, and some more each: the process keeps 6 GiB
    # at most, gives back the others after each call, and a mesh that is closed
    # makes room; the results do not depend on it
    mi = mg.river(1000, 126, seed=4, n_bumps=20)
    before = torch.cuda.mem_get_info()[0]
    meshes, kept, first = [], [], None
    for k in range(6):
        m = _mesh(mi)
        base = _held(m)
        out = m.adjoint(48, [5, 700], [1.0, 2.0])
        kept.append(_held(m) - base)
        first = first or out
        assert out[0] == first[0] and all(np.array_equal(a, b) for a, b in zip(out[1:], first[1:]))
        meshes.append(m)
    assert kept[0] > 48 * 90 * mi.n_cells and sum(kept) <= 6 * 2**30 and kept[-1] == 0
    meshes[0].close()
    base = _held(meshes[-1])
    meshes[-1].adjoint(48, [5, 700], [1.0, 2.0])
    assert _held(meshes[-1]) - base == kept[0]
    for m in meshes:
        m.close()
    assert torch.cuda.mem_get_info()[0] > before - 2**28
