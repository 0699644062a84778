"""Batched ensemble (uncertainty propagation, Section 6.4.3's sampled runs):
members of uneven sizes advanced together must receive exactly the updates
the plain solver gives each of them alone, bit for bit, with their own CFL
steps."""
import numpy as np
import pytest

import oracle
from oracle import rel_err
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


def _members(n=8, seed=3):
    return mg.ensemble_members(n, seed=seed, lo=1500, hi=30000)


def _mesh(mi, precision, **kw):
    m = capi.Mesh(mi.nodes, mi.tris, mi.z, mi.manning, precision=precision, **kw)
    for pairs, kind, value in mi.bcs:
        m.set_bc(pairs, kind, value)
    dt = m.dtype
    m.set_state(mi.h.astype(dt), mi.hu.astype(dt), mi.hv.astype(dt))
    return m


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
def test_ensemble_matches_plain_solver_bitwise(precision):
    mis = _members()
    assert len({mi.n_cells % 256 for mi in mis}) > 1          # uneven, ragged sizes
    rng = np.random.default_rng(1)
    cfl = rng.uniform(0.5, 0.9, len(mis))
    meshes = [_mesh(mi, precision) for mi in mis]
    ens = capi.Ensemble(meshes)
    t_a = ens.step(100, cfl)
    t_b = ens.step(101, cfl)                                   # second call starts mid-phase
    for k, (mi, m) in enumerate(zip(mis, meshes)):
        t_plain = m.step(201, cfl[k])
        assert t_b[k] == t_plain and t_a[k] < t_b[k]
        got = ens.get_state(k)
        ref = m.get_state()
        assert all(np.array_equal(a, b) for a, b in zip(got, ref)), f"member {k}"
        assert ens.info(k)["status"] == 0
    ens.close()
    for m in meshes:
        m.close()


def test_ensemble_member_against_oracle_fp64():
    mis = _members(4, seed=5)
    meshes = [_mesh(mi, capi.SWE_FP64) for mi in mis]
    ens = capi.Ensemble(meshes)
    t = ens.step(300)
    for k in (0, 3):
        mi = mis[k]
        M = oracle.Mesh(mi.nodes, mi.tris, mi.z, mi.manning)
        for pairs, kind, value in mi.bcs:
            M.set_bc(pairs, kind, value)
        oh, ohu, ohv, ot, _ = M.run(mi.h, mi.hu, mi.hv, 300, 0.9)
        assert t[k] == pytest.approx(ot, rel=1e-12)
        for a, b in zip(ens.get_state(k), (oh, ohu, ohv)):
            assert rel_err(a, b) <= 1e-10
    ens.close()


def test_ensemble_device_output_and_errors():
    mis = _members(3, seed=7)
    meshes = [_mesh(mi, capi.SWE_FP64) for mi in mis]
    ens = capi.Ensemble(meshes)
    ens.step(12)
    out = [torch.empty(mis[1].n_cells, dtype=torch.float64, device="cuda") for _ in range(3)]
    ens.get_state(1, out)
    torch.cuda.synchronize()
    host = ens.get_state(1)
    assert all(np.array_equal(a.cpu().numpy(), b) for a, b in zip(out, host))
    ens.close()
    # a member without a state, or of another precision, is refused
    bare = capi.Mesh(mis[0].nodes, mis[0].tris, mis[0].z, mis[0].manning)
    with pytest.raises(capi.SWEError) as e:
        capi.Ensemble([meshes[0], bare])
    assert e.value.code == capi.SWE_EINVAL
    f32 = _mesh(mis[0], capi.SWE_FP32)
    with pytest.raises(capi.SWEError) as e:
        capi.Ensemble([meshes[0], f32])
    assert e.value.code == capi.SWE_EINVAL


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
def test_ensemble_launch_shapes_are_bitwise_neutral(precision):
    # every batched kernel shape -- tile size, staging, geometry placement,
    # activity bytes, chunk, grid and (FP32) the split step over cell pairs and
    # the per-warp queues -- gives each member the plain solver's updates bit
    # for bit, also when the shape changes between calls
    mis = _members(6, seed=13)
    meshes = [_mesh(mi, precision) for mi in mis]
    ens = capi.Ensemble(meshes)
    f32 = precision == capi.SWE_FP32
    shapes = [dict(block_size=128, min_blocks=8 if f32 else 1, activity=1, chunk=4),
              dict(block_size=256, min_blocks=4 if f32 else 1, activity=1, chunk=16, grid=37),
              dict(block_size=256, min_blocks=4 if f32 else 1, stages=3 if f32 else 1, chunk=8),
              dict(block_size=128, min_blocks=8 if f32 else 1, geometry_early=1 if f32 else 0, activity=1,
                   chunk=64, grid=5)]
    # chunks taken dynamically from a per-step counter, switched to and from
    shapes += [dict(block_size=128, min_blocks=8 if f32 else 1, dynamic=1, chunk=1),
               dict(block_size=256, min_blocks=4 if f32 else 1, stages=3 if f32 else 1, chunk=4),
               dict(block_size=256, min_blocks=4 if f32 else 1, dynamic=1, chunk=8, grid=17)]
    # activity bytes with dynamically taken chunks (at least 4 tiles)
    shapes += [dict(block_size=128, min_blocks=8 if f32 else 1, activity=1, dynamic=1, chunk=4),
               dict(block_size=256, min_blocks=4 if f32 else 1, activity=1, dynamic=1, chunk=32, grid=23),
               dict(block_size=128, min_blocks=8 if f32 else 1, geometry_early=1 if f32 else 0, activity=1,
                    dynamic=1, chunk=8, grid=3)]
    if not f32:   # the edge pass of FP64 ensembles
        shapes += [dict(block_size=256, min_blocks=1, edge_pass=1, chunk=8),
                   dict(block_size=128, min_blocks=1, edge_pass=1, chunk=4, grid=11)]
    else:   # split steps: the members wet at creation on the cell-pair kernel, the rest on the given one
        shapes += [dict(block_size=128, min_blocks=8, activity=1, dynamic=1, chunk=4, cell_pairs=1),
                   dict(block_size=256, min_blocks=4, activity=1, chunk=16, grid=37, cell_pairs=1),
                   dict(block_size=128, min_blocks=8, dynamic=1, chunk=1, cell_pairs=1),
                   dict(block_size=256, min_blocks=4, stages=3, chunk=8, cell_pairs=1),
                   dict(block_size=128, min_blocks=8, geometry_early=1, activity=1, chunk=64, grid=5, cell_pairs=1)]
        # per-warp queues of the cells that run the flux path, alone and in split steps
        shapes += [dict(block_size=128, min_blocks=7, geometry_early=1, activity=1, chunk=8, queue=1),
                   dict(block_size=128, min_blocks=7, activity=1, dynamic=1, chunk=4, grid=9, queue=1, cell_pairs=1),
                   dict(block_size=128, min_blocks=6, geometry_early=1, activity=1, dynamic=1, chunk=16, queue=1),
                   dict(block_size=128, min_blocks=7, geometry_early=1, activity=1, chunk=4, grid=3, queue=1,
                        cell_pairs=1)]
    steps = 0
    for k, sh in enumerate(shapes):
        ens.set_shape(**sh)
        ens.step(37 + k)
        steps += 37 + k
    t_ens = ens.step(0)
    for k, m in enumerate(meshes):
        assert m.step(steps) == t_ens[k]
        assert all(np.array_equal(a, b) for a, b in zip(ens.get_state(k), m.get_state())), f"member {k}"
    assert ens.info(0)["n_active"] == sum(m.info()["n_active"] for m in meshes)
    with pytest.raises(capi.SWEError):
        ens.set_shape(block_size=512, min_blocks=2, activity=1)
    with pytest.raises(capi.SWEError):
        ens.set_shape(block_size=256, min_blocks=4 if f32 else 1, activity=1, edge_pass=1)
    with pytest.raises(capi.SWEError):   # dynamic activity chunks hold at least 4 tiles
        ens.set_shape(block_size=128, min_blocks=8 if f32 else 1, activity=1, dynamic=1, chunk=2)
    with pytest.raises(capi.SWEError):
        ens.set_shape(block_size=256, min_blocks=4 if f32 else 1, dynamic=1, edge_pass=1)
    if not f32:   # the split step and the queues are FP32 only
        with pytest.raises(capi.SWEError):
            ens.set_shape(block_size=128, min_blocks=1, activity=1, chunk=4, cell_pairs=1)
        with pytest.raises(capi.SWEError):
            ens.set_shape(block_size=128, min_blocks=1, activity=1, chunk=4, queue=1)
    else:   # queues need the activity kernel
        with pytest.raises(capi.SWEError):
            ens.set_shape(block_size=128, min_blocks=7, dynamic=1, chunk=4, queue=1)
    ens.close()
    for m in meshes:
        m.close()


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
def test_ensemble_debug_checks_change_nothing(precision):
    # members created with debug checks: the batched kernels check every
    # index and boundary group before use; a valid ensemble steps exactly as
    # without them, with status 0
    mis = _members(4, seed=9)
    ref_meshes = [_mesh(mi, precision) for mi in mis]
    ref = capi.Ensemble(ref_meshes)
    t_ref = ref.step(120)
    dbg_meshes = [_mesh(mi, precision, debug_checks=1) for mi in mis]
    dbg = capi.Ensemble(dbg_meshes)
    shapes = [None, dict(block_size=128, min_blocks=8 if precision == capi.SWE_FP32 else 1, activity=1, chunk=4)]
    if precision == capi.SWE_FP64:
        shapes.append(dict(block_size=256, min_blocks=1, edge_pass=1, chunk=4))
    else:
        shapes.append(dict(block_size=128, min_blocks=8, activity=1, dynamic=1, chunk=4, cell_pairs=1))
        shapes.append(dict(block_size=128, min_blocks=7, geometry_early=1, activity=1, chunk=4, queue=1))
    for shape in shapes:
        for k, m in enumerate(dbg_meshes):
            m.set_state(*(a.astype(m.dtype) for a in (mis[k].h, mis[k].hu, mis[k].hv)))
        dbg.close()
        dbg = capi.Ensemble(dbg_meshes)
        if shape:
            dbg.set_shape(**shape)
        t = dbg.step(120)
        assert np.array_equal(t, t_ref), shape
        for k in range(len(mis)):
            assert dbg.info(k)["status"] == 0
            assert all(np.array_equal(a, b) for a, b in zip(dbg.get_state(k), ref.get_state(k))), (shape, k)
    for e in (ref, dbg):
        e.close()
    for m in ref_meshes + dbg_meshes:
        m.close()


@pytest.mark.parametrize("pairs", [0, 1])
def test_list_mode_resumes_where_other_activity_steps_moved_the_water(pairs):
    # list steps (queue=1) pass over spans of 4,096 cells that their flags call
    # dry; the steps of another activity kernel in between carry the front
    # across several such spans, and the list steps that follow must see it
    dry = mg.canal(600, 80, 600.0, 80.0, 0.2, seed=5, hL=6.0, hR=0.0, x_dam=30.0, manning=0.0)
    wet = mg.canal(300, 12, 300.0, 12.0, 0.2, seed=6, hL=3.0, hR=1.0, x_dam=150.0, manning=0.02)
    meshes = [_mesh(mi, capi.SWE_FP32) for mi in (dry, wet)]
    ens = capi.Ensemble(meshes)
    listed = dict(block_size=128, min_blocks=7, geometry_early=1, activity=1, chunk=8, queue=1, cell_pairs=pairs)
    other = dict(block_size=128, min_blocks=8, geometry_early=1, activity=1, chunk=8, cell_pairs=pairs)
    for shape, steps in ((listed, 12), (other, 2000), (listed, 60), (other, 1), (listed, 7)):
        ens.set_shape(**shape)
        t = ens.step(steps)
    cell_x = dry.nodes[dry.tris].mean(1)[:, 0]
    for k, m in enumerate(meshes):
        m.step(12)
        before = m.get_state()[0] > 1e-6
        assert m.step(2000 + 60 + 1 + 7) == t[k]
        ref = m.get_state()
        if k == 0:   # a span holds about 45 x 45 quads: the front has crossed three of them
            assert cell_x[ref[0] > 1e-6].max() - cell_x[before].max() > 150.0
        assert all(np.array_equal(a, b) for a, b in zip(ens.get_state(k), ref)), f"member {k}"
    ens.close()
    for m in meshes:
        m.close()


def test_list_mode_steps_a_member_beside_one_that_has_no_water():
    # a member without water keeps its state and reports it, the others step on;
    # water that later enters spans passed over for many steps is updated too
    empty = mg.canal(400, 12, 400.0, 12.0, 0.2, seed=7, hL=0.0, hR=0.0, x_dam=200.0, manning=0.02)
    dry = mg.canal(600, 40, 600.0, 40.0, 0.2, seed=8, hL=5.0, hR=0.0, x_dam=50.0, manning=0.0)
    meshes = [_mesh(mi, capi.SWE_FP32) for mi in (dry, empty, dry)]
    ens = capi.Ensemble(meshes)
    ens.set_shape(block_size=128, min_blocks=7, geometry_early=1, activity=1, chunk=8, queue=1)
    ens.step(700, sync=False)
    for k in (0, 2):
        meshes[k].step(700)
        assert all(np.array_equal(a, b) for a, b in zip(ens.get_state(k), meshes[k].get_state())), f"member {k}"
        assert ens.info(k)["status"] == 0 and ens.info(k)["t"] == meshes[k].info()["t"]
    assert ens.info(1)["status"] == capi.SWE_EDRY
    assert all(np.array_equal(a, np.zeros_like(a)) for a in ens.get_state(1))
    ens.close()
    for m in meshes:
        m.close()
