"""GPU parity: the CUDA path (through the C ABI) against the FP64 CPU oracle.

Tolerances: FP64 GPU vs oracle <= 1e-10 max relative error per field
(max_i |f_i - f_i^ref| / max_i |f_i^ref|) after 1000 steps; FP32 GPU vs FP64
<= 1e-4 with the same norm.  Integer results (clamp counts, status codes)
are exact."""
import math

import numpy as np
import pytest

import oracle
from oracle import rel_err
from paper_2010_14416_gb300 import build as libbuild
from paper_2010_14416_gb300 import capi
from paper_2010_14416_gb300 import meshgen as mg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FP64_TOL = 1e-10
FP32_TOL = 1e-4
# element-wise relative error on wet cells, with floors of 1 mm depth and
# 1e-3 m^2/s discharge per unit width (elem_rel_err), per field (h, hu, hv),
# measured (FP64 against the oracle) at 7e-13 / 1.2e-10 / 1.2e-10 on the 13M
# river after 1000 steps, 1e-13 / 4.5e-9 / 2.4e-9 on the 1M dry-bed canal
# after 2000 steps (at the wetting front) and 1.5e-15 / 2.1e-10 / 2.7e-10 on
# the 1M wet river after 1000 steps; FP32 on the 13M river 1.1e-4 / 5.1e-2 /
# 4.9e-2 (largest in slow shallow water near wet/dry fronts, where the
# momentum is far below the field's maximum)
ELEM_TOL_FP64 = (1e-11, 1e-8, 1e-8)
ELEM_TOL_FP32 = (1e-3, 0.2, 0.2)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    libbuild.build()
    return capi.load()


def elem_rel_err(state, ref, h_dry=1e-6, floors=(1e-3, 1e-3, 1e-3)):
    """Element-wise relative error per field (h, hu, hv) over the cells that
    are wet in either state: max_i |a_i - r_i| / max(|r_i|, floor).  The
    normwise figure (rel_err) divides by the field's largest value instead,
    which hides errors in shallow or slow cells."""
    wet = (np.asarray(ref[0]) > h_dry) | (np.asarray(state[0]) > h_dry)
    out = []
    for a, r, fl in zip(state, ref, floors):
        a = np.asarray(a, np.float64)[wet]
        r = np.asarray(r, np.float64)[wet]
        out.append(float((np.abs(a - r) / np.maximum(np.abs(r), fl)).max()) if r.size else 0.0)
    return out


def _gpu_mesh(mi, precision=capi.SWE_FP64, **kw):
    m = capi.Mesh(mi.nodes, mi.tris, mi.z, mi.manning, precision=precision, **kw)
    for pairs, kind, value in mi.bcs:
        m.set_bc(pairs, kind, value)
    return m


def _orc_mesh(mi):
    M = oracle.Mesh(mi.nodes, mi.tris, mi.z, mi.manning)
    for pairs, kind, value in mi.bcs:
        M.set_bc(pairs, kind, value)
    return M


def _gpu_run(mi, nsteps, precision=capi.SWE_FP64, cfl=0.9, state=None, **kw):
    m = _gpu_mesh(mi, precision, **kw)
    dt = np.float32 if precision == capi.SWE_FP32 else np.float64
    h, hu, hv = state if state is not None else (mi.h, mi.hu, mi.hv)
    m.set_state(h.astype(dt), hu.astype(dt), hv.astype(dt))
    t = m.step(nsteps, cfl)
    out = m.get_state()
    info = m.info()
    m.close()
    return [o.astype(np.float64) for o in out], t, info


# ---------------------------------------------------------------------------
# Riemann flux (Eq 17-26) on random normal-frame states
# ---------------------------------------------------------------------------

def _random_states(n, seed):
    rng = np.random.default_rng(seed)
    hL = rng.uniform(0, 10, n)
    hR = rng.uniform(0, 10, n)
    hL[rng.random(n) < 0.1] = 0.0
    hR[rng.random(n) < 0.1] = 0.0
    hL[rng.random(n) < 0.05] = 5e-7       # below h_dry
    unL, unR = rng.uniform(-15, 15, n), rng.uniform(-15, 15, n)
    utL, utR = rng.uniform(-3, 3, n), rng.uniform(-3, 3, n)
    same = rng.random(n) < 0.05          # consistency cases
    hR[same], unR[same], utR[same] = hL[same], unL[same], utL[same]
    hL[0], hR[0], unL[0], unR[0] = 10.0, 1.0, 0.0, 0.0  # the dam-break state
    return hL, unL, utL, hR, unR, utR


TIE_MARGIN = 1e-4   # relative distance of a branch decision from its threshold


def _tie_margin(hL, unL, utL, hR, unR, utR, contact, g=9.81, h_dry=1e-6):
    """Smallest relative distance, over the decisions of the Riemann solver
    whose two outcomes give different fluxes (the dry tests of Eq 26, the
    choice between the star-depth estimates of Eq 22 and Eq 23 and, for HLLC,
    the sign of S* in Eq 24), between the decided quantity and its threshold,
    from the FP64 oracle's intermediate values.  The shock tests of Eq 20,
    the vacuum clamp and the signs of S_L and S_R switch between expressions
    that agree at the threshold, so FP32 rounding there cannot produce an
    outlier and they are not counted."""
    m = [abs(hL - h_dry) / h_dry, abs(hR - h_dry) / h_dry]
    if hL > h_dry and hR > h_dry and (hL != hR or unL != unR):
        _, h0 = oracle.hstar(hL, unL, hR, unR)
        hmin = min(hL, hR)
        m.append(abs(h0 - hmin) / max(abs(h0), hmin))
    if contact and (hL > h_dry or hR > h_dry):
        _, S = oracle.hllc(hL, unL, utL, hR, unR, utR)
        sc = max(abs(S[0]), abs(S[1]), abs(unL), abs(unR), math.sqrt(g * max(hL, hR)))
        m.append(abs(S[2]) / sc)
    return min(m)


def test_riemann_flux_hand_worked_asymmetric_states():
    # Eq 19-25 worked by hand (tests/golden/sstar_asym.txt) through the
    # kernel's batched entry point, FP64 and FP32
    from tests.golden_cases import read_cases
    cases = read_cases("sstar_asym.txt")
    keys = ("hL", "unL", "utL", "hR", "unR", "utR")
    for precision, rel in ((capi.SWE_FP64, 1e-12), (capi.SWE_FP32, 2e-6)):
        tdt = torch.float64 if precision == capi.SWE_FP64 else torch.float32
        names = sorted(cases)
        dev = [torch.tensor([cases[c][k] for c in names], dtype=tdt, device="cuda") for k in keys]
        G = [torch.empty(len(names), dtype=tdt, device="cuda") for _ in range(3)]
        S = torch.empty((len(names), 3), dtype=tdt, device="cuda")
        capi.riemann_flux(precision, *dev, *G, S)
        torch.cuda.synchronize()
        for j, c in enumerate(names):
            gc = cases[c]
            got_s = S[j].double().cpu().numpy()
            for k, key in enumerate(("SL", "SR", "Sstar")):
                assert got_s[k] == pytest.approx(gc[key], rel=rel), (c, key, precision)
            for k in range(3):
                assert float(G[k][j]) == pytest.approx(gc[f"G{k + 1}"], rel=rel), (c, k, precision)


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
def test_riemann_flux_matches_oracle(precision):
    n = 4000
    st = _random_states(n, 7)
    tdt = torch.float64 if precision == capi.SWE_FP64 else torch.float32
    dev = [torch.tensor(a, dtype=tdt, device="cuda") for a in st]
    G = [torch.empty(n, dtype=tdt, device="cuda") for _ in range(3)]
    S = torch.empty((n, 3), dtype=tdt, device="cuda")
    capi.riemann_flux(precision, *dev, *G, S)
    torch.cuda.synchronize()
    got = np.stack([g.double().cpu().numpy() for g in G], axis=1)
    # the reference takes the inputs the kernel received (rounded to FP32 on the FP32 path)
    st_in = [d.double().cpu().numpy() for d in dev]
    ref = np.zeros((n, 3))
    for i in range(n):
        ref[i], _ = oracle.hllc(*(float(a[i]) for a in st_in))
    scale = np.maximum(np.abs(ref).max(axis=1), 1.0)
    err = (np.abs(got - ref).max(axis=1) / scale)
    tol = 1e-13 if precision == capi.SWE_FP64 else 2e-5
    bad = np.where(err > tol)[0]
    assert len(bad) <= (0 if precision == capi.SWE_FP64 else n // 500), (err.max(), bad)
    # an FP32 result off by more than the tolerance must sit at a branch tie,
    # where FP32 rounding may legitimately take the other branch
    for i in bad:
        margin = _tie_margin(*(float(a[i]) for a in st_in), contact=True)
        assert margin <= TIE_MARGIN, (i, err[i], margin, [float(a[i]) for a in st_in])
    # the dam-break state of Section 6.3: h* = 3.9529... gives S_L = -sqrt(g h_L)
    s0 = S[0].double().cpu().numpy()
    assert s0[0] == pytest.approx(-math.sqrt(9.81 * 10.0), rel=1e-12 if precision == 0 else 1e-6)


# ---------------------------------------------------------------------------
# Whole-step parity on small meshes (several tiles plus a ragged tail)
# ---------------------------------------------------------------------------

def test_dam_break_4k_fp64_1000_steps_all_orderings_bitwise_equal():
    mi = mg.dam_break_4k()
    M = _orc_mesh(mi)
    oh, ohu, ohv, ot, oc = M.run(mi.h, mi.hu, mi.hv, 1000, 0.9)
    results = {}
    for r in (capi.SWE_REORDER_NONE, capi.SWE_REORDER_RCM, capi.SWE_REORDER_HILBERT):
        (gh, ghu, ghv), t, info = _gpu_run(mi, 1000, reorder=r)
        assert info["n_clamped"] == oc == 0
        assert t == pytest.approx(ot, rel=1e-12)
        assert rel_err(gh, oh) <= FP64_TOL
        assert rel_err(ghu, ohu) <= FP64_TOL
        assert rel_err(ghv, ohv) <= FP64_TOL
        results[r] = (gh, ghu, ghv, t)
    a = results[capi.SWE_REORDER_NONE]
    for r in (capi.SWE_REORDER_RCM, capi.SWE_REORDER_HILBERT):
        b = results[r]
        assert all(np.array_equal(x, y) for x, y in zip(a[:3], b[:3])), "ordering changed the result"
        assert a[3] == b[3]


def test_river_with_all_boundary_kinds_fp64():
    # partially dry reach: wet/dry fronts, inflow, stage, walls, friction,
    # bumps, shuffled numbering
    mi = mg.river(160, 32, seed=5, shuffle=True)
    M = _orc_mesh(mi)
    oh, ohu, ohv, ot, oc = M.run(mi.h, mi.hu, mi.hv, 1000, 0.9)
    (gh, ghu, ghv), t, info = _gpu_run(mi, 1000)
    assert t == pytest.approx(ot, rel=1e-12)
    assert info["n_clamped"] == oc
    for a, b in ((gh, oh), (ghu, ohu), (ghv, ohv)):
        assert rel_err(a, b) <= FP64_TOL


def test_transmissive_and_friction_fp64():
    mi = mg.canal(50, 8, 50.0, 8.0, 0.2, 6, side_bc=mg.BC_TRANSMISSIVE, hL=3.0, hR=1.0,
                  x_dam=25.0, manning=0.05)
    rng = np.random.default_rng(3)
    h0 = mi.h.copy()
    hu0 = rng.uniform(-1, 1, mi.n_cells) * h0
    hv0 = rng.uniform(-1, 1, mi.n_cells) * h0
    M = _orc_mesh(mi)
    oh, ohu, ohv, ot, oc = M.run(h0, hu0, hv0, 1000, 0.9)
    (gh, ghu, ghv), t, info = _gpu_run(mi, 1000, state=(h0, hu0, hv0))
    assert t == pytest.approx(ot, rel=1e-12)
    for a, b in ((gh, oh), (ghu, ohu), (ghv, ohv)):
        assert rel_err(a, b) <= FP64_TOL


@pytest.mark.parametrize("maker", [mg.dam_break_4k, lambda: mg.river(160, 32, seed=5)])
def test_fp32_against_fp64(maker):
    mi = maker()
    M = _orc_mesh(mi)
    oh, ohu, ohv, ot, oc = M.run(mi.h, mi.hu, mi.hv, 1000, 0.9)
    (gh, ghu, ghv), t, info = _gpu_run(mi, 1000, precision=capi.SWE_FP32)
    assert t == pytest.approx(ot, rel=1e-4)
    for a, b in ((gh, oh), (ghu, ohu), (ghv, ohv)):
        assert rel_err(a, b) <= FP32_TOL


def test_mass_conserved_and_lake_at_rest_on_gpu():
    mi = mg.dam_break_4k()
    area = oracle.Mesh(mi.nodes, mi.tris, mi.z, mi.manning).geometry()["area"]
    (gh, _, _), t, _ = _gpu_run(mi, 1000)
    m0 = (area * mi.h).sum()
    assert abs((area * gh).sum() - m0) / m0 < 1e-13
    lake = mg.river(120, 24, seed=2)
    eta0 = lake.meta["eta0"]
    lake.bcs = [(lake.bcs[1][0], mg.BC_STAGE, eta0)]
    h0 = np.maximum(eta0 - lake.z, 0.0)
    z0 = np.zeros_like(h0)
    (gh, ghu, ghv), t, _ = _gpu_run(lake, 1000, state=(h0, z0, z0))
    wet = h0 > 0
    assert np.abs(gh + lake.z - eta0)[wet].max() < 1e-12
    assert np.all(gh[~wet] == 0.0)
    assert np.abs(ghu).max() < 1e-10 and np.abs(ghv).max() < 1e-10


@pytest.mark.parametrize("precision,variants", [
    (capi.SWE_FP64, [(128, 1, 1, 0), (256, 1, 1, 0), (512, 1, 1, 0), (128, 1, 2, 0), (256, 1, 2, 0),
                     (128, 1, 1, 1), (256, 1, 1, 1)]),
    (capi.SWE_FP32, [(256, 4, 1, 0), (256, 4, 2, 0), (256, 4, 3, 0), (256, 4, 4, 0), (128, 8, 3, 0),
                     (128, 8, 4, 0), (512, 2, 1, 0), (256, 5, 1, 0), (256, 4, 1, 1), (256, 4, 3, 1),
                     (128, 8, 1, 1), (128, 8, 3, 1)]),
])
def test_kernel_variants_are_bitwise_identical(precision, variants):
    # launch shape, register cap, cp.async staging depth and the placement of
    # the geometry loads change nothing
    mi = mg.river(100, 20, seed=8)
    ref = None
    for b, mb, st, ge in variants:
        got, t, _ = _gpu_run(mi, 301, precision=precision, block_size=b, min_blocks=mb, stages=st,
                             geometry_early=ge)
        if ref is None:
            ref, tref = got, t
            continue
        assert t == tref, (b, mb, st, ge)
        assert all(np.array_equal(x, y) for x, y in zip(ref, got)), (b, mb, st, ge)


def _odd_canal():
    # a dam-break canal with its last triangle removed: an odd cell count, so
    # the last pair has one cell; walls all round
    mi = mg.canal(201, 10, Lx=100.0, Ly=5.0, hR=0.0, seed=5, manning=0.03)
    keep = mi.n_cells - 1
    mi.tris, mi.z, mi.manning = mi.tris[:keep], mi.z[:keep], mi.manning[:keep]
    mi.h, mi.hu, mi.hv = mi.h[:keep], mi.hu[:keep], mi.hv[:keep]
    mi.bcs = []
    return mi


@pytest.mark.parametrize("maker", ["river", "odd_canal"])
def test_cell_pair_kernel_is_bitwise_identical(maker):
    # the pair kernel hands each shared edge 0 from the first cell of a pair to
    # the second; states, times and the count of cells that ran the flux path
    # equal the one-cell kernel's for every shape, grid, flux, reorder and with
    # the debug checks, through wetting fronts, an inflow and a fixed stage
    mi = mg.river(101, 21, seed=8) if maker == "river" else _odd_canal()
    if maker == "odd_canal":
        assert mi.n_cells % 2 == 1
    f32 = capi.SWE_FP32
    for extra in (dict(), dict(flux=capi.SWE_FLUX_HLL), dict(reorder=capi.SWE_REORDER_RCM),
                  dict(reorder=capi.SWE_REORDER_NONE)):
        ref, tref, iref = _gpu_run(mi, 301, precision=f32, **extra)
        shapes = [dict(), dict(block_size=128, min_blocks=8, geometry_early=1), dict(block_size=128, min_blocks=8),
                  dict(block_size=256, min_blocks=4, geometry_early=1),
                  dict(block_size=256, min_blocks=4, grid=3),
                  dict(block_size=256, min_blocks=3, geometry_early=1, grid=100000, graph_steps=-1),
                  dict(block_size=256, min_blocks=4, geometry_early=1, debug_checks=1)]
        for kw in shapes:
            got, t, info = _gpu_run(mi, 301, precision=f32, cell_pairs=1, **kw, **extra)
            assert t == tref, (kw, extra)
            assert all(np.array_equal(x, y) for x, y in zip(ref, got)), (kw, extra)
            assert info["n_active"] == iref["n_active"], (kw, extra)
            assert info["status"] == 0


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
@pytest.mark.parametrize("maker", ["river", "dry_canal"])
def test_activity_mode_is_bitwise_neutral(precision, maker):
    # activity bytes replace the quiet-cell neighbour test: same states, times
    # and count of cells that ran the flux path, through wetting fronts, an
    # inflow and a fixed stage, on a cell count that is not a multiple of 32
    if maker == "river":
        mi = mg.river(101, 21, seed=8)
    else:
        mi = mg.canal(401, 20, Lx=200.0, Ly=10.0, hR=0.0, seed=3, manning=0.03)
    assert mi.n_cells % 32 != 0
    ref, tref, iref = _gpu_run(mi, 301, precision=precision)
    f32 = precision == capi.SWE_FP32
    shapes = [dict(), dict(block_size=128, min_blocks=8 if f32 else 1), dict(graph_steps=-1),
              dict(geometry_early=1, block_size=128, min_blocks=8 if f32 else 1),
              dict(block_size=128, min_blocks=8 if f32 else 1, stages=4),
              dict(grid=3), dict(grid=100000)]
    if f32:
        shapes += [dict(block_size=512, min_blocks=2), dict(block_size=128, min_blocks=8, geometry_early=1, stages=5)]
    for kw in shapes:
        got, t, info = _gpu_run(mi, 301, precision=precision, activity=1, **kw)
        assert t == tref, kw
        assert all(np.array_equal(x, y) for x, y in zip(ref, got)), kw
        assert info["n_active"] == iref["n_active"], kw


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
def test_activity_kernel_leaves_quiet_states_in_place_exactly(precision):
    # the activity kernel writes no state for a cell that is quiet in this and
    # the previous step (the output buffer, two steps old, holds it already);
    # through a caller state whose dry cells carry momentum, a set_state and a
    # boundary change in mid-run, calls of uneven length (graph boundaries) and
    # both grids, every step equals the one-cell kernel bit for bit
    mi = mg.river(101, 21, seed=8)
    dt = np.float32 if precision == capi.SWE_FP32 else np.float64
    rng = np.random.default_rng(3)
    dry = mi.h <= 1e-6
    hu, hv = mi.hu.copy(), mi.hv.copy()
    hu[dry] = rng.uniform(-0.5, 0.5, dry.sum())          # dry cells with momentum: zeroed by the first step
    hv[dry] = rng.uniform(-0.5, 0.5, dry.sum())
    h2 = mi.h.copy()
    h2[rng.random(mi.n_cells) < 0.02] += 0.3               # a second state: scattered wet cells
    runs = []
    for kw in (dict(), dict(activity=1), dict(activity=1, grid=5), dict(activity=1, block_size=128, min_blocks=8
                                                                            if precision == capi.SWE_FP32 else 1)):
        m = _gpu_mesh(mi, precision, **kw)
        m.set_state(mi.h.astype(dt), hu.astype(dt), hv.astype(dt))
        snaps = []
        for n in (1, 2, 53, 7):
            m.step(n)
            snaps.append(m.get_state())
        m.set_state(h2.astype(dt), mi.hu.astype(dt), mi.hv.astype(dt))
        for n in (3, 61):
            m.step(n)
            snaps.append(m.get_state())
        m.set_bc(mi.bcs[1][0], mg.BC_WALL)                 # static activity changes
        for n in (2, 49):
            m.step(n)
            snaps.append(m.get_state())
        runs.append((snaps, m.info()["t"]))
        m.close()
    ref, tref = runs[0]
    for snaps, t in runs[1:]:
        assert t == tref
        for a, b in zip(ref, snaps):
            assert all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
@pytest.mark.parametrize("maker", ["river", "dry_canal", "dam"])
def test_edge_pass_is_bitwise_neutral(precision, maker):
    # each interior flux evaluated once by the edge pass and applied with the
    # left/right sign: the same states, times and active counts as the cells'
    # own evaluations, through wet/dry fronts and every boundary kind
    if maker == "river":
        mi = mg.river(101, 21, seed=8)
    elif maker == "dry_canal":
        mi = mg.canal(401, 20, Lx=200.0, Ly=10.0, hR=0.0, seed=3, manning=0.03)
    else:
        mi = mg.dam_break_4k()
    ref, tref, iref = _gpu_run(mi, 301, precision=precision)
    f32 = precision == capi.SWE_FP32
    shapes = [dict(), dict(graph_steps=-1),
              dict(block_size=128, min_blocks=8) if f32 else dict(block_size=256, min_blocks=1)]
    for kw in shapes:
        got, t, info = _gpu_run(mi, 301, precision=precision, edge_pass=1,
                                **({"block_size": 256, "min_blocks": 4, "stages": 1} if f32 else {}) | kw)
        assert t == tref, kw
        assert all(np.array_equal(x, y) for x, y in zip(ref, got)), kw
        assert info["n_active"] == iref["n_active"], kw


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
def test_debug_checks_change_nothing_on_valid_meshes(precision):
    # with every index and boundary group checked before use, a valid mesh
    # steps to the same states and times, with status 0, in every step mode
    # (the check itself is tested on the host; no corrupt table reaches a GPU)
    mi = mg.river(101, 21, seed=8)
    f32 = precision == capi.SWE_FP32
    modes = [dict(), dict(activity=1), dict(edge_pass=1, **(dict(stages=1) if f32 else {})),
             dict(block_size=128, min_blocks=8 if f32 else 1, geometry_early=1)]
    for kw in modes:
        ref, tref, iref = _gpu_run(mi, 301, precision=precision, **kw)
        got, t, info = _gpu_run(mi, 301, precision=precision, debug_checks=1, **kw)
        assert info["status"] == 0, kw
        assert t == tref and info["n_active"] == iref["n_active"], kw
        assert all(np.array_equal(x, y) for x, y in zip(ref, got)), kw


def test_edge_pass_and_activity_exclude_each_other():
    mi = mg.dam_break_4k()
    with pytest.raises(capi.SWEError):
        capi.Mesh(mi.nodes, mi.tris, mi.z, mi.manning, activity=1, edge_pass=1)
    with pytest.raises(capi.SWEError):
        capi.Mesh(mi.nodes, mi.tris, mi.z, mi.manning, edge_pass=2)


def test_graphs_block_sizes_and_device_io_are_bitwise_neutral():
    mi = mg.river(100, 20, seed=8)
    ref, tref, _ = _gpu_run(mi, 301, graph_steps=-1, block_size=128)
    for kw in (dict(graph_steps=12, block_size=256), dict(graph_steps=48, block_size=512)):
        got, t, _ = _gpu_run(mi, 301, **kw)
        assert t == tref
        assert all(np.array_equal(a, b) for a, b in zip(ref, got))
    # device tensors in and out, split step calls
    m = _gpu_mesh(mi)
    dev = [torch.tensor(a, device="cuda") for a in (mi.h, mi.hu, mi.hv)]
    m.set_state(*dev)
    m.step(100, sync=False)
    m.step(0)
    m.step(201, sync=False)
    out = [torch.empty(mi.n_cells, dtype=torch.float64, device="cuda") for _ in range(3)]
    m.get_state(out)
    torch.cuda.synchronize()
    assert m.info()["t"] == tref
    assert all(np.array_equal(a, b.cpu().numpy()) for a, b in zip(ref, out))
    m.close()


def test_edge_cases():
    # one triangle with walls: stays at rest exactly, in every step mode (no
    # interior edge for the edge pass; one cell in a warp for the activity bytes)
    nodes = np.array([[0.0, 0.0], [1.0, 0.0], [0.0, 1.0]])
    for kw in (dict(), dict(activity=1), dict(edge_pass=1), dict(activity=1, precision=capi.SWE_FP32)):
        m = capi.Mesh(nodes, [[0, 1, 2]], [0.0], [0.0], **kw)
        m.set_state(*(np.array([v], dtype=m.dtype) for v in (1.0, 0.0, 0.0)))
        m.step(10)
        h, hu, hv = m.get_state()
        # the three wall pressures cancel to round-off (FP32: ~1e-6 of h sqrt(g h))
        tol = 1e-5 if m.dtype == np.float32 else 1e-14
        assert h[0] == 1.0 and abs(hu[0]) < tol and abs(hv[0]) < tol, kw
        ch = m.autotune(trial_steps=1)
        assert ch["grid"] == 1
        m.step(5)
        assert m.get_state()[0][0] == 1.0
        m.close()
    # all dry: no CFL step, in every mode
    mi = mg.dam_break_4k()
    zero = np.zeros(mi.n_cells)
    for kw in (dict(), dict(activity=1), dict(edge_pass=1)):
        m = _gpu_mesh(mi, **kw)
        m.set_state(zero, zero, zero)
        with pytest.raises(capi.SWEError) as e:
            m.step(3)
        assert e.value.code == capi.SWE_EDRY
        assert np.array_equal(m.get_state()[0], zero)
        m.close()
    # a non-finite depth in a wet cell: the step flags it (SWE_ENONFINITE), in
    # every mode and precision (the failure is made on the host, in the input)
    bad = mi.h.copy()
    k = int(np.flatnonzero(mi.h > 5.0)[mi.n_cells // 8])
    bad[k] = np.nan
    for kw in (dict(), dict(activity=1), dict(edge_pass=1), dict(precision=capi.SWE_FP32)):
        m = _gpu_mesh(mi, **kw)
        m.set_state(*(a.astype(m.dtype) for a in (bad, mi.hu, mi.hv)))
        with pytest.raises(capi.SWEError) as e:
            m.step(3)
        assert e.value.code == capi.SWE_ENONFINITE, kw
        m.close()
    # bad arguments are rejected on the host
    m = _gpu_mesh(mi)
    with pytest.raises(capi.SWEError) as e:
        m.step(1)
    assert e.value.code == capi.SWE_EINVAL        # no state yet
    with pytest.raises(capi.SWEError) as e:
        m.set_bc(np.array([[0, 5000]]), capi.SWE_BC_WALL)
    assert e.value.code == capi.SWE_EINVAL
    m.set_state(mi.h, mi.hu, mi.hv)
    with pytest.raises(capi.SWEError):
        m.step(1, cfl=-1.0)
    assert m.step(0) == 0.0
    m.close()


# ---------------------------------------------------------------------------
# Full-size workloads, in the launch configuration the bench times
# ---------------------------------------------------------------------------

def _first_step_sampled(mi, precision, n_sample=20000, seed=0):
    """GPU U^1 from the seeded U^0 against the oracle's step at sampled cells
    (the oracle computes its own time step from U^0)."""
    m = _gpu_mesh(mi, precision)
    npdt = np.float32 if precision == capi.SWE_FP32 else np.float64
    m.set_state(mi.h.astype(npdt), mi.hu.astype(npdt), mi.hv.astype(npdt))
    t1 = m.step(1)
    g1 = [a.astype(np.float64) for a in m.get_state()]
    m.close()
    M = _orc_mesh(mi)
    u0 = [a.astype(npdt).astype(np.float64) for a in (mi.h, mi.hu, mi.hv)]
    odt = M.dt(*u0, 0.9)
    # a random sample plus every cell on an inflow or stage edge, where the
    # first step already moves water (elsewhere the water starts at rest)
    nbr = M.geometry()["nbr"]
    driven = np.flatnonzero((nbr < -1).any(axis=1))
    rnd = np.random.default_rng(seed).choice(mi.n_cells, size=min(n_sample, mi.n_cells), replace=False)
    cells = np.unique(np.concatenate([rnd, driven]))
    o = M.step_cells(*u0, odt, cells)
    return g1, o, cells, t1, odt, M


def test_full_size_dry_canal_1m_fp64_against_oracle():
    # the 1,000,000-cell dry-bed canal, 2000 FP64 steps, element by element
    mi = mg.dam_break_dry_1m()
    M = _orc_mesh(mi)
    oh, ohu, ohv, ot, oc = M.run(mi.h, mi.hu, mi.hv, 2000, 0.9)
    (gh, ghu, ghv), t, info = _gpu_run(mi, 2000)
    assert info["status"] == 0 and info["n_clamped"] == oc
    assert t == pytest.approx(ot, rel=1e-12)
    for a, b in ((gh, oh), (ghu, ohu), (ghv, ohv)):
        assert rel_err(a, b) <= FP64_TOL
    wet = elem_rel_err((gh, ghu, ghv), (oh, ohu, ohv))
    print(f"1M dry-bed canal, 2000 steps: element-wise error on wet cells {wet}")
    assert all(e <= t for e, t in zip(wet, ELEM_TOL_FP64)), wet
    # Ritter: the wet front never passes 2 c0 t beyond the dam
    cx = mi.centroids()[:, 0]
    front = cx[gh > 1e-3].max()
    assert 100.0 + 0.5 * 2 * math.sqrt(9.81 * 10.0) * t < front <= 100.0 + 2 * math.sqrt(9.81 * 10.0) * t + 0.2
    # FP32 against FP64 after the same 2000 steps
    (f32, _, _), t32, _ = _gpu_run(mi, 2000, precision=capi.SWE_FP32)
    assert t32 == pytest.approx(t, rel=1e-4)
    assert rel_err(f32, gh) <= FP32_TOL
    # the edge pass (each interior flux once) at full size: bit for bit
    (eh, ehu, ehv), te, _ = _gpu_run(mi, 2000, edge_pass=1)
    assert te == t
    assert all(np.array_equal(x, y) for x, y in ((eh, gh), (ehu, ghu), (ehv, ghv)))


def _oracle_to_time(mi, T):
    """The oracle's state at time T (CFL 0.9 steps, the last one shortened)."""
    M = _orc_mesh(mi)
    h, hu, hv, t = mi.h.copy(), mi.hu.copy(), mi.hv.copy(), 0.0
    while t < T:
        dt = min(M.dt(h, hu, hv, 0.9), T - t)
        h, hu, hv, _ = M.step(h, hu, hv, dt)
        t += dt
    return h


def _cell_areas(mi):
    p = mi.nodes[mi.tris]
    return 0.5 * np.abs((p[:, 1, 0] - p[:, 0, 0]) * (p[:, 2, 1] - p[:, 0, 1]) -
                        (p[:, 2, 0] - p[:, 0, 0]) * (p[:, 1, 1] - p[:, 0, 1]))


def test_full_size_ritter_dam_break_against_exact_solution():
    # the 1M dry-bed canal's frictionless twin (Ritter, Section 6.3), 2000 FP64
    # steps on the GPU: the L1 depth error against the exact solution at the
    # run's time is below the oracle's own error on the 800 x 40 canal of the
    # convergence pin at that time (the scheme converges at first order, so
    # the 2.5x finer mesh must do better), and the front lies behind 2 c0 t
    from oracle import analytic
    mi = mg.dam_break_dry_1m(manning=0.0)
    (gh, _, _), t, info = _gpu_run(mi, 2000)
    assert info["status"] == 0
    area = _cell_areas(mi)
    cx = mi.centroids()[:, 0]
    he, _ = analytic.dam_break(cx, t, 10.0, 0.0, 100.0)
    err = float(np.sum(np.abs(gh - he) * area) / area.sum())
    coarse = mg.canal(800, 40, 200.0, 10.0, 0.2, 1, 10.0, 0.0, 100.0, 0.0)
    oh = _oracle_to_time(coarse, t)
    ca, ccx = _cell_areas(coarse), coarse.centroids()[:, 0]
    hc, _ = analytic.dam_break(ccx, t, 10.0, 0.0, 100.0)
    err_coarse = float(np.sum(np.abs(oh - hc) * ca) / ca.sum())
    print(f"Ritter at t = {t:.3f} s: L1 depth error {err:.4e} (1M cells, GPU) against {err_coarse:.4e} "
          f"(64k cells, oracle)")
    assert err < err_coarse, (err, err_coarse)
    c0 = math.sqrt(9.81 * 10.0)
    front = cx[gh > 1e-3].max() - 100.0
    assert 0.8 * 2 * c0 * t < front <= 2 * c0 * t + 0.2, (front, 2 * c0 * t)


def test_full_size_wet_river_1m_fp64_against_oracle():
    # the 1,001,728-cell fully wet river of the adjoint workload, 1000 FP64 steps
    mi = mg.river_adjoint_1m()
    M = _orc_mesh(mi)
    oh, ohu, ohv, ot, oc = M.run(mi.h, mi.hu, mi.hv, 1000, 0.9)
    (gh, ghu, ghv), t, info = _gpu_run(mi, 1000)
    assert info["n_clamped"] == oc == 0        # no depth clamped on this workload
    assert t == pytest.approx(ot, rel=1e-12)
    for a, b in ((gh, oh), (ghu, ohu), (ghv, ohv)):
        assert rel_err(a, b) <= FP64_TOL
    wet = elem_rel_err((gh, ghu, ghv), (oh, ohu, ohv))
    print(f"1M wet river, 1000 steps: element-wise error on wet cells {wet}")
    assert all(e <= t for e, t in zip(wet, ELEM_TOL_FP64)), wet


def test_full_size_river_13m_first_step_and_fp32_against_fp64():
    mi = mg.river_13m()
    for precision, tol in ((capi.SWE_FP64, 1e-13), (capi.SWE_FP32, 1e-5)):
        g1, o, cells, t1, odt, _ = _first_step_sampled(mi, precision)
        assert t1 == pytest.approx(odt, rel=1e-13 if precision == capi.SWE_FP64 else 1e-6)
        # a momentum field that is zero in exact arithmetic (water at rest)
        # is normalised by the shallow-water momentum scale h sqrt(g h)
        hmax = float(np.abs(o[0]).max())
        qscale = hmax * math.sqrt(9.81 * hmax)
        for k in range(3):
            d = np.abs(g1[k][cells] - o[k])
            w = int(np.argmax(d))
            den = max(float(np.abs(o[k]).max()), qscale if k else 0.0, 1e-30)
            assert d.max() / den <= tol, (precision, k, int(cells[w]), g1[k][cells][w], o[k][w], den)
    # after 1000 steps (the bench's launch configuration) FP32 stays within
    # 1e-4 of FP64
    (s32, t32, i32) = _gpu_run(mi, 1000, precision=capi.SWE_FP32)
    (s64, t64, i64) = _gpu_run(mi, 1000)
    assert i32["status"] == 0 and i64["status"] == 0
    assert t32 == pytest.approx(t64, rel=1e-4)
    for a, b in zip(s32, s64):
        assert rel_err(a, b) <= FP32_TOL
    # the activity kernel (the shape the autotuner picks for this mesh) at full
    # size: bit for bit the neighbour-test kernel, with the same active count
    (sa, ta, ia) = _gpu_run(mi, 1000, precision=capi.SWE_FP32, activity=1, block_size=128, min_blocks=8,
                            geometry_early=1)
    assert ta == t32 and ia["n_active"] == i32["n_active"]
    assert all(np.array_equal(x, y) for x, y in zip(sa, s32))


def test_full_size_river_13m_1000_steps_against_oracle():
    # the headline workload: the 12,999,168-cell river, 1000 whole-mesh steps
    # of the FP64 oracle on the host cores (a few minutes) against the GPU in
    # FP64 and in FP32 in the launch shape the library's autotuner picks for it
    mi = mg.river_13m()
    M = _orc_mesh(mi)
    oh, ohu, ohv, ot, oc = M.run(mi.h, mi.hu, mi.hv, 1000, 0.9)
    ref = (oh, ohu, ohv)
    (s64, t64, i64) = _gpu_run(mi, 1000)
    assert i64["status"] == 0 and i64["n_clamped"] == oc
    assert t64 == pytest.approx(ot, rel=1e-12)
    for a, b in zip(s64, ref):
        assert rel_err(a, b) <= FP64_TOL
    wet64 = elem_rel_err(s64, ref)
    # FP32 state, FP64 time step, tuned as the bench tunes it (after a warm-up;
    # the tuner's trials leave the state untouched)
    m = _gpu_mesh(mi, capi.SWE_FP32)
    m.set_state(mi.h.astype(np.float32), mi.hu.astype(np.float32), mi.hv.astype(np.float32))
    m.step(100, 0.9)
    shape = m.autotune(8)
    t32 = m.step(900, 0.9)
    s32 = [o.astype(np.float64) for o in m.get_state()]
    i32 = m.info()
    m.close()
    assert i32["status"] == 0
    assert t32 == pytest.approx(ot, rel=1e-4)
    for a, b in zip(s32, ref):
        assert rel_err(a, b) <= FP32_TOL, shape
    wet32 = elem_rel_err(s32, ref)
    print(f"13M river, 1000 steps: element-wise error on wet cells FP64 {wet64}, FP32 {wet32}; shape {shape}")
    assert all(e <= t for e, t in zip(wet64, ELEM_TOL_FP64)), wet64
    assert all(e <= t for e, t in zip(wet32, ELEM_TOL_FP32)), wet32


@pytest.mark.parametrize("init", ["inclined_plane", "dam_failure"])
def test_river_initialisations_fp64(init):
    # the paper's other river initial states (Sections 6.5.1 and 6.4.2) on
    # the synthetic reach: GPU against the oracle after 600 steps
    mi = mg.river(160, 32, seed=9)
    if init == "inclined_plane":
        mi = mg.inclined_plane(mi, eta_up=3.0, eta_down=1.0)
    else:
        mi = mg.dam_failure(mi, x_dam=10000.0)
    M = _orc_mesh(mi)
    oh, ohu, ohv, ot, oc = M.run(mi.h, mi.hu, mi.hv, 600, 0.9)
    (gh, ghu, ghv), t, info = _gpu_run(mi, 600)
    assert t == pytest.approx(ot, rel=1e-12) and info["n_clamped"] == oc
    for a, b in ((gh, oh), (ghu, ohu), (ghv, ohv)):
        assert rel_err(a, b) <= FP64_TOL


@pytest.mark.parametrize("precision", [capi.SWE_FP64, capi.SWE_FP32])
def test_hll_flux_variant(precision):
    # the HLL flux (Eq 17-18 for all components) against the oracle's
    n = 3000
    st = _random_states(n, 11)
    tdt = torch.float64 if precision == capi.SWE_FP64 else torch.float32
    dev = [torch.tensor(a, dtype=tdt, device="cuda") for a in st]
    G = [torch.empty(n, dtype=tdt, device="cuda") for _ in range(3)]
    capi.riemann_flux(precision, *dev, *G, flux=capi.SWE_FLUX_HLL)
    torch.cuda.synchronize()
    got = np.stack([g.double().cpu().numpy() for g in G], axis=1)
    st_in = [d.double().cpu().numpy() for d in dev]
    ref = np.array([oracle.hll(*(float(a[i]) for a in st_in)) for i in range(n)])
    err = np.abs(got - ref).max(axis=1) / np.maximum(np.abs(ref).max(axis=1), 1.0)
    tol = 1e-13 if precision == capi.SWE_FP64 else 2e-5
    bad = np.where(err > tol)[0]
    assert len(bad) <= (0 if precision == capi.SWE_FP64 else n // 500), (err.max(), bad)
    for i in bad:
        margin = _tie_margin(*(float(a[i]) for a in st_in), contact=False)
        assert margin <= TIE_MARGIN, (i, err[i], margin, [float(a[i]) for a in st_in])
    if precision == capi.SWE_FP64:
        mi = mg.river(160, 32, seed=5)
        M = _orc_mesh(mi)
        M.set_flux(1)
        oh, ohu, ohv, ot, oc = M.run(mi.h, mi.hu, mi.hv, 1000, 0.9)
        (gh, ghu, ghv), t, info = _gpu_run(mi, 1000, flux=capi.SWE_FLUX_HLL)
        assert t == pytest.approx(ot, rel=1e-12)
        for a, b in ((gh, oh), (ghu, ohu), (ghv, ohv)):
            assert rel_err(a, b) <= FP64_TOL


def _hllc_wide(hL, unL, utL, hR, unR, utR, h_dry):
    """Eq 17-26 in numpy's extended type, whose exponents neither under- nor
    overflow here: G, (S_L, S_R)."""
    t = np.longdouble
    hL, unL, utL, hR, unR, utR, g, h_dry = (t(x) for x in (hL, unL, utL, hR, unR, utR, 9.81, h_dry))
    dryL, dryR = hL <= h_dry, hR <= h_dry
    if dryL and dryR:
        return np.zeros(3), np.zeros(2)
    aL, aR = np.sqrt(g * hL), np.sqrt(g * hR)
    if dryL:
        SL, SR, left = unR - 2 * aR, unR + aR, None
    elif dryR:
        SL, SR, left = unL - aL, unL + 2 * aL, None
    else:
        h0 = (hL + hR) * (t(0.5) - t(0.25) * (unR - unL) / (aL + aR))
        pL = pR = t(1)
        if h0 > min(hL, hR):
            gL, gR = (np.sqrt(g * (h0 + h) / (2 * h0 * h)) for h in (hL, hR))
            hs = (hL * gL + hR * gR + unL - unR) / (gL + gR)
            pL, pR = (np.sqrt(hs * (hs + h) / 2) / h if hs > h else t(1) for h in (hL, hR))
        SL, SR = unL - aL * pL, unR + aR * pR
        left = SL >= 0 or (SR > 0 and (SL * hR * (unR - SR) - SR * hL * (unL - SL)) /
                           (hR * (unR - SR) - hL * (unL - SL)) >= 0)
    if left is None:
        left = (SL if dryL else SR) >= 0
    F = [(h * u, h * u * u + g * h * h / 2) for h, u in ((hL, unL), (hR, unR))]
    if SL >= 0:
        G = F[0]
    elif SR <= 0:
        G = F[1]
    else:
        U = [(h, h * u) for h, u in ((hL, unL), (hR, unR))]
        G = [(SR * F[0][c] - SL * F[1][c] + SR * SL * (U[1][c] - U[0][c])) / (SR - SL) for c in range(2)]
    return np.array([G[0], G[1], G[0] * (utL if left else utR)], t), np.array([SL, SR], t)


def test_riemann_flux_far_from_any_flow_fp64():
    # depths from denormal to 1e150 and a dry threshold of 1e-322, which the
    # flux alone takes.  Equal depths below 1e-300, whose reciprocals overflow.
    # Some 40 operations of 2^-53 each on terms that nearly cancel by at most
    # 2^4: 1e-13 of the largest term.  Products below the normal range are
    # rounded to 2^-1074, and so is g h under the root
    rng = np.random.default_rng(12)
    states = []
    for _ in range(4000):
        h = float(10.0 ** rng.uniform(-315.0, 150.0)) if rng.random() < 0.9 else 0.0
        k = float(rng.choice([1.0, 1.0, 0.5, 2.0])) if h > 1e-300 else 1.0
        a = math.sqrt(9.81 * h)
        f = np.sort(rng.uniform(-0.9, 0.9, 2)) + float(rng.choice([0.0, 3.0, -3.0]))
        states.append((h, a * f[0], a, h * k, a * f[1], -0.5 * a))
    states += [(0.0, 0.0, 0.0, 3e-310, 0.0, 1.0), (3e-310, 0.0, 1.0, 0.0, 0.0, 0.0),
               (1e-250, 1e30, 2.0, 2e-250, 1e30, 1.0)]
    st = [np.array(c) for c in zip(*states)]
    dev = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in st]
    G = [torch.empty(len(states), dtype=torch.float64, device="cuda") for _ in range(3)]
    S = torch.empty((len(states), 3), dtype=torch.float64, device="cuda")
    capi.riemann_flux(capi.SWE_FP64, *dev, *G, S, h_dry=1e-322)
    torch.cuda.synchronize()
    got_g, got_s = torch.stack(G, 1).cpu().numpy(), S.cpu().numpy()[:, :2]
    for s, gg, gs in zip(states, got_g, got_s):
        hL, unL, utL, hR, unR, utR = s
        ref_g, ref_s = _hllc_wide(*s, h_dry=1e-322)
        h = np.longdouble(max(hL, hR))
        c = max(abs(unL), abs(unR), abs(utL), abs(utR), math.sqrt(9.81 * max(hL, hR)))
        root = 5e-324 / max(float(h), 5e-324)   # of g h
        assert np.all(np.abs(gs - ref_s) <= (1e-13 + root) * 4 * c), (s, gs, ref_s)
        scale = np.array([h * c, h * c * c, h * c * c], np.longdouble)
        assert np.all(np.abs(gg - ref_g) <= 1e-13 * 4 * scale + 1e-320), (s, gg, ref_g)


@pytest.mark.parametrize("flux", [capi.SWE_FLUX_HLLC, capi.SWE_FLUX_HLL])
def test_riemann_flux_without_gravity_fp64(flux):
    # the flux alone takes any g.  Without gravity the wave speeds are the
    # velocities (no star depth exists where they converge, and none is needed);
    # negative g has no wave speeds: NaN, not a number that looks like a flux
    st = [(1.0, -1.0, 2.0, 3.0, 0.5, -1.0), (2.0, 1.0, 0.5, 1.0, 2.0, 0.25), (1.0, -3.0, 0.5, 2.0, -1.0, 4.0),
          (1.0, 1.0, 0.0, 2.0, -1.0, 0.0), (4.0, -0.5, 1.0, 0.25, -2.0, 1.0)]
    dev = [torch.tensor(c, dtype=torch.float64, device="cuda") for c in zip(*st)]
    G = [torch.empty(len(st), dtype=torch.float64, device="cuda") for _ in range(3)]
    for g in (0.0, -9.81):
        capi.riemann_flux(capi.SWE_FP64, *dev, *G, g=g, flux=flux)
        got = torch.stack(G, 1).cpu().numpy()
        for k, (hL, uL, vL, hR, uR, vR) in enumerate(st):
            if g < 0.0:
                assert np.all(np.isnan(got[k])), (g, st[k], got[k])
                continue
            FL, FR = [np.array([h * u, h * u * u, h * u * v]) for h, u, v in ((hL, uL, vL), (hR, uR, vR))]
            dU = np.array([hR - hL, hR * uR - hL * uL, hR * vR - hL * vL])
            F = FL if uL >= 0.0 else (FR if uR <= 0.0 else (uR * FL - uL * FR + uL * uR * dU) / (uR - uL))
            n = 3 if flux == capi.SWE_FLUX_HLL else 2   # (HLLC: S* is 0/0 here, either side's tangential velocity)
            assert np.allclose(got[k][:n], F[:n], rtol=1e-14, atol=1e-14), (st[k], got[k], F)
