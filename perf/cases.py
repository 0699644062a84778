"""The work that users of this solver have it do, as timed cases.

A program builds a mesh once (and lets the library tune its launch shape when
the run is long), then sets initial states and advances them; it runs
ensembles, differentiates a gauge misfit, drives a reach to its steady state
with the diagnostics, or evaluates the Riemann flux alone.  The meshes are the
handles that such a program keeps; the states, target depths and flux inputs
are made from the seed.

``exact`` restates the scheme (Eq 12-37 of the paper, the readings of the
solver's documentation) in plain PyTorch FP64 on a geometry of its own.
"""
from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

from paper_2010_14416_gb300 import capi

G, H_DRY, CFL = 9.81, 1e-6, 0.9
WALL, INFLOW, TRANSMISSIVE, STAGE = 0, 1, 2, 3
CANAL_L, RIVER_L = (200.0, 10.0), (20000.0, 2000.0)


def listed():
    return [
        # the dam break in a 4,000-cell canal, the smallest run: 500 steps, each bound by latency; no tuning
        dict(name="canal4k_f64", kind="run", domain="canal", nx=200, ny=10, f32=False, steps=500, tuned=False,
             h_right=1.0, manning=0.0, hll=False),
        # a coarse partly dry reach in FP32 with the library's defaults, as in a quick scenario study
        dict(name="river20k_f32", kind="run", domain="river", nx=316, ny=32, f32=True, steps=240, tuned=False,
             wet=False, hll=False),
        # the dam break onto a dry bed refined to 1M cells, in both precisions, tuned
        dict(name="canal1m_f64", kind="run", domain="canal", nx=2000, ny=250, f32=False, steps=48, tuned=True,
             h_right=0.0, manning=0.03, hll=False),
        dict(name="canal1m_f32", kind="run", domain="canal", nx=2000, ny=250, f32=True, steps=192, tuned=True,
             h_right=0.0, manning=0.03, hll=False),
        # the 13M-cell reach, 94 % dry: the flagship run and the largest mesh
        dict(name="river13m_f32", kind="run", domain="river", nx=8064, ny=806, f32=True, steps=96, tuned=True,
             wet=False, hll=False),
        # a reach in flood, every cell wet
        dict(name="river3m_wet_f32", kind="run", domain="river", nx=4000, ny=401, f32=True, steps=48, tuned=True,
             wet=True, hll=False),
        # uncertainty propagation: uneven canal and river members advanced together, in both precisions
        dict(name="ensemble24_f32", kind="ensemble", members=24, lo=20000, hi=500000, f32=True, steps=48),
        dict(name="ensemble12_f64", kind="ensemble", members=12, lo=20000, hi=200000, f32=False, steps=12),
        # inverse analysis: gradient of a gauge misfit, a coarse reach and a finer one
        dict(name="adjoint20k", kind="adjoint", nx=316, ny=32, steps=200, every=50, gauges=64),
        dict(name="adjoint250k", kind="adjoint", nx=1118, ny=112, steps=48, every=16, gauges=64),
        # the stabilisation run before a production run, with its inflow and outflow rates
        dict(name="steady100k_f32", kind="steady", nx=707, ny=71, f32=True, steps=200, check=20),
        # the Riemann flux alone, on a batch
        dict(name="riemann1m_f64", kind="riemann", n=1 << 20, f32=False, hll=False),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "ensemble", "adjoint", "steady", "riemann"])
    f32 = rng.random() < 0.5
    hll = rng.random() < 0.2
    if kind == "run":
        n = _between(rng, 2000, 4000000 if f32 else 1000000)
        steps = max(6, min(500, int((1e8 if f32 else 3e7) / n)) + rng.randint(0, 5))
        if rng.random() < 0.4:
            ny = max(2, int(math.sqrt(n / 40.0)))
            return dict(kind="run", domain="canal", nx=max(8, n // (2 * ny)), ny=ny, f32=f32, steps=steps,
                        tuned=rng.random() < 0.7, h_right=rng.choice([0.0, 1.0]),
                        manning=rng.choice([0.0, 0.03]), hll=hll)
        ny = max(4, int(math.sqrt(n / 20.0)))
        return dict(kind="run", domain="river", nx=max(16, n // (2 * ny)), ny=ny, f32=f32, steps=steps,
                    tuned=rng.random() < 0.7, wet=rng.random() < 0.4, hll=hll)
    if kind == "ensemble":
        lo = _between(rng, 5000, 50000)
        return dict(kind="ensemble", members=rng.randint(3, 16), lo=lo, hi=_between(rng, 2 * lo, 200000), f32=f32,
                    steps=rng.randint(6, 40) if f32 else rng.randint(3, 12))
    if kind == "adjoint":
        n = _between(rng, 4000, 250000)
        ny = max(4, int(math.sqrt(n / 20.0)))
        return dict(kind="adjoint", nx=n // (2 * ny), ny=ny, steps=max(12, min(150, int(8e6 / n))),
                    every=rng.choice([8, 13, 25]), gauges=rng.randint(1, 100))
    if kind == "steady":
        n = _between(rng, 5000, 300000)
        ny = max(4, int(math.sqrt(n / 20.0)))
        return dict(kind="steady", nx=n // (2 * ny), ny=ny, f32=f32, steps=rng.randint(30, 120),
                    check=rng.choice([7, 10, 25]))
    return dict(kind="riemann", n=_between(rng, 1000, 8000000), f32=f32, hll=hll)


# ---- inputs ------------------------------------------------------------------------------


def _grid(nx, ny, lengths, seed):
    """Jittered quads, each split into two triangles: nodes, tris, the node
    pairs of the left and right side."""
    r = np.random.default_rng(seed)
    lx, ly = lengths
    x, y = np.meshgrid(np.linspace(0.0, lx, nx + 1), np.linspace(0.0, ly, ny + 1))
    if nx > 1 and ny > 1:
        x[1:-1, 1:-1] += r.uniform(-0.2, 0.2, (ny - 1, nx - 1)) * lx / nx
        y[1:-1, 1:-1] += r.uniform(-0.2, 0.2, (ny - 1, nx - 1)) * ly / ny
    p = (np.arange(ny)[:, None] * (nx + 1) + np.arange(nx)).ravel().astype(np.int32)
    q = p + nx + 1
    tris = np.stack([p, p + 1, q + 1, p, q + 1, q], 1).reshape(-1, 3)
    j = np.arange(ny, dtype=np.int32) * (nx + 1)
    left, right = np.stack([j, j + nx + 1], 1), np.stack([j + nx, j + 2 * nx + 1], 1)
    return np.stack([x.ravel(), y.ravel()], 1), tris, left, right, r


def _centroids(nodes, tris):
    return (nodes[tris[:, 0]] + nodes[tris[:, 1]] + nodes[tris[:, 2]]) / 3.0


def _bed(x, y):
    """A meandering channel 200 m wide and 5 m deep below a floodplain at +2 m."""
    d = np.abs(y - (1000.0 + 400.0 * np.sin(2.0 * np.pi * x / 2000.0)))
    return np.where(d < 100.0, 2.0 - 2.5 * (1.0 + np.cos(np.pi * d / 100.0)), 2.0), d < 100.0


@lru_cache(maxsize=64)
def _inputs(domain, nx, ny, wet=False, manning=0.0, discharge=2000.0, seed=1):
    """The mesh as a file of it would hold it: nodes, tris, bed, Manning
    coefficients, boundary groups, centroids, the free surface it starts from."""
    if domain == "canal":
        nodes, tris, left, _, _ = _grid(nx, ny, CANAL_L, seed)
        n = len(tris)
        groups = [(left, INFLOW, discharge)] if discharge > 0.0 else []
        return nodes, tris, np.zeros(n), np.full(n, manning), groups, _centroids(nodes, tris), 0.0
    nodes, tris, left, right, r = _grid(nx, ny, RIVER_L, seed)
    c = _centroids(nodes, tris)
    z, channel = _bed(c[:, 0], c[:, 1])
    bump = np.zeros(len(tris), np.float64)
    order = np.argsort(c[:, 0])
    xs = c[order, 0]
    for _ in range(60):      # mounds on the floodplain
        s, a, bx, by = r.uniform(50.0, 300.0), r.uniform(0.5, 3.0), r.uniform(0, RIVER_L[0]), r.uniform(0, RIVER_L[1])
        k = order[np.searchsorted(xs, bx - 3.5 * s):np.searchsorted(xs, bx + 3.5 * s)]
        bump[k] += a * np.exp(-0.5 * ((c[k, 0] - bx) ** 2 + (c[k, 1] - by) ** 2) / (s * s))
    z = z + np.where(channel, 0.0, bump) + 1e-4 * (RIVER_L[0] - c[:, 0])
    man = r.uniform(0.02, 0.06, len(tris)) if manning == 0.0 else np.full(len(tris), manning)
    eta = float(z.max()) + 0.5 if wet else 1.0
    mid = 0.5 * (nodes[left[:, 0], 1] + nodes[left[:, 1], 1])
    inflow = left[_bed(np.zeros_like(mid), mid)[1]]
    # the numbering of an unstructured mesher: no locality
    cells, points = r.permutation(len(tris)), r.permutation(len(nodes)).astype(np.int32)
    back = np.empty_like(points)
    back[points] = np.arange(len(points), dtype=np.int32)
    nodes, tris = nodes[points], np.ascontiguousarray(back[tris[cells]])
    groups = [(back[inflow], INFLOW, discharge)] if len(inflow) else []
    return nodes, tris, z[cells], man[cells], groups + [(back[right], STAGE, eta)], c[cells], eta


@lru_cache(maxsize=64)
def _mesh(args, f32, hll=False):
    """A program's mesh handle: built once, kept for all its states."""
    nodes, tris, z, man, groups, _, _ = _inputs(*args)
    m = capi.Mesh(nodes, tris, z, man, precision=capi.SWE_FP32 if f32 else capi.SWE_FP64,
                  flux=capi.SWE_FLUX_HLL if hll else capi.SWE_FLUX_HLLC)
    for pairs, kind, value in groups:
        m.set_bc(pairs, kind, value)
    return m


@lru_cache(maxsize=64)
def _tuned(args, f32, hll):
    """The same with the launch shape that the library's tuner keeps for it."""
    m = _mesh.__wrapped__(args, f32, hll)
    m.set_state(*_state(args, f32, 0, dam=100.0))
    m.autotune()
    return m


def _state(args, f32, seed, dam=None, h_right=0.0, u0=0.0, slope=0.0, h_left=10.0):
    """Depth and discharge of a smooth initial state, on the device."""
    _, _, z, _, _, c, eta = _inputs(*args)
    r = np.random.default_rng((seed, 77))
    dev = torch.device("cuda")
    x, zt = torch.from_numpy(c[:, 0]).to(dev), torch.from_numpy(z).to(dev)
    lx = CANAL_L[0] if args[0] == "canal" else RIVER_L[0]
    wave = torch.sin(2.0 * math.pi * (r.uniform(1.0, 4.0) * x / lx + r.uniform()))
    if args[0] == "canal":
        where = r.uniform(85.0, 115.0)
        h = torch.where(x < where, h_left * (1.0 + 0.01 * wave), torch.full_like(x, h_right))
    else:
        h = torch.clamp(eta + 0.1 * wave + slope * (1.0 - x / lx) - zt, min=0.0)
    hu = h * (u0 * r.uniform(0.6, 1.4))
    dt = torch.float32 if f32 else torch.float64
    return h.to(dt).contiguous(), hu.to(dt).contiguous(), torch.zeros_like(h, dtype=dt)


def _mesh_args(case):
    if case["kind"] == "run" and case["domain"] == "canal":
        return ("canal", case["nx"], case["ny"], False, case["manning"], 0.0)
    if case["kind"] == "adjoint":
        return ("river", case["nx"], case["ny"], True)
    return ("river", case["nx"], case["ny"], bool(case.get("wet", False)))


def _members(case):
    """(mesh args, downstream depth) of the ensemble's members: uneven sizes,
    Manning and inflow of their own, canals and rivers in turn."""
    r = np.random.default_rng(5)
    sizes = np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), case["members"])).astype(int)
    out = []
    for k, n in enumerate(sizes):
        man, q = float(r.uniform(0.015, 0.08)), float(r.uniform(500.0, 3000.0))
        if k % 2 == 0:
            ny = max(2, int(math.sqrt(n / 40.0)))
            out.append(("canal", int(n) // (2 * ny), ny, False, man, q / 20.0, k + 1))
        else:
            ny = max(4, int(math.sqrt(n / 20.0)))
            out.append(("river", int(n) // (2 * ny), ny, False, man, q, k + 1))
    return out


def _start_of(case, seed):
    """The initial state of a run, an adjoint or a steady run."""
    args = _mesh_args(case)
    if case["kind"] == "adjoint":
        return _state(args, False, seed, u0=0.5, slope=1.0)
    if case["kind"] == "steady":
        return _state(args, case["f32"], seed, u0=0.5)
    return _state(args, case["f32"], seed, h_right=case.get("h_right", 0.0), u0=0.5 if case["domain"] == "river" else 0.0)


def _observed(case, seed, h):
    r = np.random.default_rng((seed, 99))
    at = np.sort(r.choice(h.numel(), case["gauges"], replace=False)).astype(np.int32)
    return at, h[torch.from_numpy(at).to(h.device).long()].cpu().numpy() + 0.05 * r.standard_normal(case["gauges"])


def _flux_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = lambda lo, hi: lo + (hi - lo) * torch.rand(case["n"], generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    hl = torch.exp(u(-3.0, 2.5))
    hr = hl * torch.exp(u(-0.7, 0.7))
    dry = u(0.0, 1.0)
    hl, hr = torch.where(dry < 0.03, torch.zeros_like(hl), hl), torch.where(dry > 0.97, torch.zeros_like(hr), hr)
    v = [hl, u(-3.0, 3.0), u(-2.0, 2.0), hr, u(-3.0, 3.0), u(-2.0, 2.0)]
    return [x.to(torch.float32 if case["f32"] else torch.float64) for x in v]


def prepare(case, seed):
    if case["kind"] == "riemann":
        v = _flux_inputs(case, seed)
        return dict(case=case, inputs=v, out=[torch.empty_like(v[0]) for _ in range(3)])
    if case["kind"] == "ensemble":
        members = _members(case)
        meshes = []
        for k, args in enumerate(members):
            m = _mesh(args, case["f32"])
            m.set_state(*_state(args, case["f32"], 1000 * seed + k, h_right=1.0))
            meshes.append(m)
        e = capi.Ensemble(meshes)
        e.autotune()
        sizes = [m.n_cells for m in meshes]
        dt = torch.float32 if case["f32"] else torch.float64
        out = [torch.empty(sum(sizes), dtype=dt, device="cuda") for _ in range(3)]
        return dict(case=case, ensemble=e, out=out, parts=list(zip(*(o.split(sizes) for o in out))))
    args = _mesh_args(case)
    hll = bool(case.get("hll", False))
    tuned = case.get("tuned", True)
    f32 = bool(case.get("f32", False))
    m = _tuned(args, f32, hll) if tuned else _mesh(args, f32, hll)
    start = _start_of(case, seed)
    state = dict(case=case, mesh=m, start=start, out=[torch.empty_like(x) for x in start])
    if case["kind"] == "adjoint":
        state["gauges"], state["target"] = _observed(case, seed, start[0])
        state["gradients"] = [torch.empty_like(start[0]) for _ in range(2)]
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "riemann":
        capi.riemann_flux(capi.SWE_FP32 if case["f32"] else capi.SWE_FP64, *state["inputs"], *state["out"],
                          flux=capi.SWE_FLUX_HLL if case["hll"] else capi.SWE_FLUX_HLLC)
        return state["out"]
    if case["kind"] == "ensemble":
        e = state["ensemble"]
        t = e.step(case["steps"])
        for k, part in enumerate(state["parts"]):
            e.get_state(k, out=part)
        return dict(state=state["out"], t=t)
    m = state["mesh"]
    m.set_state(*state["start"])
    out = {}
    if case["kind"] == "run":
        out["t"] = m.step(case["steps"], CFL)
    elif case["kind"] == "steady":
        _, _, out["t"] = m.run_to_steady(1e-12, cfl=CFL, check_every=case["check"], max_steps=case["steps"])
        d = m.diagnostics()
        out["volume"], out["discharge"] = d["volume"], d["discharge"]
    else:
        loss, gm, gz, dts = m.adjoint(case["steps"], state["gauges"], state["target"], cfl=CFL,
                                      checkpoint_every=case["every"], out=state["gradients"])
        out.update(loss=loss, grad_manning=gm, grad_bathy=gz, dts=dts)
    out["state"] = m.get_state(out=state["out"])
    return out


def work(case):
    """Each step reads and writes the state, and reads the bed, Manning
    coefficient, area, radius, edge vectors and neighbour indices (19 values
    less the indices' size), of the cells that have water or a wet neighbour;
    about 400 operations for each of them."""
    if case["kind"] == "riemann":
        return dict(bytes=case["n"] * 9 * (4 if case["f32"] else 8), flops=case["n"] * 120)
    if case["kind"] == "ensemble":
        cells = sum(2 * a[1] * a[2] * (1.0 if a[0] == "canal" else 0.07) for a in _members(case))
    else:
        share = 1.0
        if case["kind"] != "adjoint" and case.get("domain", "river") == "river" and not case.get("wet", False):
            share = 0.07
        elif case.get("domain") == "canal" and case["h_right"] == 0.0:
            share = 0.5
        cells = 2 * case["nx"] * case["ny"] * share
    per = 76 if case.get("f32", False) else 140
    times = 4.0 if case["kind"] == "adjoint" else 1.0   # the forward step, again, and its transpose
    return dict(bytes=cells * case["steps"] * per * times, flops=cells * case["steps"] * 400 * times)


# ---- the scheme in plain PyTorch, 64 bits --------------------------------------------------


def _or(mask, x, fill=1.0):
    return torch.where(mask, x, torch.full_like(x, fill))


def _flux(hl, unl, utl, hr, unr, utr, hll=False):
    """G~(U_L, U_R) in the edge's frame (Eq 17-26)."""
    wl, wr = hl > H_DRY, hr > H_DRY
    both, some = wl & wr, wl | wr
    al = torch.where(hl > 0, torch.sqrt(G * _or(hl > 0, hl)), torch.zeros_like(hl))
    ar = torch.where(hr > 0, torch.sqrt(G * _or(hr > 0, hr)), torch.zeros_like(hr))
    total = hl + hr
    h0 = 0.5 * total - 0.25 * (unr - unl) * total / _or(both, al + ar)
    rare = h0 <= torch.minimum(hl, hr)
    base = torch.clamp(0.5 * (al + ar) + 0.25 * (unl - unr), min=0.0)
    shock = both & ~rare
    h0s, ls, rs = _or(shock, h0), _or(shock, hl), _or(shock, hr)
    gl, gr = torch.sqrt(G * (h0s + ls) / (2.0 * h0s * ls)), torch.sqrt(G * (h0s + rs) / (2.0 * h0s * rs))
    hs = torch.where(rare, base * base / G, (ls * gl + rs * gr + unl - unr) / (gl + gr))
    upl, upr = both & (hs > hl), both & (hs > hr)

    def factor(up, h):
        a, b = _or(up, hs), _or(up, h)
        return torch.where(up, torch.sqrt(0.5 * a * (a + b)) / b, torch.ones_like(hs))

    sl, sr = unl - al * factor(upl, hl), unr + ar * factor(upr, hr)
    ml, mr = hl * (unl - sl), hr * (unr - sr)
    star = (sl * mr - sr * ml) / _or(both, mr - ml)
    sl = torch.where(both, sl, torch.where(wl, unl - al, unr - 2.0 * ar))
    sr = torch.where(both, sr, torch.where(wl, unl + 2.0 * al, unr + ar))
    star = torch.where(both, star, torch.where(wl, sr, sl))
    ql, qr = hl * unl, hr * unr
    pl, pr = ql * unl + 0.5 * G * hl * hl, qr * unr + 0.5 * G * hr * hr
    inside = (sl < 0) & (sr > 0) & some
    span = 1.0 / _or(inside, sr - sl)

    def middle(fl, fr, ul, ur):
        return torch.where(sl >= 0, fl, torch.where(sr <= 0, fr, (sr * fl - sl * fr + sr * sl * (ur - ul)) * span))

    g1, g2 = middle(ql, qr, hl, hr), middle(pl, pr, ql, qr)
    g3 = middle(ql * utl, qr * utr, hl * utl, hr * utr) if hll else g1 * torch.where(star >= 0, utl, utr)
    none = torch.zeros_like(g1)
    return torch.where(some, g1, none), torch.where(some, g2, none), torch.where(some, g3, none)


class _Scheme:
    """One mesh's explicit Euler step."""

    def __init__(self, args, hll=False):
        nodes, tris, z, man, groups, _, _ = _inputs(*args)
        dev = torch.device("cuda")
        self.hll = hll
        self.z, self.man = torch.from_numpy(z).to(dev), torch.from_numpy(man).to(dev)
        p, t = torch.from_numpy(nodes).to(dev), torch.from_numpy(tris).to(dev).long()
        n = t.shape[0]
        a, b = t, t.roll(-1, 1)
        e = p[b] - p[a]
        self.len = torch.sqrt((e * e).sum(2))
        self.n1, self.n2 = e[..., 1] / self.len, -e[..., 0] / self.len
        d1, d2 = p[t[:, 1]] - p[t[:, 0]], p[t[:, 2]] - p[t[:, 0]]
        self.area = 0.5 * (d1[:, 0] * d2[:, 1] - d1[:, 1] * d2[:, 0])
        self.radius = 2.0 * self.area / self.len.sum(1)
        size = p.shape[0]
        key = torch.minimum(a, b) * size + torch.maximum(a, b)
        order = torch.argsort(key.view(-1))
        sorted_key = key.view(-1)[order]
        twin = sorted_key[1:] == sorted_key[:-1]
        i, j = order[:-1][twin], order[1:][twin]
        k = torch.full((3 * n,), -1, dtype=torch.long, device=dev)
        k[i], k[j] = j // 3, i // 3
        self.inner = (k >= 0).view(n, 3)
        self.k = torch.where(self.inner, k.view(n, 3), torch.arange(n, device=dev)[:, None])
        self.kind = torch.where(self.inner, -1, 0)
        self.group = torch.where(self.inner, -1, 0)
        self.value = torch.zeros_like(self.len)
        self.groups = 1 + len(groups)
        for g, (pairs, kind, value) in enumerate(groups):
            q = torch.from_numpy(np.ascontiguousarray(pairs)).to(dev).long()
            there = torch.isin(key, q.min(1).values * size + q.max(1).values)
            self.kind[there], self.group[there] = kind, g + 1
            self.value[there] = value / self.len[there].sum() if kind == INFLOW else value

    def dt(self, h, hu, hv):
        wet = h > H_DRY
        hs = _or(wet, h)
        c = self.radius / (torch.sqrt(G * hs) + torch.sqrt((hu / hs) ** 2 + (hv / hs) ** 2))
        return CFL * torch.where(wet, c, torch.full_like(c, math.inf)).min()

    def fluxes(self, h, hu, hv, z):
        wet = h > H_DRY
        hs = _or(wet, h)
        none = torch.zeros_like(h)
        u, v = torch.where(wet, hu / hs, none), torch.where(wet, hv / hs, none)
        hi, ui, vi, zi = h[:, None], u[:, None], v[:, None], z[:, None]
        hk, uk, vk, zk = (torch.where(self.inner, q[self.k], q[:, None]) for q in (h, u, v, z))
        top = torch.maximum(zi.expand_as(zk), zk)
        own = torch.where(self.inner, torch.clamp(hi + zi - top, min=0.0), hi)
        ghost = torch.where(self.kind == STAGE, torch.clamp(self.value - zi, min=0.0), hi)
        other = torch.where(self.inner, torch.clamp(hk + zk - top, min=0.0), ghost)
        n1, n2 = self.n1, self.n2
        un, ut, unk, utk = ui * n1 + vi * n2, vi * n1 - ui * n2, uk * n1 + vk * n2, vk * n1 - uk * n2
        g1, g2, g3 = _flux(own, un, ut, other, unk, utk, self.hll)
        press = 0.5 * G * hi * hi
        wall, inflow = self.kind == WALL, self.kind == INFLOW
        rate = self.value * self.value / _or(wet, h)[:, None]
        jet = torch.where(inflow & wet[:, None], rate, torch.zeros_like(rate))
        zero = torch.zeros_like(g1)
        g1 = torch.where(wall, zero, torch.where(inflow, -self.value, g1))
        g2 = torch.where(wall | inflow, press + jet, g2)
        g3 = torch.where(wall | inflow, zero, g3)
        bed = torch.where(self.inner, 0.5 * G * (own * own - hi * hi), zero)
        return g1, g2 - bed, g2, g3

    def step(self, h, hu, hv, z, man, dt):
        n1, n2 = self.n1, self.n2
        g1, g2, _, g3 = self.fluxes(h, hu, hv, z)
        rh = -(self.len * g1).sum(1) / self.area
        rx = -(self.len * (g2 * n1 - g3 * n2)).sum(1) / self.area
        ry = -(self.len * (g2 * n2 + g3 * n1)).sum(1) / self.area
        # semi-implicit friction (Eq 33-37)
        qq = hu * hu + hv * hv
        on = (h > H_DRY) & (man > 0) & (qq > 0)
        hs, q = _or(on, h), torch.sqrt(_or(on, qq))
        c = G * man * man * hs ** (-7.0 / 3.0)
        dh = dt * rh
        pull = c * q * (dt - (7.0 / 6.0) * dt * dh / hs)
        bx, by = dt * rx - pull * hu, dt * ry - pull * hv
        a = 0.5 * dt * c
        one = 1.0 + a * q
        along = (bx * hu + by * hv) * a / (q * (one + a * q))
        none = torch.zeros_like(h)
        dx = torch.where(on, (bx - along * hu) / one, dt * rx)
        dy = torch.where(on, (by - along * hv) / one, dt * ry)
        h, hu, hv = h + dh, hu + dx, hv + dy
        dry = h <= H_DRY
        return torch.where(h < 0, none, h), torch.where(dry, none, hu), torch.where(dry, none, hv)


def _advance(s, h, hu, hv, steps):
    t = 0.0
    for _ in range(steps):
        dt = s.dt(h, hu, hv)
        h, hu, hv = s.step(h, hu, hv, s.z, s.man, dt)
        t = t + dt
    return h, hu, hv, float(t)


def exact(case, seed):
    with torch.no_grad():
        if case["kind"] == "riemann":
            return list(_flux(*(x.double() for x in _flux_inputs(case, seed)), hll=case["hll"]))
        if case["kind"] == "ensemble":
            done = []
            for k, args in enumerate(_members(case)):
                start = _state(args, case["f32"], 1000 * seed + k, h_right=1.0)
                done.append(_advance(_Scheme(args), *(x.double() for x in start), case["steps"]))
            return dict(state=[torch.cat([d[j] for d in done]) for j in range(3)], t=np.array([d[3] for d in done]))
        s = _Scheme(_mesh_args(case), bool(case.get("hll", False)))
        h, hu, hv = (x.double() for x in _start_of(case, seed))
        if case["kind"] != "adjoint":
            h, hu, hv, t = _advance(s, h, hu, hv, case["steps"])
            out = dict(state=(h, hu, hv), t=t)
            if case["kind"] == "steady":
                g1, _, _, _ = s.fluxes(h, hu, hv, s.z)
                through = (s.len * g1)[~s.inner]
                rates = torch.zeros(s.groups, dtype=torch.float64, device=h.device)
                out["volume"] = float((s.area * h).sum())
                out["discharge"] = rates.index_add_(0, s.group[~s.inner], through).cpu().numpy()
            return out
    # the gradient with the step sizes held, by autograd over the whole run
    at, target = _observed(case, seed, h)
    z, man = s.z.clone().requires_grad_(), s.man.clone().requires_grad_()
    dts = []
    for _ in range(case["steps"]):
        with torch.no_grad():
            dts.append(s.dt(h, hu, hv))
        h, hu, hv = s.step(h, hu, hv, z, man, dts[-1])
    off = h[torch.from_numpy(at).to(h.device).long()] - torch.from_numpy(target).to(h.device)
    loss = (off * off).sum()
    gm, gz = torch.autograd.grad(loss, [man, z])
    return dict(loss=float(loss.detach()), grad_manning=gm, grad_bathy=gz,
                dts=np.array([float(d) for d in dts]), state=(h.detach(), hu.detach(), hv.detach()))
