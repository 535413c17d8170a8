"""Cases that stand for what a program has this library do, and the inputs, work and 64-bit results of each.

Meshes are periodic: Voronoi tessellations of jittered lattices (a moving-mesh code's cells, 15.4 faces each),
Cartesian grids (6 faces) and staggered grids (14 faces).  States are those of a box that sources have been
ionising for some time, or the neutral gas that a run begins from.
"""
import functools
import itertools
import math
import types

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2404_17630_gb300 import RT, autograd, make_config, rt as rtb

KPC, C_LIGHT, EV = 3.0856775814913673e21, 2.99792458e10, 1.602176634e-12
SIGMA = [[3.0e-18, 0.0, 0.0], [5.7e-19, 4.5e-18, 0.0], [7.9e-20, 1.1e-18, 1.1e-18]]
EPS = [[5.3 * EV, 0.0, 0.0], [21.5 * EV, 10.5 * EV, 0.0], [52.1 * EV, 41.1 * EV, 11.3 * EV]]
SPLIT = np.array([1e50, 5e48, 3e48]) / 1.08e50
Y_HE = 0.24 / (4 * 0.76)
FIELDS = rtb.RT_FIELD_N | rtb.RT_FIELD_F | rtb.RT_FIELD_X | rtb.RT_FIELD_T
DEV = "cuda"


def listed():
    return [
        # the smallest call: a thousand cells, a few subcycles; launches and transfers are most of it
        dict(name="step_tiny", kind="step", mesh="voronoi", n=10, precision="mixed", n_sub=4, bins=3, gather_sum=1,
             splitting=0, c=0.01, state="evolved", host=False),
        # a uniform grid in full precision, whose program keeps its state on the host between RT steps
        dict(name="step_grid_fp64_host", kind="step", mesh="grid", n=32, precision="fp64", n_sub=20, bins=3,
             gather_sum=0, splitting=0, c=0.01, state="evolved", host=True),
        # the common production step: 2e5 cells, mixed precision, many subcycles
        dict(name="step_mixed", kind="step", mesh="voronoi", n=56, precision="mixed", n_sub=50, bins=3, gather_sum=1,
             splitting=0, c=0.01, state="evolved", host=False),
        # the same box in full precision
        dict(name="step_fp64", kind="step", mesh="voronoi", n=63, precision="fp64", n_sub=4, bins=3, gather_sum=0,
             splitting=0, c=0.01, state="evolved", host=False),
        # a reionisation box of two million cells
        dict(name="step_box", kind="step", mesh="voronoi", n=128, precision="mixed", n_sub=5, bins=3, gather_sum=1,
             splitting=0, c=0.2, state="evolved", host=False),
        # the first step of an expanding HII region: cold neutral gas, stiff chemistry around the source; fluxes
        # summed in 64 bits (the default of the mixed precision)
        dict(name="first_step_hii", kind="step", mesh="staggered", n=24, precision="mixed", n_sub=8, bins=3,
             gather_sum=0, splitting=0, c=1e-3, state="neutral", host=False),
        # cells on a four-level time-step hierarchy: a whole cycle of steps with the levels' masks
        dict(name="hierarchy", kind="levels", mesh="voronoi", n=49, precision="mixed", n_sub=5, bins=3, gather_sum=1,
             splitting=0, c=0.01, state="evolved", host=False),
        # a moving mesh: every RT step comes with a new tessellation, made on the host, and a context of its own
        dict(name="new_mesh", kind="remesh", mesh="voronoi", n=40, precision="mixed", n_sub=5, bins=3, gather_sum=0,
             splitting=1, c=0.01, state="evolved", host=False),
        # the photon-transport test: one bin, no chemistry, Heun's method, in full precision
        dict(name="transport_wave", kind="transport", mesh="grid", n=64, precision="fp64", n_sub=2, bins=1,
             time_order=2),
        # the chemistry alone, as an operator-split program calls it
        dict(name="chemistry", kind="chemistry", mesh="voronoi", n=60, precision="mixed", bins=3),
        # gradients for a caller that owns all device memory
        dict(name="gradients", kind="gradients", mesh="voronoi", n=45, bins=3, limiter=1),
        # gradients of the ionised mass in the source rates and densities through a checkpointed step
        dict(name="adjoint", kind="adjoint", mesh="voronoi", n=42, precision="fp64", n_sub=6, bins=3, every=3,
             chem_mode=2),
    ]


def draw(rng):
    """One more case of the same ranges (n, then the smallest multiple of a tile above it)."""
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        while not any(n % m == 0 for m in range(5, 12)):
            n += 1
        return n
    kind = rng.choice(["step"] * 5 + ["levels", "remesh", "transport", "chemistry", "gradients", "adjoint"])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    mesh = rng.choice(["voronoi", "voronoi", "voronoi", "grid", "staggered"])
    bins = rng.choice([3, 3, 3, 2, 1])
    if kind == "transport":
        return dict(kind=kind, mesh=mesh, n=size(10, 60), precision=prec, n_sub=rng.randint(1, 4), bins=bins,
                    time_order=rng.randint(1, 2))
    if kind == "chemistry":
        return dict(kind=kind, mesh="voronoi", n=size(10, 70), precision=prec, bins=bins)
    if kind == "gradients":
        return dict(kind=kind, mesh=mesh, n=size(10, 49), bins=bins, limiter=rng.choice([1, 1, 0]))
    if kind == "adjoint":
        return dict(kind=kind, mesh="voronoi", n=size(10, 40), precision="fp64", n_sub=rng.randint(2, 6), bins=bins,
                    every=rng.randint(1, 4), chem_mode=rng.choice([2, 2, 1]))
    if kind == "levels":
        mesh, prec = "voronoi", "mixed"
    n = size(10, 110 if prec == "mixed" and mesh != "staggered" and kind == "step" else 45)
    most = max(2, min(40, int((3e7 if prec == "mixed" else 1.2e6) / n ** 3)))
    return dict(kind=kind, mesh=mesh, n=n, precision=prec, n_sub=rng.randint(1, most), bins=bins,
                gather_sum=rng.choice([1, 1, 0]), splitting=rng.choice([0, 0, 1]), c=rng.choice([0.01, 0.01, 0.2]),
                state="evolved", host=kind == "step" and n <= 45 and rng.random() < 0.3)


# ---------------------------------------------------------------------------
# meshes
# ---------------------------------------------------------------------------

def _edges(cells, ids, lat, d, area, fc, L):
    """Mesh from both directions of every face: cell ids[0] -> ids[1]; each pair is kept once, by its smaller id."""
    keep = ids[0] < ids[1]
    order = torch.argsort(ids[0][keep].to(torch.int32), stable=True)
    l, r, d, area, fc = (a[keep][order] for a in (ids[0], ids[1], d, area, fc))
    nrm = d / d.norm(dim=1, keepdim=True)
    fc = torch.remainder(fc, L)
    fc = torch.where(fc >= L, torch.zeros_like(fc), fc)
    vol, cen = cells
    return types.SimpleNamespace(
        n_cells=vol.numel(), n_faces=l.numel(), box=float(L), lattice=lat, volume=vol.contiguous(),
        left=l.to(torch.int32).contiguous(), right=r.to(torch.int32).contiguous(), area=area.contiguous(),
        **{k: cen[:, i].contiguous() for i, k in enumerate(("cx", "cy", "cz"))},
        **{k: nrm[:, i].contiguous() for i, k in enumerate(("nx", "ny", "nz"))},
        **{k: fc[:, i].contiguous() for i, k in enumerate(("fx", "fy", "fz"))})


def _lattice(n):
    i = torch.arange(n ** 3, device=DEV)
    return torch.stack([i % n, i // n % n, i // (n * n)], 1)


def _id(p, n):
    p = p % n
    return p[..., 0] + n * (p[..., 1] + n * p[..., 2])


@functools.lru_cache(maxsize=16)
def _tile(m, seed):
    """Periodic Voronoi tessellation of an m^3 lattice (spacing 1) with jitter 0.3: vertices are the points of
    three bisector planes that lie inside every other one; faces are their polygons."""
    rng = np.random.default_rng(seed)
    lat = _lattice(m).cpu().numpy()
    gen = lat + 0.5 + rng.uniform(-0.3, 0.3, (m ** 3, 3))
    reach = np.array([o for o in itertools.product(range(-3, 4), repeat=3) if any(o)])
    nb = lat[:, None] + reach[None]
    w = nb % m
    d = gen[w[..., 0] + m * (w[..., 1] + m * w[..., 2])] + (nb - w) - gen[:, None]
    K = 48
    near = np.argsort((d ** 2).sum(-1), axis=1, kind="stable")[:, :K + 1]
    d = np.take_along_axis(d, near[..., None], 1)
    edge, d, near = (d[:, K] ** 2).sum(-1), d[:, :K], near[:, :K]
    P = torch.as_tensor(d, device=DEV)
    h = 0.5 * (P * P).sum(-1)
    tri = torch.as_tensor(list(itertools.combinations(range(K), 3)), device=DEV)
    cell, three, vert = [], [], []
    for c in range(m ** 3):
        a, b, e = (P[c][tri[:, q]] for q in range(3))
        bc, ca, ab = torch.linalg.cross(b, e), torch.linalg.cross(e, a), torch.linalg.cross(a, b)
        det = (a * bc).sum(1)
        v = (h[c][tri[:, 0], None] * bc + h[c][tri[:, 1], None] * ca + h[c][tri[:, 2], None] * ab) / det[:, None]
        out = (v[:, 0, None] * P[c, :, 0] + v[:, 1, None] * P[c, :, 1] + v[:, 2, None] * P[c, :, 2]) > h[c] + 1e-9
        good = torch.nonzero((det.abs() > 1e-12) & ~out.any(1))[:, 0]
        cell.append(torch.full_like(good, c)); three.append(tri[good]); vert.append(v[good])
    cell, three, vert = (torch.cat(a).cpu().numpy() for a in (cell, three, vert))
    assert (4 * (vert ** 2).sum(1) < edge[cell]).all(), "a neighbour may be missing"
    # the polygon of each (cell, candidate): its vertices by their angle about their mean
    key = (cell[:, None] * K + three).ravel()
    pts = np.repeat(vert, 3, axis=0)
    order = np.argsort(key, kind="stable")
    key, pts = key[order], pts[order]
    face, first, count = np.unique(key, return_index=True, return_counts=True)
    of = np.repeat(np.arange(face.size), count)
    fd = d[face // K, face % K]
    mean = np.add.reduceat(pts, first, axis=0) / count[:, None]
    nrm = fd / np.linalg.norm(fd, axis=1, keepdims=True)
    u = np.cross(nrm, np.eye(3)[np.argmin(np.abs(nrm), axis=1)])
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    q = pts - mean[of]
    ang = np.arctan2((q * np.cross(nrm, u)[of]).sum(1), (q * u[of]).sum(1))
    order = np.lexsort((ang, of))
    pts = pts[order]
    nxt = np.arange(of.size) + 1
    nxt[first + count - 1] = first
    a3 = 0.5 * np.linalg.norm(np.cross(pts - mean[of], pts[nxt] - mean[of]), axis=1)
    area = np.add.reduceat(a3, first)
    fc = np.add.reduceat(a3[:, None] * (pts + pts[nxt] + mean[of]) / 3, first, axis=0) / area[:, None]
    big = area > 1e-11
    face, fd, area, fc = face[big], fd[big], area[big], fc[big]
    own = face // K
    at = np.searchsorted(own, np.arange(m ** 3))
    pyr = area * np.linalg.norm(fd, axis=1) / 6
    vol = np.add.reduceat(pyr, at)
    cen = gen + np.add.reduceat(pyr[:, None] * 0.75 * fc, at, axis=0) / vol[:, None]
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=DEV)  # noqa: E731
    off = reach[near[own, face % K]]
    return t(vol), t(cen), t(own), t(off), t(fd), t(area), t(fc + gen[own])


def _voronoi(n, L, seed):
    """The n^3 box as (n / m)^3 copies of an m^3 tile, in lattice order."""
    m = max(k for k in range(5, 12) if n % k == 0)
    vol, cen, own, off, d, area, fc = _tile(m, seed)
    h, lat, tl = L / n, _lattice(n), _lattice(m)
    home = _id(lat % m, m)
    base = (lat // m * m).double()
    shift = _lattice(n // m) * m
    ids = torch.stack([_id(tl[own] + shift[:, None], n), _id(tl[own] + off + shift[:, None], n)]).reshape(2, -1)
    rep = lambda a: a.expand(shift.shape[0], *a.shape).reshape(-1, *a.shape[1:])  # noqa: E731
    fcs = (fc + shift[:, None].double()).reshape(-1, 3)
    cen = torch.remainder((cen[home] + base) * h, L)
    return _edges((vol[home] * h ** 3, cen), ids, lat, rep(d) * h, rep(area) * h * h, fcs * h, L)


def _mesh(kind, n, L, seed):
    if kind == "voronoi":
        return _voronoi(n, L, seed)
    lat, h = _lattice(n), L / n
    one = torch.ones(n ** 3, dtype=torch.float64, device=DEV)
    if kind == "grid":
        ids, d, fc = [], [], []
        for ax, s in itertools.product(range(3), (-1, 1)):
            o = torch.zeros(3, dtype=torch.int64, device=DEV)
            o[ax] = s
            ids.append(torch.stack([_id(lat, n), _id(lat + o, n)]))
            d.append((o.double() * h).expand(n ** 3, 3))
            fc.append((lat + 0.5 + 0.5 * o.double()) * h)
        area = one.repeat(6) * h * h
        return _edges((one * h ** 3, (lat.double() + 0.5) * h), torch.cat(ids, 1), lat, torch.cat(d), area, torch.cat(fc), L)
    # staggered: corners and body centres; truncated octahedra with 8 hexagons and 6 squares
    pos = torch.cat([lat.double(), lat.double() + 0.5])
    cid = _id(lat, n)
    ids, d, area = [], [], []
    for s in itertools.product((-1, 1), repeat=3):
        o = torch.tensor([(v - 1) // 2 for v in s], device=DEV)
        other = n ** 3 + _id(lat + o, n)
        ids += [torch.stack([cid, other]), torch.stack([other, cid])]
        v = torch.tensor(s, dtype=torch.float64, device=DEV) * 0.5
        d += [v.expand(n ** 3, 3), -v.expand(n ** 3, 3)]
        area += [one * (3 * 3 ** 0.5 / 16)] * 2
    for lot, ax, s in itertools.product((0, 1), range(3), (-1, 1)):
        o = torch.zeros(3, dtype=torch.int64, device=DEV)
        o[ax] = s
        ids.append(torch.stack([cid, _id(lat + o, n)]) + lot * n ** 3)
        d.append(o.double().expand(n ** 3, 3))
        area.append(one / 8)
    ids, d = torch.cat(ids, 1), torch.cat(d)
    fc = (pos[ids[0]] + 0.5 * d) * h
    return _edges((one.repeat(2) * 0.5 * h ** 3, pos * h), ids, torch.cat([lat, lat]), d * h, torch.cat(area) * h * h, fc, L)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _config(case):
    B = case["bins"]
    hii = case["mesh"] == "staggered"
    return dict(n_bins=B, c_red=case.get("c", 0.01) * C_LIGHT, unit_length_cm=KPC,
                box=1.6 if hii else 3580.0 * case["n"] / 128 if case.get("c") == 0.2 else 10.0, cfl=0.3,
                chem_mode={"transport": 0}.get(case["kind"], case.get("chem_mode", 2)), chem_flags=15,
                limiter=case.get("limiter", 1), lim_eps=1e-5, order=2, f_s=0.05, f_max=0.1, x_floor=1e-4,
                max_substeps=10000, y_he=Y_HE, sigma=SIGMA[:B], eps=EPS[:B], gather_sum=case.get("gather_sum", 0),
                splitting=case.get("splitting", 0), time_order=case.get("time_order", 1))


def _density(case, mesh, gen):
    n, C = case["n"], mesh.n_cells
    if case["mesh"] == "staggered":     # a core and an r^-2 envelope
        x = torch.stack([mesh.cx, mesh.cy, mesh.cz], 1) - 0.5 * mesh.box
        x = x - mesh.box * torch.round(x / mesh.box)
        return 3.2 * (0.0915 / x.norm(dim=1).clamp(min=0.0915)) ** 2
    z = torch.randn(n, n, n, generator=gen, device=DEV, dtype=torch.float64)
    if case.get("c") != 0.2:
        return 1e-3 * torch.exp(z.reshape(-1)[:C])
    k = torch.fft.fftfreq(n, device=DEV, dtype=torch.float64)      # exp of a Gaussian field, P(k) ~ k^-2
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :n // 2 + 1] ** 2
    g = torch.fft.irfftn(torch.fft.rfftn(z) * torch.where(k2 > 0, k2.clamp(min=1e-30) ** -0.5, 0.0), s=(n, n, n))
    rho = torch.exp(1.5 * g / g.std())
    return (rho * (2e-4 / rho.mean())).reshape(-1)


def _inputs(case, seed):
    """Mesh, gas, radiation and sources of one case, made from the seed (a mesh that stays is the same for all)."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    cfg = _config(case)
    mesh = _mesh(case["mesh"], case["n"], cfg["box"], seed % 1000 if case["kind"] == "remesh" else 0)
    C, B, h = mesh.n_cells, case["bins"], cfg["box"] / case["n"]
    rnd = lambda *s: torch.rand(*s, generator=gen, device=DEV, dtype=torch.float64)  # noqa: E731
    st = types.SimpleNamespace(mesh=mesh, cfg=cfg, nH=_density(case, mesh, gen).contiguous())
    pos = torch.stack([mesh.cx, mesh.cy, mesh.cz], 1)
    if case["kind"] in ("transport", "gradients"):
        # waves over the box in every bin, with the cells' own scatter in the gradients' case
        k = 2 * math.pi / mesh.box
        ph = rnd(B, 3) * 6.28
        N = 1e-3 * (1 + 0.5 * torch.cos(k * pos[:, 0] + ph[:, :1]) * torch.cos(k * pos[:, 1] + ph[:, 1:2]))
        if case["kind"] == "gradients":
            N = N * torch.exp(0.3 * torch.randn(B, C, generator=gen, device=DEV, dtype=torch.float64))
        u = torch.stack([torch.cos(k * pos[:, 2] + ph[b, 2]) * 0.7 for b in range(B)])
        f = torch.stack([u, 0.3 * torch.sin(k * pos[:, 0]) * torch.ones_like(u), 0.2 - 0.1 * u], 1) * N[:, None]
        x5 = torch.zeros(5, C, dtype=torch.float64, device=DEV)
        x5[0], x5[2] = 1, 1
        st.N, st.fr, st.x5, st.T = N.contiguous(), f.contiguous(), x5, torch.full((C,), 1e4, device=DEV).double()
        st.cells, st.Q = np.zeros(0, np.int64), np.zeros((0, B))
        return st
    if case["mesh"] == "staggered":
        x = pos - 0.5 * mesh.box
        x = (x - mesh.box * torch.round(x / mesh.box)).norm(dim=1)
        cells = torch.argsort(x, stable=True)[:max(1, int((x < 0.05).sum()))]
        Qt = 1.08e50 * mesh.volume[cells] / mesh.volume[cells].sum() * (0.5 + rnd(1))
        centre, front, Qc = pos[torch.argsort(x, stable=True)[:1]], torch.full((1,), 0.3 * mesh.box).to(DEV), Qt.sum()[None]
    else:
        S = 16 if case.get("c") != 0.2 else min(512, max(16, C // 4096))
        cells = torch.topk(st.nH, S)[1] if case.get("c") == 0.2 else torch.randperm(C, generator=gen, device=DEV)[:S]
        Qt = 10 ** (49 + 2 * rnd(S))
        centre, front, Qc = pos[cells], h * (2 + 0.3 * case["n"] * (Qt / Qt.max()) ** (1 / 3) * rnd(S)), Qt
    st.cells = cells.cpu().numpy().astype(np.int64)
    st.Q = Qt.cpu().numpy()[:, None] * SPLIT[None, :B] / SPLIT[:B].sum()
    N = torch.full((B, C), 1e-16, dtype=torch.float64, device=DEV) * (1 + 0.5 * rnd(B, 1))
    f = torch.zeros(B, 3, C, dtype=torch.float64, device=DEV)
    if case.get("state", "evolved") == "neutral":
        x = torch.full((C,), 1e-6, dtype=torch.float64, device=DEV)
        st.x5 = torch.stack([1 - x, x, 1 - x, 0.9 * x, 0.1 * x]).contiguous()
        st.T = torch.full((C,), 100.0, dtype=torch.float64, device=DEV) * (1 + 0.1 * rnd(C))
    else:
        # every source's light, thinning as r^-2 and stopped at its front, over the background of a box whose fronts
        # have met (the large boxes, and those of the adjoint, are still neutral between theirs); gas in ionisation
        # balance with it
        sp = torch.as_tensor(SPLIT[:B] / SPLIT[:B].sum(), device=DEV)
        if case.get("c") != 0.2 and case["kind"] != "adjoint":
            wave = 1 + 0.1 * torch.sin(2 * math.pi / mesh.box * pos[:, 0] + 6.28 * rnd(1))
            N += 5e-3 * (0.5 + rnd(1)) * sp[:, None] * wave
        for s in range(centre.shape[0]):
            x = pos - centre[s]
            x = x - mesh.box * torch.round(x / mesh.box)
            r = x.norm(dim=1)
            rc = r.clamp(min=0.6 * h)
            lum = Qc[s] / (4 * math.pi * cfg["c_red"] * (rc * KPC) ** 2) * torch.exp(-(r / front[s]) ** 4 * 5)
            N += sp[:, None] * lum
            f += (sp[:, None] * lum)[:, None] * (0.95 * x / (r[:, None] + 0.5 * h)).T
        sig = torch.tensor(SIGMA[:B], dtype=torch.float64, device=DEV)
        G = cfg["c_red"] * (sig.T @ N)
        q = G[0] / (2.6e-13 * st.nH)
        st.T = (8e3 + 1.2e4 * q / (1 + q)) * (0.97 + 0.06 * rnd(C))
        t = (st.T / 1e4) ** -0.77
        q = q / t
        ion = 2 * q / (q + torch.sqrt(q * q + 4 * q))        # ion^2 = q (1 - ion)
        neu = ion * ion / q
        ne = st.nH * ion * 1.1
        r1, r2 = G[1] / (2.6e-13 * t * ne), G[2] / (1.55e-12 * t * ne)
        y1, y2, y3 = 1 / (1 + r1 * (1 + r2)), r1 / (1 + r1 * (1 + r2)), r1 * r2 / (1 + r1 * (1 + r2))
        st.x5 = torch.stack([neu, 1 - neu, y1, y2, y3]).contiguous()
    st.N, st.fr, st.T = N.contiguous(), f.contiguous(), st.T.contiguous()
    return st


def _masks(case, C, lat):
    """Active sets of one cycle: levels of 10, 20, 30 and 40 % by a smooth field, level k active in steps that 2^k
    divides."""
    k = 2 * math.pi / case["n"]
    ph = torch.arange(6, device=DEV) * 1.3
    p = lat.double() * k
    f = sum(torch.sin((1 + i % 3) * p[:, i % 3] + ph[i]) * torch.cos(p[:, (i + 1) % 3] * (1 + i // 3)) for i in range(6))
    order = torch.argsort(f, stable=True)
    level = torch.empty(C, dtype=torch.int64, device=DEV)
    cut = torch.tensor([0.1, 0.3, 0.6], device=DEV) * C
    level[order] = torch.searchsorted(cut, torch.arange(C, device=DEV, dtype=cut.dtype), right=True)
    level = level.cpu().numpy()
    return [(level <= max(k for k in range(4) if s % 2 ** k == 0)).astype(np.uint8) for s in range(8)]


def prepare(case, seed):
    st = _inputs(case, seed)
    cfg, mesh, B = st.cfg, st.mesh, case["bins"]
    st.case, st.C = case, mesh.n_cells
    st.F = (st.fr * cfg["c_red"]).contiguous()
    if case["kind"] == "gradients":
        # the caller's own arrays: per-cell face lists, ascending face ids
        F, C = mesh.n_faces, mesh.n_cells
        cell = torch.cat([mesh.left, mesh.right]).long()
        entry = torch.cat([torch.arange(F, device=DEV) * 2, torch.arange(F, device=DEV) * 2 + 1])
        order = torch.argsort(cell * (2 * F) + entry)
        st.csr = entry[order].to(torch.int32).contiguous()
        st.off = torch.zeros(C + 1, dtype=torch.int32, device=DEV)
        st.off[1:] = torch.bincount(cell, minlength=C).cumsum(0).to(torch.int32)
        ptr = lambda k: getattr(mesh, k).data_ptr()  # noqa: E731
        st.rc = rtb.rt_cells(C, *[ptr(k) for k in ("volume", "cx", "cy", "cz")])
        st.rf = rtb.rt_faces(F, *[ptr(k) for k in ("left", "right", "area", "nx", "ny", "nz", "fx", "fy", "fz")])
        return st
    st.made = make_config(precision=case["precision"], **cfg)
    st.rt = RT(st.made, mesh, stream=torch.cuda.current_stream())
    if case["kind"] == "remesh":
        st.host = types.SimpleNamespace(n_cells=mesh.n_cells, n_faces=mesh.n_faces, **{
            k: getattr(mesh, k).cpu().numpy()
            for k in ("volume", "cx", "cy", "cz", "left", "right", "area", "nx", "ny", "nz", "fx", "fy", "fz")})
    st.rt.set_sources(st.cells, st.Q)
    st.dt = st.rt.max_dt() * case.get("n_sub", 1) * 0.9
    if case["kind"] == "levels":
        st.masks = _masks(case, st.C, mesh.lattice)
    if case.get("host"):
        pin = lambda a: a.cpu().pin_memory()  # noqa: E731
        st.N, st.F, st.nH, st.x5, st.T = (pin(a) for a in (st.N, st.F, st.nH, st.x5, st.T))
    if case["kind"] == "adjoint":
        st.mass = st.nH * mesh.volume / (st.nH * mesh.volume).sum()
        st.Qd = torch.as_tensor(st.Q, device=DEV).requires_grad_()
        st.nHd = st.nH.clone().requires_grad_()
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _fields(st, host=False):
    """The fields after a step; the mixed precision's, which carry 32-bit accuracy, are kept in 32 bits."""
    C, B = st.C, st.case["bins"]
    new = lambda *s: torch.empty(*s, dtype=torch.float64, device="cpu" if host else DEV)  # noqa: E731
    out = [new(B, C), new(B, 3, C), new(5, C), new(C)]
    rtb.rt_get_fields(st.rt.ctx, FIELDS, out)
    if st.case["precision"] == "mixed":
        out = [o.float() for o in out]
    return dict(zip(("N", "F", "x5", "T"), out))


def run(st):
    case, rt = st.case, getattr(st, "rt", None)
    kind = case["kind"]
    if kind == "gradients":
        G = torch.empty(st.C, case["bins"], 4, 3, dtype=torch.float64, device=DEV)
        bad = torch.empty(1, dtype=torch.int32, device=DEV)
        rtb.rt_gradients_noalloc(st.rc, st.rf, st.off, st.csr, case["bins"], 2, case["limiter"], 1e-5, st.mesh.box,
                                 st.N, st.fr, G, bad, torch.cuda.current_stream())
        return dict(G=G, bad=bad)
    if kind == "adjoint":
        st.Qd.grad = st.nHd.grad = None
        N, F, x5, T = autograd.rt_step_autograd(rt, st.cells, st.Qd, st.nHd, st.N, st.F, st.x5, st.T, st.dt,
                                                case["n_sub"], case["every"])
        (st.mass * x5[1]).sum().backward()
        return dict(N=N.detach(), x5=x5.detach(), T=T.detach(), dQ=st.Qd.grad, dnH=st.nHd.grad)
    if kind == "remesh":
        st.rt = rt = RT(st.made, st.host, stream=torch.cuda.current_stream())
        rt.set_sources(st.cells, st.Q)
    rt.set_radiation(st.N, st.F)
    rt.set_gas(st.nH, st.x5, st.T)
    if kind == "levels":
        for m in st.masks:
            rt.set_active(m)
            rt.step(st.dt, case["n_sub"])
    elif kind == "transport":
        for _ in range(case["n_sub"]):
            rt.transport(st.dt / case["n_sub"])
    elif kind == "chemistry":
        rt.thermochemistry(st.dt)
    else:
        rt.step(st.dt, case["n_sub"])
    return _fields(st, case.get("host", False))


def work(case):
    n, B, w = case["n"], case["bins"], 8 if case.get("precision", "fp64") == "fp64" else 4
    C, fbar = {"voronoi": (n ** 3, 7.7), "grid": (n ** 3, 3), "staggered": (2 * n ** 3, 7)}[case["mesh"]]
    F = fbar * C
    kind = case["kind"]
    # per subcycle: the mesh (pair of ids, normal, area, both offsets, weight; volume, inverse matrix) and the state
    # once in, the state once out; operations of the gradients, the face states and fluxes, the update, an attempt
    mesh = F * (8 + 13 * w) + C * (8 + 6 * w)
    rad, gas = C * B * (8 + 3 * w), C * 56
    grad, face, upd, chem = C * B * (fbar * 2 * 53 + 90), F * B * 130, C * B * (fbar * 8 + 8), C * 250
    ends = C * (8 * (2 * 4 * B + 2 * 6 + 1))
    if kind == "gradients":
        return dict(bytes=F * (8 + 7 * 8) + C * (8 * 3 + 8 + 8 * fbar) + C * B * 16 * 8, flops=grad + C * fbar * 2 * 40)
    if kind == "chemistry":
        return dict(bytes=ends + 2 * (C * B * 8 + gas), flops=chem)
    sub = case["n_sub"] * (2 if case.get("time_order") == 2 else 1)
    move = sub * (mesh + 2 * rad)
    do = sub * (grad + face + upd)
    if kind != "transport":
        move += case["n_sub"] * 2 * gas
        do += case["n_sub"] * chem * (1 + case.get("splitting", 0))
    if kind == "adjoint":
        move, do = 3 * move, 4 * do
    if kind == "levels":
        # 1.0, 0.1, 0.3, 0.1, 0.6, 0.1, 0.3, 0.1 of the cells in the cycle's steps
        move, do = 2.6 * move, 2.6 * do
    if kind == "remesh":
        ends += F * (8 + 7 * 8) + C * 32
    return dict(bytes=ends + move, flops=do)


# ---------------------------------------------------------------------------
# the same in 64 bits, from the method's definitions
# ---------------------------------------------------------------------------

def _geometry(mesh):
    L, R = mesh.left.long(), mesh.right.long()
    cen = torch.stack([mesh.cx, mesh.cy, mesh.cz], 1)
    fc = torch.stack([mesh.fx, mesh.fy, mesh.fz], 1)
    near = lambda d: d - mesh.box * torch.round(d / mesh.box)  # noqa: E731
    d = near(cen[R] - cen[L])
    w = mesh.area[:, None] * d / (d * d).sum(1, keepdim=True)
    m = mesh.area[:, None, None] * d[:, :, None] * d[:, None, :] / (d * d).sum(1)[:, None, None]
    M = torch.zeros(mesh.n_cells, 3, 3, dtype=torch.float64, device=DEV).index_add(0, L, m).index_add(0, R, m)
    return types.SimpleNamespace(L=L, R=R, xL=near(fc - cen[L]), xR=near(fc - cen[R]), w=w, Minv=torch.linalg.inv(M),
                                 n=torch.stack([mesh.nx, mesh.ny, mesh.nz], 1), A=mesh.area, V=mesh.volume,
                                 C=mesh.n_cells)


def _gradients(g, U, limiter, eps):
    """Limited least-squares gradients [C, B, 4, 3] of U [C, B, 4]."""
    UL, UR = U[g.L], U[g.R]
    t = (UR - UL)[..., None] * g.w[:, None, None, :]
    r = torch.zeros(*U.shape, 3, dtype=U.dtype, device=DEV).index_add(0, g.L, t).index_add(0, g.R, t)
    G = (r[..., None, :] * g.Minv[:, None, None]).sum(-1)
    if not limiter:
        return G
    ix = lambda i: i[:, None, None].expand_as(UL)  # noqa: E731
    hi = U.scatter_reduce(0, ix(g.L), UR, "amax").scatter_reduce(0, ix(g.R), UL, "amax")
    lo = U.scatter_reduce(0, ix(g.L), UR, "amin").scatter_reduce(0, ix(g.R), UL, "amin")
    up, dn = hi - U, lo - U
    psi = torch.ones_like(U)
    for i, x in ((g.L, g.xL), (g.R, g.xR)):
        d = (G[i] * x[:, None, None, :]).sum(-1)
        tall = d * d > eps * eps * (G[i] ** 2).sum(-1) * (x * x).sum(1)[:, None, None]
        lim = torch.where(d > 0, up[i], dn[i]) / torch.where(tall, d, torch.ones_like(d))
        psi = psi.scatter_reduce(0, ix(i), torch.where(tall, lim, torch.ones_like(lim)), "amin")
    return G * psi[..., None]


def _face_flux(g, U, G):
    """(A Phi_N, A Phi_F) / c of every face [F, B, 4]."""
    v, P = [], []
    n = g.n[:, None, :]
    for i, x in ((g.L, g.xL), (g.R, g.xR)):
        s = U[i] + (G[i] * x[:, None, None, :]).sum(-1)
        N, f = s[..., 0].clamp(min=0), s[..., 1:]
        f2 = (f * f).sum(-1)
        fl = torch.where(f2 > 0, f2, torch.ones_like(f2)).sqrt()
        f = f * torch.where(f2 > N * N, N / fl, torch.ones_like(N))[..., None]
        f2 = (f * f).sum(-1)
        some = (N > 0) & (f2 > 0)
        fl = torch.where(some, f2, torch.ones_like(f2)).sqrt()
        red = torch.where(some, fl / torch.where(some, N, torch.ones_like(N)), torch.zeros_like(N)).clamp(max=1)
        chi = (3 + 4 * red ** 2) / (5 + 2 * (4 - 3 * red ** 2).sqrt())
        u = torch.where(some[..., None], f / fl[..., None], torch.zeros_like(f))
        v.append(torch.cat([N[..., None], f], -1))
        P.append(N[..., None] * (0.5 * (1 - chi)[..., None] * n + 0.5 * ((3 * chi - 1) * (u * n).sum(-1))[..., None] * u))
    fn = 0.5 * ((v[0] + v[1])[..., 1:] * n).sum(-1)
    phi = torch.cat([fn[..., None], 0.5 * (P[0] + P[1])], -1) - 0.5 * (v[1] - v[0])
    return g.A[:, None, None] * phi


def _transport(g, cfg, U, dt, on=None):
    def euler(U):
        G = _gradients(g, U, cfg["limiter"], cfg["lim_eps"])
        phi = _face_flux(g, U, G)
        if on is not None:
            phi = phi * (on[g.L] | on[g.R])[:, None, None]
        div = torch.zeros_like(U).index_add(0, g.L, phi).index_add(0, g.R, -phi)
        return U - (cfg["c_red"] * dt / KPC / g.V)[:, None, None] * div
    if cfg["time_order"] == 1:
        return euler(U)
    return 0.5 * U + 0.5 * euler(euler(U))


def _rates(T):
    """Recombination, collisional ionisation (cm^3/s) and cooling coefficients per species (erg cm^3/s)."""
    lam = lambda t: 2 * t / T  # noqa: E731
    hg = lambda l: 2.753e-14 * l ** 1.5 / (1 + (l / 2.740) ** 0.407) ** 2.242  # noqa: E731
    sT, tf = T.sqrt(), 1 / (1 + (T / 1e5).sqrt())
    die = T ** -1.5 * torch.exp(-470000 / T) * (1 + 0.3 * torch.exp(-94000 / T))
    e1, e2, e3 = torch.exp(-157809.1 / T), torch.exp(-285335.4 / T), torch.exp(-631515.0 / T)
    rec = [hg(lam(157807.0)), 1.26e-14 * lam(285335.0) ** 0.75 + 1.9e-3 * die, 2 * hg(lam(631515.0))]
    col = [5.85e-11 * sT * e1 * tf, 2.38e-11 * sT * e2 * tf, 5.68e-12 * sT * e3 * tf]
    t3 = (T / 1e3) ** -0.2 / (1 + (T / 1e6) ** 0.7)
    br = 1.42e-27 * (1.1 + 0.34 * torch.exp(-(5.5 - torch.log10(T)) ** 2 / 3)) * sT
    cool = [(7.5e-19 * torch.exp(-118348.0 / T) + 1.27e-21 * sT * e1) * tf, 8.7e-27 * sT * t3 + br,
            9.38e-22 * sT * e2 * tf,
            (5.54e-17 * T ** -0.397 * torch.exp(-473638.0 / T) + 4.95e-22 * sT * e3) * tf + 1.55e-26 * T ** 0.3647
            + 1.24e-13 * die + br, 3.48e-26 * sT * t3 + 4 * br]
    return rec, col, cool


def _attempt(cfg, nH, dt, N, x, T):
    """One semi-implicit attempt: N [B, c], x [5, c], T [c] -> the same after dt, the photons' factors, the measure."""
    sig, eps, c, kB = cfg["sigma"], cfg["eps"], cfg["c_red"], 1.380649e-16
    B, nHe = N.shape[0], cfg["y_he"] * nH
    (aH2, aHe2, aHe3), (bH, bHe, bHe2), cool = _rates(T)
    absorb = lambda ns, b: sum(sig[b][s] * ns[s] for s in range(3))  # noqa: E731
    ns = (nH * x[0], nHe * x[2], nHe * x[3])
    bar = [N[b] / (1 + c * dt * absorb(ns, b)) for b in range(B)]
    G = [c * sum(sig[b][s] * bar[b] for b in range(B)) for s in range(3)]
    ne = nH * x[1] + nHe * (x[3] + 2 * x[4])
    a, b = dt * (G[0] + bH * ne), dt * aH2 * ne
    h1, h2 = (x[0] * (1 + b) + b * x[1]) / (1 + a + b), (x[1] * (1 + a) + a * x[0]) / (1 + a + b)
    n1 = nH * h2 + nHe * (x[3] + 2 * x[4])
    A, Bb, Cc, D = dt * (G[1] + bHe * n1), dt * aHe2 * n1, dt * (G[2] + bHe2 * n1), dt * aHe3 * n1
    y2 = (x[3] + A * x[2] / (1 + A) + D * x[4] / (1 + D)) / (1 + Bb / (1 + A) + Cc / (1 + D))
    y1, y3 = (x[2] + Bb * y2) / (1 + A), (x[4] + Cc * y2) / (1 + D)
    xn = torch.stack([h1, h2, y1, y2, y3])
    m = (nH * h1, nHe * y1, nHe * y2)
    gone = [c * dt * bar[b] * absorb(m, b) for b in range(B)]
    heat = sum(c * dt * bar[b] * sum(eps[b][s] * sig[b][s] * m[s] for s in range(3)) for b in range(B))
    Nn = torch.stack([(N[b] - gone[b]).clamp(min=0) for b in range(B)])
    share = torch.where(N > 0, Nn / torch.where(N > 0, N, torch.ones_like(N)), torch.zeros_like(N))
    f = ((xn - x).abs() / x.abs().clamp(min=cfg["x_floor"])).amax(0)
    if cfg["chem_mode"] == 2:
        dens = (nH * x[0], nH * x[1], nHe * x[2], nHe * x[3], nHe * x[4])
        e0 = 1.5 * kB * (nH * (1 + cfg["y_he"]) + ne) * T
        e1 = e0 + heat - dt * ne * sum(k * d for k, d in zip(cool, dens))
        T = e1 / (1.5 * kB * (nH * (1 + cfg["y_he"]) + nH * h2 + nHe * (y2 + 2 * y3)))
        f = torch.maximum(f, (e1 - e0).abs() / e0.abs())
    return Nn, xn, T, share, f


def _chemistry(cfg, nH, U, x, T, dt, on=None):
    """Adaptive substeps over dt of the cells `on` (None: all); U [C, B, 4], x [5, C], T [C]."""
    idx = torch.arange(nH.numel(), device=DEV) if on is None else torch.nonzero(on)[:, 0]
    N, sc = U[..., 0].T, torch.ones_like(U[..., 0].T)
    rem = torch.full_like(T, dt)
    step = rem
    while idx.numel():
        Ni, xi, Ti, ri, di = N[:, idx], x[:, idx], T[idx], rem[idx], step[idx]
        Nn, xn, Tn, sh, f = _attempt(cfg, nH[idx], di, Ni, xi, Ti)
        ok = f <= cfg["f_max"]
        safe = torch.where(f > 0, f, torch.ones_like(f))
        ratio = torch.where(f > 0, cfg["f_s"] / safe, torch.full_like(f, 2.0))
        left = torch.where(ok, torch.where(di == ri, torch.zeros_like(ri), ri - di), ri)
        grow = di * torch.where(ok, ratio.clamp(max=2.0), ratio)
        nxt = torch.where(ok & (grow > left), left, grow)
        put = lambda full, new: full.index_copy(full.dim() - 1, idx, new)  # noqa: E731
        N, x, T = put(N, torch.where(ok, Nn, Ni)), put(x, torch.where(ok, xn, xi)), put(T, torch.where(ok, Tn, Ti))
        sc = put(sc, torch.where(ok, sc[:, idx] * sh, sc[:, idx]))
        rem, step = put(rem, left), put(step, nxt)
        idx = idx[(left > 0).detach()]
    return torch.cat([N.T[..., None], U[..., 1:] * sc.T[..., None]], -1), x, T


def exact(case, seed):
    st = _inputs(case, seed)
    cfg, mesh, kind = st.cfg, st.mesh, case["kind"]
    g = _geometry(mesh)
    C, B = g.C, case["bins"]
    U = torch.cat([st.N[:, None], st.fr], 1).permute(2, 0, 1).contiguous()      # [C, B, 4]
    if kind == "gradients":
        return dict(G=_gradients(g, U, case["limiter"], 1e-5), bad=None)
    n_sub = case.get("n_sub", 1)
    dts = cfg["cfl"] * float(mesh.volume.min()) ** (1 / 3) * KPC / cfg["c_red"] * 0.9
    cells = torch.as_tensor(st.cells, device=DEV)

    def chem(U, x, T, Q, nH, dt, on=None):
        S = torch.zeros(C, B, dtype=torch.float64, device=DEV).index_add(0, cells, Q) * dt / (g.V * KPC ** 3)[:, None]
        if on is not None:
            S = S * on[:, None]
        U = torch.cat([(U[..., 0] + S)[..., None], U[..., 1:]], -1)
        return _chemistry(cfg, nH, U, x, T, dt, on)

    def sub(U, x, T, Q, nH, on=None):
        half = 0.5 if cfg["splitting"] else 1.0
        U, x, T = chem(U, x, T, Q, nH, half * dts, on)
        U = _transport(g, cfg, U, dts, on)
        return chem(U, x, T, Q, nH, half * dts, on) if cfg["splitting"] else (U, x, T)

    x, T, nH, Q = st.x5, st.T, st.nH, torch.as_tensor(st.Q, device=DEV)
    if kind == "transport":
        for _ in range(n_sub):
            U = _transport(g, cfg, U, dts)
    elif kind == "chemistry":
        U, x, T = chem(U, x, T, Q, nH, dts)
    elif kind == "levels":
        for m in _masks(case, C, mesh.lattice):
            on = torch.as_tensor(m, device=DEV).bool()
            for _ in range(n_sub):
                U, x, T = sub(U, x, T, Q, nH, None if bool(on.all()) else on)
    elif kind == "adjoint":
        Q, nH = Q.requires_grad_(), nH.requires_grad_()
        mass = (nH * g.V / (nH * g.V).sum()).detach()
        for _ in range(n_sub):
            U, x, T = checkpoint(sub, U, x, T, Q, nH, use_reentrant=False)
        dQ, dnH = torch.autograd.grad((mass * x[1]).sum(), (Q, nH))
        return dict(N=U[..., 0].T.detach(), x5=x.detach(), T=T.detach(), dQ=dQ, dnH=dnH)
    else:
        for _ in range(n_sub):
            U, x, T = sub(U, x, T, Q, nH)
    out = U.permute(1, 2, 0)
    return dict(N=out[:, 0], F=out[:, 1:] * cfg["c_red"], x5=x, T=T)
