"""The FP64 gradients' search for the limiting faces (an FP32 leader per sign,
all faces in FP64 where the lead is too small): random fields on ragged cells,
and fields whose extrapolations tie by symmetry or vanish -- waves along an
axis and along the diagonal of a Cartesian and a staggered grid, a uniform
field, a spike, amplitudes far outside the FP32 range.  Against the oracle,
1e-12 of the largest gradient; the context's gradients and the allocation-free
ones, the latter also on cells with twice the faces (more half-edges than a
block can hold in shared memory)."""
import dataclasses

import numpy as np
import pytest

import synth
from _cases import base_config, neutral_gas

pytestmark = pytest.mark.gpu

MESHES = {"voronoi": lambda: synth.voronoi_mesh(9, 10.0, 0.3, seed=4), "grid": lambda: synth.cartesian_mesh(8, 10.0),
          "staggered": lambda: synth.bcc_mesh(5, 10.0)}


def _twice(mesh):
    """Every face as two of half its area."""
    two = {k: np.concatenate([getattr(mesh, k)] * 2) for k in ("left", "right", "nx", "ny", "nz", "fx", "fy", "fz")}
    return dataclasses.replace(mesh, area=np.concatenate([0.5 * mesh.area] * 2), **two)


def _field(kind, mesh):
    C = mesh.n_cells
    rng = np.random.default_rng(8)
    k = 2 * np.pi / mesh.box
    if kind == "wave_x":
        N = 1 + 0.5 * np.sin(k * mesh.cx)
    elif kind == "diagonal":
        N = 1 + 0.2 * (np.sin(k * mesh.cx) + np.sin(k * mesh.cy) + np.sin(k * mesh.cz))
    elif kind == "uniform":
        N = np.full(C, 0.7)
    elif kind == "spike":
        N = np.zeros(C)
        N[C // 2] = 1.0
    else:
        N = rng.uniform(0, 1, C)
    N = N * (1e-200 if kind == "tiny" else 1.0)
    d = rng.standard_normal((3, C))
    return N[None], (N * 0.5 * d / np.linalg.norm(d, axis=0))[None]


@pytest.mark.parametrize("kind", ["random", "wave_x", "diagonal", "uniform", "spike", "tiny"])
@pytest.mark.parametrize("name", list(MESHES) + ["voronoi2"])
def test_limited_gradients(name, kind):
    import torch
    from oracle import Oracle, default_config
    from paper_2404_17630_gb300 import RT, make_config
    from paper_2404_17630_gb300 import rt as rtb
    mesh = _twice(MESHES["voronoi"]()) if name == "voronoi2" else MESHES[name]()
    C, F = mesh.n_cells, mesh.n_faces
    N, f = _field(kind, mesh)
    cfg = base_config(n_bins=1, c_red=1.0)
    o = Oracle(default_config(**cfg), mesh)
    o.set_radiation(N, f)
    o.set_gas(*neutral_gas(C, 1e-3))
    ref = o.gradients().reshape(C, 1, 4, 3)
    scale = np.abs(ref).max() or 1.0
    rt = RT(make_config(**cfg), mesh)
    rt.set_radiation(N, f)
    assert np.abs(rt.gradients() - ref).max() <= 1e-12 * scale
    cell = np.concatenate([mesh.left, mesh.right]).astype(np.int64)
    entry = np.concatenate([2 * np.arange(F), 2 * np.arange(F) + 1])
    csr = entry[np.lexsort((entry, cell))].astype(np.int32)
    off = np.concatenate([[0], np.cumsum(np.bincount(cell, minlength=C))]).astype(np.int32)
    dev = {k: torch.as_tensor(np.ascontiguousarray(getattr(mesh, k)), device="cuda")
           for k in ("volume", "cx", "cy", "cz", "left", "right", "area", "nx", "ny", "nz", "fx", "fy", "fz")}
    cells = rtb.rt_cells(C, *[dev[k].data_ptr() for k in ("volume", "cx", "cy", "cz")])
    faces = rtb.rt_faces(F, *[dev[k].data_ptr() for k in ("left", "right", "area", "nx", "ny", "nz", "fx", "fy", "fz")])
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    G = torch.empty(C, 1, 4, 3, dtype=torch.float64, device="cuda")
    bad = torch.empty(1, dtype=torch.int32, device="cuda")
    toff, tcsr, tN, tf = t(off), t(csr), t(N), t(f)
    rtb.rt_gradients_noalloc(cells, faces, toff, tcsr, 1, 2, 1, 1e-5, mesh.box, tN, tf, G, bad)
    torch.cuda.synchronize()
    assert int(bad) == 0
    assert np.abs(G.cpu().numpy() - ref).max() <= 1e-12 * scale
