"""rt_init_mesh's face lists, built on the device: faces in random order, a cell
with far more faces than the usual handful (its list is sorted by a heap), cell
counts around a multiple of the prefix sums' block, meshes that are refused
(the first offender named), a context given another mesh.  The steps against
the oracle as in the parity tests (FP64 1e-12)."""
import dataclasses

import numpy as np
import pytest

import synth
from _cases import EPS3, SIGMA3, make_oracle, voronoi_case

pytestmark = pytest.mark.gpu

FACE_ARRAYS = ("left", "right", "area", "nx", "ny", "nz", "fx", "fy", "fz")


def _rt(mesh, cfg, st, **kw):
    from paper_2404_17630_gb300 import RT, make_config
    rt = RT(make_config(**dict(cfg, **kw)), mesh)
    _state(rt, cfg, st)
    return rt


def _state(rt, cfg, st):
    rt.set_radiation(st["N"], st["fr"] * cfg["c_red"])
    rt.set_gas(st["nH"], st["x5"], st["T"])
    rt.set_sources(st["cells"], st["Q"])


def _shuffled(mesh, seed=0):
    p = np.random.default_rng(seed).permutation(mesh.n_faces)
    return dataclasses.replace(mesh, **{k: getattr(mesh, k)[p] for k in FACE_ARRAYS})


def _hub(mesh, n):
    """Small faces from cell 0 to n other cells."""
    rng = np.random.default_rng(1)
    to = rng.choice(np.arange(1, mesh.n_cells), n, replace=False).astype(np.int32)
    c = mesh.centroids()
    d = c[to] - c[0]
    d -= mesh.box * np.round(d / mesh.box)
    nrm = d / np.linalg.norm(d, axis=1, keepdims=True)
    f = np.mod(c[0] + 0.5 * d, mesh.box)
    new = dict(left=np.zeros(n, np.int32), right=to, area=np.full(n, 1e-4), nx=nrm[:, 0], ny=nrm[:, 1], nz=nrm[:, 2],
               fx=f[:, 0], fy=f[:, 1], fz=f[:, 2])
    return dataclasses.replace(mesh, **{k: np.concatenate([getattr(mesh, k), new[k]]) for k in FACE_ARRAYS})


@pytest.mark.parametrize("kind", ["shuffled", "hub", "c1000", "c1331"])
def test_built_lists(kind):
    mesh, cfg, st = voronoi_case(n={"c1000": 10, "c1331": 11}.get(kind, 8), seed=6)
    mesh = _shuffled(_hub(mesh, 150) if kind == "hub" else mesh)
    rt, o = _rt(mesh, cfg, st), make_oracle(mesh, cfg, st)
    g = o.gradients()
    assert np.abs(rt.gradients().reshape(g.shape) - g).max() <= 1e-12 * np.abs(g).max()
    deg = np.bincount(np.concatenate([mesh.left, mesh.right]), minlength=mesh.n_cells)
    assert rt.mesh_info() == (mesh.n_cells, mesh.n_faces, deg.max())
    dt = 0.5 * o.max_dt()
    assert rt.max_dt() == pytest.approx(o.max_dt(), rel=1e-15)
    rt.step(2 * dt, 2)
    rt.sync()
    assert o.step(2 * dt, 2) == 0
    f = rt.fields()
    N, fr = o.radiation()
    x5, T = o.gas()
    for a, b in ((f["N"], N), (f["F"] / cfg["c_red"], fr), (f["x5"], x5), (f["T"], T)):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()


def test_refused_meshes():
    from paper_2404_17630_gb300 import RT, make_config
    from paper_2404_17630_gb300 import rt as rtb
    mesh, cfg, st = voronoi_case(n=8, seed=6)

    def refused(**kw):
        bad = dataclasses.replace(mesh, **kw)
        with pytest.raises(rtb.RTError) as e:
            RT(make_config(**cfg), bad)
        assert e.value.status == rtb.RT_BAD_MESH
        return str(e.value)

    left, right, vol = mesh.left.copy(), mesh.right.copy(), mesh.volume.copy()
    left[[70, 900]] = [-3, 5000]
    assert "face 70 joins cells -3" in refused(left=left)
    right[41] = mesh.left[41]
    assert "face 41 joins" in refused(right=right)
    vol[[33, 400]] = [0.0, np.nan]
    assert "cell 33 has volume 0" in refused(volume=vol)
    keep = (mesh.left != 77) & (mesh.right != 77)
    assert "cell 77 has no faces" in refused(**{k: getattr(mesh, k)[keep] for k in FACE_ARRAYS})


def test_context_takes_another_mesh():
    """The second mesh's sources, active masks and reverse mode start afresh."""
    from _cases import base_config
    cfg = base_config(sigma=SIGMA3, eps=EPS3)
    first, _, st1 = voronoi_case(n=10, seed=1, n_src=7)
    second, _, st2 = voronoi_case(n=8, seed=2, n_src=5)
    rt = _rt(first, cfg, st1)
    lx = np.ones((5, first.n_cells))
    rt.adjoint(rt.max_dt(), 1, 1, lam_x5=lx, n_src=7)
    rt.init_mesh(second)
    _state(rt, cfg, st2)
    new = _rt(second, cfg, st2)
    lx = np.ones((5, second.n_cells))
    a, b = (r.adjoint(2 * r.max_dt(), 2, 1, lam_x5=lx, n_src=5) for r in (rt, new))
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    assert np.array_equal(rt.fields()["N"], new.fields()["N"])
