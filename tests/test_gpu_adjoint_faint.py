"""The reverse mode over photon densities beyond a light front: N zero or log-uniform
from far below the range of its square to 1e-3, |F| up to N and, after the linear
reconstruction, beyond it, so that squares, quotients and roots of the face
states leave the normal range.  Every output finite, and dL/dQ, dL/dn_H and the
abundances' cotangents those of the oracle (1e-9)."""
import numpy as np
import pytest

from _cases import make_oracle, voronoi_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lowest", [-30, -170, -300])
def test_faint_fields(lowest):
    from paper_2404_17630_gb300 import RT, make_config
    mesh, cfg, st = voronoi_case(n=10, seed=3)
    rng = np.random.default_rng(12)
    scale = 10.0 ** rng.uniform(lowest, -3, mesh.n_cells)
    scale[::97] = 0.0
    N = scale * rng.uniform(0.5, 1, (3, mesh.n_cells))
    d = rng.standard_normal((3, 3, mesh.n_cells))
    fr = d / np.linalg.norm(d, axis=1, keepdims=True) * N[:, None] * rng.uniform(0, 1, (3, 1, mesh.n_cells))
    st = dict(st, N=N, fr=fr)
    rt = RT(make_config(**cfg), mesh)
    rt.set_radiation(N, fr * cfg["c_red"])
    rt.set_gas(st["nH"], st["x5"], st["T"])
    rt.set_sources(st["cells"], st["Q"])
    o = make_oracle(mesh, cfg, st)
    dt = 0.2 * o.max_dt()
    lx = np.zeros((5, mesh.n_cells))
    lx[1] = st["nH"] * mesh.volume
    g = rt.adjoint(3 * dt, 3, 2, lam_x5=lx, n_src=len(st["cells"]))
    for k, v in g.items():
        assert np.isfinite(v).all(), k
    ref = o.adjoint(3 * dt, 3, lam_x5=lx)
    assert ref["status"] == 0
    for a, b in ((g["dnH"], ref["g_nH"]), (g["x5"], ref["lam0"]["x5"]), (g["dQ"], ref["g_src"][:, st["cells"]].T)):
        assert np.abs(a - b).max() <= 1e-9 * np.abs(b).max()
