"""The FP64 closure at photon densities whose squares leave the range of doubles, in
either direction: the face fluxes of a uniform state are the oracle's (1e-12 of the
largest), and the reverse mode of the transport, which does not change when the
whole state is scaled by a power of two, is that of the unscaled state (1e-12)."""
import numpy as np
import pytest

from _cases import make_oracle, voronoi_case

pytestmark = pytest.mark.gpu


def _gpu(mesh, cfg, N, fr, st):
    from paper_2404_17630_gb300 import RT, make_config
    rt = RT(make_config(**cfg), mesh)
    rt.set_gas(st["nH"], st["x5"], st["T"])
    rt.set_radiation(N, fr * cfg["c_red"])
    return rt


# the reduced flux times c_red has to stay finite too
@pytest.mark.parametrize("N0,F0", [(1e-3, 0.97e-3), (2.7e-162, 2.65e-162), (1e-158, 0.9e-158), (1e-170, 1e-170),
                                   (1e-170, 1e-100), (6e153, 5e153), (1e154, 0.9e154), (1.35e154, 1.33e154),
                                   (1e155, 1e100), (1e155, 0.9e155), (1e100, 1e155)])
def test_fluxes(N0, F0):
    mesh, cfg, st = voronoi_case(n=6, seed=5, order=1, chem_mode=0, n_bins=1)
    C = mesh.n_cells
    N, fr = np.full((1, C), N0), np.zeros((1, 3, C))
    fr[0, 0] = F0
    o = make_oracle(mesh, cfg, dict(st, N=N, fr=fr, cells=[], Q=None))
    ref = o.face_fluxes(o.gradients())
    got = _gpu(mesh, cfg, N, fr, st).face_fluxes()
    assert np.isfinite(got).all()
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()


def test_reverse_mode():
    mesh, cfg, st = voronoi_case(n=6, seed=5, order=1, chem_mode=0, n_bins=1)
    C = mesh.n_cells
    rng = np.random.default_rng(3)
    N = rng.uniform(0.5, 1, (1, C))
    d = rng.standard_normal((1, 3, C))
    fr = d / np.linalg.norm(d, axis=1, keepdims=True) * N[:, None] * rng.uniform(0, 0.9, (1, 1, C))
    lam = rng.standard_normal((1, C))
    out = []
    for k in (0, 511, 512):   # N^2 below, N^2 and 4 N^2 above the largest double
        rt = _gpu(mesh, cfg, np.ldexp(N, k), np.ldexp(fr, k), st)
        dt = 0.5 * rt.max_dt()
        out.append(rt.adjoint(2 * dt, 2, 1, lam_N=lam))
    for g in out[1:]:
        for k in ("N", "F"):
            assert np.abs(g[k] - out[0][k]).max() <= 1e-12 * np.abs(out[0][k]).max(), k
