"""The mixed flux application with FP64 sums (gather_sum = 0) at photon densities
whose face fluxes, formed in FP32, lie in FP32's subnormal range: they are widened
exactly.  First order and F = 0, so that a flux is a difference of two densities.
Bound: a term is off by at most four roundings, 2.4e-7 of itself or 2^-148 absolute
(4e-6 of the smallest density's share), and a cell has at most 30: 1e-5."""
import numpy as np
import pytest

from _cases import make_oracle, voronoi_case

pytestmark = pytest.mark.gpu


def test_subnormal_terms():
    from paper_2404_17630_gb300 import RT, make_config
    mesh, cfg, st = voronoi_case(n=6, seed=5, order=1, chem_mode=0, n_bins=1)
    C = mesh.n_cells
    N = 10 ** np.random.default_rng(4).uniform(-37.5, -36.5, (1, C))
    st = dict(st, N=N, fr=np.zeros((1, 3, C)), cells=[], Q=None)
    o = make_oracle(mesh, cfg, st)
    rt = RT(make_config(precision="mixed", gather_sum=0, **cfg), mesh)
    rt.set_gas(st["nH"], st["x5"], st["T"])
    rt.set_radiation(N)
    dt = 0.9 * o.max_dt()
    flux = np.abs(rt.face_fluxes()[..., 0])
    assert ((flux > 0) & (flux < 1.17e-38)).mean() > 0.3   # the case does what it is for
    o.transport(dt)
    rt.transport(dt)
    rt.sync()
    ref = o.radiation()[0]
    assert (np.abs(rt.fields()["N"] - ref) / ref).max() < 1e-5
