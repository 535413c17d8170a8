"""The rate fits and the cooling function over the whole range of temperatures, by
groups of lanes (1,000 cells) and by one thread per cell (50,653 cells with long
chains): gas at 1e3 to 3e7 K, where collisional ionisation of HeII, dielectronic
recombination and the excitation of HeII set the chains.  Bounds as in the parity
tests (1e-12 with the oracle's substep counts, mixed 1e-4), the temperature per cell."""
import numpy as np
import pytest

from _cases import make_oracle, voronoi_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [10, 37])
def test_hot_gas(prec, n):
    from paper_2404_17630_gb300 import RT, make_config
    mesh, cfg, st = voronoi_case(n=n, seed=5)
    st["T"] = 10 ** np.random.default_rng(1).uniform(3, 7.5, mesh.n_cells)
    rt = RT(make_config(precision=prec, gather_sum=1, **cfg), mesh)
    rt.set_radiation(st["N"], st["fr"] * cfg["c_red"])
    rt.set_gas(st["nH"], st["x5"], st["T"])
    rt.set_sources(st["cells"], st["Q"])
    o = make_oracle(mesh, cfg, st)
    dt = 0.9 * o.max_dt()
    o.thermochemistry(dt)
    rt.thermochemistry(dt)
    rt.sync()
    g = rt.fields()
    x5, T = o.gas()
    tol = 1e-12 if prec == "fp64" else 1e-4
    assert (np.abs(g["T"] - T) / T).max() < tol
    assert np.abs(g["x5"] - x5).max() < tol
    assert np.abs(g["N"] - o.radiation()[0]).max() < tol * o.radiation()[0].max()
    if prec == "fp64":
        assert np.array_equal(g["nsub"], o.substeps())
