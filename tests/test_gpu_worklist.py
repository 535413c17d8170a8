"""The chemistry's worklist by groups of lanes and by one thread per cell, which
take over at 49,152 (FP64) and 24,576 (mixed) rejected cells: far from
equilibrium almost every cell's first attempt is rejected, so the 28^3 and 30^3
meshes (mixed) and the 36^3 and 37^3 meshes (FP64) lie below and above; 1, 2 and 3
bins, thermal and isothermal, a hydrogen-only gas and rates switched off on
small meshes.  Bounds as in the parity tests: FP64 1e-12 with the oracle's
substep counts, mixed 1e-4."""
import numpy as np
import pytest

from _cases import make_oracle, voronoi_case

pytestmark = pytest.mark.gpu


def _run(n, prec, **kw):
    from paper_2404_17630_gb300 import RT, make_config
    mesh, cfg, st = voronoi_case(n=n, seed=5, **kw)
    st["N"] = st["N"] * 10.0
    st["fr"] = st["fr"] * 10.0
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
    N, fr = o.radiation()
    x5, T = o.gas()
    err = max(np.abs(a - b).max() / np.abs(b).max()
              for a, b in ((g["N"], N), (g["F"] / cfg["c_red"], fr), (g["x5"], x5), (g["T"], T)))
    return err, g["nsub"], o.substeps()


@pytest.mark.parametrize("n", [5, 15, 17])
@pytest.mark.parametrize("kw", [{}, dict(chem_mode=1, n_bins=1), dict(n_bins=2, y_he=0.0), dict(chem_flags=8),
                                dict(chem_flags=6)], ids=["full", "iso1", "H2", "photo", "coll"])
def test_worklist_fp64(n, kw):
    err, ns, ref = _run(n, "fp64", **kw)
    assert err < 1e-12
    assert np.array_equal(ns, ref)


@pytest.mark.parametrize("n", [5, 15, 17])
@pytest.mark.parametrize("kw", [{}, dict(chem_mode=1, n_bins=1), dict(n_bins=2, y_he=0.0), dict(chem_flags=8)],
                         ids=["full", "iso1", "H2", "photo"])
def test_worklist_mixed(n, kw):
    err, ns, ref = _run(n, "mixed", **kw)
    assert err < 1e-4
    assert (ns >= 1).all()


@pytest.mark.parametrize("prec,n", [("fp64", 36), ("fp64", 37), ("mixed", 28), ("mixed", 30)])
def test_worklist_lengths(prec, n):
    err, ns, ref = _run(n, prec)
    assert err < (1e-12 if prec == "fp64" else 1e-4)
    if prec == "fp64":
        assert np.array_equal(ns, ref)
