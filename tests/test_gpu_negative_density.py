"""Negative photon densities entering the chemistry.  The linear reconstruction does
not keep N >= 0: a beam beside an almost empty region leaves small negative N, and
larger ones without the limiter.  An attempt ends at max(N - removed, 0) and takes
the flux of a cell with N <= 0 away.  Accepted first attempts, groups of lanes (216
cells) and one thread per cell (50,653), whole steps, and the reverse mode, which
differentiates the clamp; in the mixed path too.  Bounds as in the parity tests: FP64
1e-12, reverse mode 1e-9, mixed 1e-4, each against the oracle."""
import numpy as np
import pytest

import synth
from _cases import base_config, make_oracle, neutral_gas, voronoi_case

pytestmark = pytest.mark.gpu


def _gpu(mesh, cfg, st, **kw):
    from paper_2404_17630_gb300 import RT, make_config
    rt = RT(make_config(**dict(cfg, **kw)), mesh)
    rt.set_radiation(st["N"], st["fr"] * cfg["c_red"])
    rt.set_gas(st["nH"], st["x5"], st["T"])
    if "cells" in st:
        rt.set_sources(st["cells"], st["Q"])
    return rt


def _errors(rt, o, cfg):
    g = rt.fields()
    N, fr = o.radiation()
    x5, T = o.gas()
    assert (g["N"] >= 0).all()
    return {k: np.abs(a - b).max() / np.abs(b).max()
            for k, a, b in (("N", g["N"], N), ("F", g["F"] / cfg["c_red"], fr), ("x5", g["x5"], x5), ("T", g["T"], T))}


def _negative(n):
    """Random state with N < 0 in 30 % of the (cell, bin)s, small enough that no rate changes sign of 1 + rate."""
    mesh, cfg, st = voronoi_case(n=n, seed=5)
    rng = np.random.default_rng(1)
    shape = st["N"].shape
    st["N"] = np.where(rng.uniform(size=shape) < 0.3, -10 ** rng.uniform(-9, -5, shape), st["N"])
    return mesh, cfg, st


def _beam(**kw):
    """A beam with |F| = c N through an almost empty periodic box."""
    n = 16
    mesh = synth.cartesian_mesh(n, 10.0)
    C = mesh.n_cells
    cfg = base_config(**kw)
    nH, x5, T = neutral_gas(C, 1e-3)
    j, k = np.arange(C) // n % n, np.arange(C) // (n * n)
    on = (abs(j - 8) < 3) & (abs(k - 8) < 3) & (np.arange(C) % n < 6)
    N = np.where(on, 1e-3, 1e-10) * np.array([[1.0], [0.1], [0.03]])
    fr = np.zeros((3, 3, C))
    fr[:, 0] = np.where(on, N, 0.0)
    return mesh, cfg, dict(nH=nH, x5=x5, T=T, N=N, fr=fr)


@pytest.mark.parametrize("n", [6, 37])
def test_chemistry_fp64(n):
    mesh, cfg, st = _negative(n)
    o, rt = make_oracle(mesh, cfg, st), _gpu(mesh, cfg, st)
    dt = 0.9 * o.max_dt()
    o.thermochemistry(dt)
    rt.thermochemistry(dt)
    rt.sync()
    e = _errors(rt, o, cfg)
    assert max(e.values()) < 1e-12, e
    assert np.array_equal(rt.fields()["nsub"], o.substeps())


@pytest.mark.parametrize("limiter", [1, 0])
def test_beam_fp64(limiter):
    mesh, cfg, st = _beam(limiter=limiter)
    o, rt = make_oracle(mesh, cfg, st), _gpu(mesh, cfg, st)
    dt = 0.9 * o.max_dt()
    lowest = 0.0
    for _ in range(30):
        o.thermochemistry(dt)
        o.transport(dt)
        lowest = min(lowest, o.radiation()[0].min())
    assert lowest < 0   # the case does what it is for
    rt.step(30 * dt, 30)
    rt.sync()
    o.thermochemistry(dt)
    rt.thermochemistry(dt)
    rt.sync()
    e = _errors(rt, o, cfg)
    assert max(e.values()) < 1e-12, e


def test_adjoint():
    mesh, cfg, st = _negative(8)
    o, rt = make_oracle(mesh, cfg, st), _gpu(mesh, cfg, st)
    dt = 0.5 * o.max_dt()
    rng = np.random.default_rng(2)
    lx, lN = np.zeros((5, mesh.n_cells)), rng.standard_normal(st["N"].shape)
    lx[1] = st["nH"] * mesh.volume
    g = rt.adjoint(3 * dt, 3, 2, lam_N=lN, lam_x5=lx)
    ref = o.adjoint(3 * dt, 3, lam_N=lN, lam_x5=lx)
    assert ref["status"] == 0
    for k, a, b in (("dnH", g["dnH"], ref["g_nH"]), ("N", g["N"], ref["lam0"]["N"]),
                    ("F", g["F"] * cfg["c_red"], ref["lam0"]["fr"]), ("x5", g["x5"], ref["lam0"]["x5"]),
                    ("T", g["T"], ref["lam0"]["T"])):
        assert np.abs(a - b).max() <= 1e-9 * np.abs(b).max(), k


@pytest.mark.parametrize("n", [6, 37])
def test_chemistry_mixed(n):
    mesh, cfg, st = _negative(n)
    o, rt = make_oracle(mesh, cfg, st), _gpu(mesh, cfg, st, precision="mixed", gather_sum=1)
    dt = 0.9 * o.max_dt()
    o.thermochemistry(dt)
    rt.thermochemistry(dt)
    rt.sync()
    e = _errors(rt, o, cfg)
    assert max(e.values()) < 1e-4, e


def test_beam_mixed():
    """One subcycle's chemistry on the state that the beam's FP64 transport leaves (N < 0 in it)."""
    mesh, cfg, st = _beam(limiter=0)
    o = make_oracle(mesh, cfg, st)
    dt = 0.9 * o.max_dt()
    for _ in range(8):
        o.transport(dt)
    N, fr = o.radiation()
    assert N.min() < 0
    rt = _gpu(mesh, cfg, dict(st, N=N, fr=fr), precision="mixed")
    o.thermochemistry(dt)
    rt.thermochemistry(dt)
    rt.sync()
    e = _errors(rt, o, cfg)
    assert max(e.values()) < 1e-4, e


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("mixed", 1e-4)])
@pytest.mark.parametrize("most", [1, 2])
def test_cap(prec, tol, most):
    """Cells that reach the cap on attempts, some before one is accepted: those keep N < 0 and their flux."""
    from paper_2404_17630_gb300.rt import RTError
    mesh, cfg, st = _negative(6)
    cfg = dict(cfg, max_substeps=most)
    o, rt = make_oracle(mesh, cfg, st), _gpu(mesh, cfg, st, precision=prec, gather_sum=1)
    dt = 0.9 * o.max_dt()
    assert o.thermochemistry(dt) == 4
    rt.thermochemistry(dt)
    with pytest.raises(RTError, match="max_substeps"):
        rt.sync()
    g = rt.fields()
    N, fr = o.radiation()
    x5, T = o.gas()
    assert N.min() < 0
    for a, b in ((g["N"], N), (g["F"] / cfg["c_red"], fr), (g["x5"], x5), (g["T"], T)):
        assert np.abs(a - b).max() < tol * np.abs(b).max()
