"""The worklist's choice between groups of lanes and one thread per cell, made from
the chains foretold by the first attempts: chains of equal length (a uniform
half-ionised gas that an intense field ionises in part of the box), where threads
are several times faster from a few thousand cells on, and very uneven ones (a
strong field in a tenth of the box), where groups are, at lengths on both sides of
the limits.  A shorter list of the same chains never takes longer than a longer
one, and either way the results are the oracle's within the parity tests' bounds."""
import numpy as np
import pytest

import synth
from _cases import SIGMA3, base_config, make_oracle, voronoi_case

pytestmark = pytest.mark.gpu

MESH = synth.cartesian_mesh(40, 10.0)


def _even(listed, g, dt, c_red):
    C = MESH.n_cells
    rng = np.random.default_rng(3)
    on = rng.choice(C, listed, replace=False)
    x5 = np.zeros((5, C))
    x5[0] = x5[2] = 1.0
    x5[:2, on] = 0.5
    N = np.zeros((3, C))
    N[0, on] = g / (c_red * SIGMA3[0][0] * dt) * rng.uniform(0.95, 1.05, listed)
    return dict(nH=np.full(C, 1e-6), x5=x5, T=np.full(C, 1e4), N=N, fr=np.zeros((3, 3, C)))


def _rt(mesh, cfg, prec):
    from paper_2404_17630_gb300 import RT, make_config
    return RT(make_config(precision=prec, gather_sum=1, **cfg), mesh)


def _run(rt, st, c_red, dt, reps=1):
    """Best chemistry time (ms) of `reps` calls from the same state."""
    import paper_2404_17630_gb300.rt as rtb
    best = np.inf
    rtb.rt_profile_enable(rt.ctx, reps > 1)
    for _ in range(reps):
        rt.set_radiation(st["N"], st["fr"] * c_red)
        rt.set_gas(st["nH"], st["x5"], st["T"])
        rtb.rt_profile_read(rt.ctx)
        rt.thermochemistry(dt)
        rt.sync()
        best = min(best, rtb.rt_profile_read(rt.ctx)["k_chem"][0])
    rtb.rt_profile_enable(rt.ctx, False)
    return best


def _check(rt, o, cfg, prec):
    g = rt.fields()
    N, fr = o.radiation()
    x5, T = o.gas()
    for k, a, b in (("N", g["N"], N), ("x5", g["x5"], x5), ("T", g["T"], T)):
        assert np.abs(a - b).max() < (1e-12 if prec == "fp64" else 1e-4) * np.abs(b).max(), k
    if prec == "fp64":
        assert np.array_equal(g["nsub"], o.substeps())


@pytest.mark.parametrize("prec,lengths", [("fp64", (1500, 20000, 60000)), ("mixed", (1000, 20000, 45000))])
@pytest.mark.parametrize("g", [0.15, 20.0])
def test_even_chains(prec, lengths, g):
    cfg = base_config(chem_mode=1)
    rt = _rt(MESH, cfg, prec)
    dt = rt.max_dt()
    ms = []
    for listed in lengths:
        st = _even(listed, g, dt, cfg["c_red"])
        ms.append(_run(rt, st, cfg["c_red"], dt, reps=4))
        assert (rt.fields()["nsub"] > 1).sum() == listed
        if g < 1 or listed < 2000:
            o = make_oracle(MESH, cfg, st)
            o.thermochemistry(dt)
            _check(rt, o, cfg, prec)
    assert ms[1] < ms[2], ms


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [23, 36])
def test_uneven_chains(prec, n):
    mesh, cfg, st = voronoi_case(n=n, seed=6)
    rng = np.random.default_rng(n)
    C = mesh.n_cells
    N = np.where(rng.uniform(size=C) < 0.9, 1e-7, 10 ** rng.uniform(-9, -2, C))
    st = dict(st, N=N * np.array([[1.0], [0.1], [0.03]]), fr=np.zeros((3, 3, C)), cells=[], Q=None)
    rt, o = _rt(mesh, cfg, prec), make_oracle(mesh, cfg, st)
    dt = 0.9 * o.max_dt()
    _run(rt, st, cfg["c_red"], dt)
    o.thermochemistry(dt)
    _check(rt, o, cfg, prec)
