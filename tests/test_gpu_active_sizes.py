"""Active sets on meshes below and above the sizes up to which the lists are built
(2,048 cells) and the masks compared (8,192) on the host: one active cell, the last
one, all but one, every other one, none, all, random ones, more than are kept, in
host and device memory with any nonzero byte.  One step per mask against the oracle
(FP64 1e-12, mixed 1e-4), each mask twice, the second time from the kept set; and a
mask costs less on a small mesh than on a large one."""
import time

import numpy as np
import pytest

from _cases import make_oracle, voronoi_case

pytestmark = pytest.mark.gpu


def _masks(C):
    rng = np.random.default_rng(4)
    one, last, but = np.zeros(C, np.uint8), np.zeros(C, np.uint8), np.full(C, 255, np.uint8)
    one[C // 3] = 7
    last[-1] = 1
    but[C // 2] = 0
    out = [one, last, but, (np.arange(C) % 2).astype(np.uint8), np.zeros(C, np.uint8), np.ones(C, np.uint8)]
    return out + [(rng.random(C) < p).astype(np.uint8) * 3 for p in (0.02, 0.2, 0.5, 0.9, 0.97)]


def _rt(n, prec):
    from paper_2404_17630_gb300 import RT, make_config
    mesh, cfg, st = voronoi_case(n=n, seed=9)
    rt = RT(make_config(precision=prec, gather_sum=1, **cfg), mesh)
    rt.set_radiation(st["N"], st["fr"] * cfg["c_red"])
    rt.set_gas(st["nH"], st["x5"], st["T"])
    rt.set_sources(st["cells"], st["Q"])
    return rt, mesh, cfg, st


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("mixed", 1e-4)])
@pytest.mark.parametrize("n", [12, 13, 20, 21])   # 1,728, 2,197, 8,000 and 9,261 cells
def test_active_sets(n, prec, tol):
    import torch
    rt, mesh, cfg, st = _rt(n, prec)
    o = make_oracle(mesh, cfg, st)
    dt = 0.3 * o.max_dt()
    masks = _masks(mesh.n_cells)
    for rnd in range(2):
        for k, m in enumerate(masks):
            rt.set_active(torch.as_tensor(m, device="cuda") if (k + rnd) % 2 else m)
            rt.step(dt, 1)
            o.set_active(m != 0)
            assert o.step(dt, 1) == 0
        rt.sync()
        f = rt.fields()
        N, fr = o.radiation()
        x5, T = o.gas()
        for a, b in ((f["N"], N), (f["F"] / cfg["c_red"], fr), (f["x5"], x5), (f["T"], T)):
            assert np.abs(a - b).max() <= tol * np.abs(b).max()


def test_time_by_size():
    known, new = [], []
    for n in (10, 30):
        rt, mesh, cfg, st = _rt(n, "mixed")
        rng = np.random.default_rng(n)
        masks = [(rng.random(mesh.n_cells) < 0.3).astype(np.uint8) for _ in range(20)]
        t = []
        for m in masks * 3:   # 20 masks, 8 kept: each one new
            t0 = time.perf_counter()
            rt.set_active(m)
            t.append(time.perf_counter() - t0)
        new.append(min(t))
        t = []
        for _ in range(20):
            t0 = time.perf_counter()
            rt.set_active(masks[0])
            rt.set_active(masks[1])
            t.append(time.perf_counter() - t0)
        known.append(min(t))
    assert new[0] < 0.7 * new[1], new
    assert known[0] < 0.5 * known[1], known
