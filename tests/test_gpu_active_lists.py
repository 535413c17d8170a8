"""The active sets' lists, built and compared on the device: cell counts that are
no multiple of a word, a block of cells or a scan's block; one active cell, all
but one, the last one, every other one; more masks than are kept; masks in host
and device memory with any nonzero byte.  One step per mask against the oracle
(FP64 1e-12), each mask twice (the second time from the kept set)."""
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


@pytest.mark.parametrize("n,prec,tol", [(8, "fp64", 1e-12), (10, "fp64", 1e-12), (11, "fp64", 1e-12), (11, "mixed", 1e-4)])
def test_active_sets(n, prec, tol):
    import torch
    from paper_2404_17630_gb300 import RT, make_config
    mesh, cfg, st = voronoi_case(n=n, seed=9)
    rt = RT(make_config(precision=prec, gather_sum=1, **cfg), mesh)
    rt.set_radiation(st["N"], st["fr"] * cfg["c_red"])
    rt.set_gas(st["nH"], st["x5"], st["T"])
    rt.set_sources(st["cells"], st["Q"])
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
