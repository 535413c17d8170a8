"""The FP64 gradients do not depend on the unit of length: with every length of the
mesh multiplied by a power of two (cells of 1e-22 to 1e22, as in a unit of cm or of
Gpc) they are the unscaled ones, scaled, bit for bit, and take the same time (the
limiter's FP32 search is to work in every unit)."""
import dataclasses

import numpy as np
import pytest

from _cases import voronoi_case

pytestmark = pytest.mark.gpu


def _scaled(mesh, k):
    one = {q: np.ldexp(getattr(mesh, q), k) for q in ("cx", "cy", "cz", "fx", "fy", "fz")}
    return dataclasses.replace(mesh, volume=np.ldexp(mesh.volume, 3 * k), area=np.ldexp(mesh.area, 2 * k), **one)


def _gradients(k, n):
    from paper_2404_17630_gb300 import RT, make_config
    import paper_2404_17630_gb300.rt as rtb
    mesh, cfg, st = voronoi_case(n=n, seed=5)
    cfg = dict(cfg, box=float(np.ldexp(cfg["box"], k)), unit_length_cm=float(np.ldexp(cfg["unit_length_cm"], -k)))
    rt = RT(make_config(**cfg), _scaled(mesh, k))
    rt.set_gas(st["nH"], st["x5"], st["T"])
    rt.set_radiation(st["N"], st["fr"] * cfg["c_red"])
    G = rt.gradients()
    rtb.rt_profile_enable(rt.ctx, True)
    best = np.inf
    for _ in range(8):
        rtb.rt_profile_read(rt.ctx)
        for _ in range(4):
            rtb.rt_stage_gradients(rt.ctx)
        best = min(best, rtb.rt_profile_read(rt.ctx)["k_grad"][0] / 4)
    return np.ldexp(G, k), best


@pytest.mark.parametrize("k", [-72, -60, 1, 60, 63, 72])
def test_values(k):
    assert np.array_equal(_gradients(k, 8)[0], _gradients(0, 8)[0])


@pytest.mark.parametrize("k", [-72, 72])
def test_time(k):
    t0, t1 = _gradients(0, 40)[1], _gradients(k, 40)[1]
    assert t1 < 1.15 * t0, (t0, t1)
