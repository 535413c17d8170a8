"""Point sources in a few and in most of the cells (the two ways to index them), some
cells named several times: the photons they give in one subcycle are those of numpy's
sums, and a source for every cell of a large mesh costs no more than a sort of
their cells."""
import time

import numpy as np
import pytest

import synth
from _cases import base_config, neutral_gas

pytestmark = pytest.mark.gpu


def _rt(n):
    from paper_2404_17630_gb300 import RT, make_config
    mesh = synth.cartesian_mesh(n, 10.0)
    cfg = base_config(chem_mode=0)
    rt = RT(make_config(**cfg), mesh)
    rt.set_gas(*neutral_gas(mesh.n_cells, 1e-3))
    return rt, mesh, cfg


@pytest.mark.parametrize("n_src", [1, 3, 15, 16, 17, 500, 4096, 20000])
def test_rates(n_src):
    rt, mesh, cfg = _rt(16)
    C = mesh.n_cells
    rng = np.random.default_rng(n_src)
    for _ in range(2):   # the second set replaces the first
        cells = rng.integers(0, C, n_src)
        Q = 10 ** rng.uniform(47, 50, (n_src, 3))
        rt.set_radiation(np.zeros((3, C)))
        rt.set_sources(cells, Q)
        dt = rt.max_dt()
        rt.thermochemistry(dt)
        rt.sync()
        S = np.zeros((3, C))
        for b in range(3):
            np.add.at(S[b], cells, Q[:, b])
        ref = S * dt / (mesh.volume * cfg["unit_length_cm"] ** 3)
        assert np.abs(rt.fields()["N"] - ref).max() <= 1e-14 * ref.max()


def test_out_of_range():
    from paper_2404_17630_gb300.rt import RTError
    rt, mesh, cfg = _rt(16)
    for n_src in (2, 3000):
        cells = np.arange(n_src)
        cells[1] = mesh.n_cells
        with pytest.raises(RTError, match="source 1 in cell 4096 out of range"):
            rt.set_sources(cells, np.ones((n_src, 3)))


def test_time_of_many():
    rt, mesh, cfg = _rt(80)
    rng = np.random.default_rng(1)
    cells = rng.permutation(mesh.n_cells)
    Q = rng.uniform(1, 2, (mesh.n_cells, 3)) * 1e48
    def best(f):
        t = []
        for _ in range(4):
            t0 = time.perf_counter()
            f()
            t.append(time.perf_counter() - t0)
        return min(t)
    assert best(lambda: rt.set_sources(cells, Q)) < best(lambda: np.argsort(cells, kind="stable"))
