"""Several contexts in one process: the staged gradient kernel's shared-memory
allowance is one attribute of the kernel, so a context for a mesh with small
blocks, made after one whose blocks need more, must leave the earlier one
usable."""
import numpy as np
import pytest

import synth
from _cases import EPS3, SIGMA3, neutral_gas

pytestmark = pytest.mark.gpu


def _context(mesh):
    from paper_2404_17630_gb300 import RT, make_config
    C = mesh.n_cells
    rt = RT(make_config(n_bins=3, precision="mixed", gather_sum=1, box=10.0, y_he=synth.helium_ratio(0.24),
                        sigma=SIGMA3, eps=EPS3), mesh)
    rng = np.random.default_rng(3)
    rt.set_gas(*neutral_gas(C, 1e-3))
    rt.set_radiation(rng.uniform(0, 1e-4, (3, C)))
    return rt


def test_contexts_with_larger_and_smaller_gradient_blocks():
    big = _context(synth.voronoi_mesh(12, 10.0, 0.3, seed=1))      # ~500 records per block of cells
    dt = big.max_dt()
    big.step(dt, 1)
    big.sync()
    alone = big.fields()
    again = _context(synth.voronoi_mesh(12, 10.0, 0.3, seed=1))
    small = _context(synth.cartesian_mesh(8, 10.0))                # 192
    small.step(0.5 * small.max_dt(), 1)
    small.sync()
    again.step(dt, 1)
    again.sync()
    got = again.fields()
    for k in ("N", "F", "x5", "T"):
        assert np.array_equal(got[k], alone[k]), k
