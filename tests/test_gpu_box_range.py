"""Periodic boxes at the end of the range: an infinite side has no minimum image, and
the mesh is refused (the allocation-free gradients mark their cells); a side of 1e308
is as good as none."""
import numpy as np
import pytest

from _cases import voronoi_case

pytestmark = pytest.mark.gpu


def _inner(box):
    """The gradients of the cells away from the box's sides."""
    from paper_2404_17630_gb300 import RT, make_config
    mesh, cfg, st = voronoi_case(n=8, seed=5)
    rt = RT(make_config(**dict(cfg, box=box)), mesh)
    rt.set_gas(st["nH"], st["x5"], st["T"])
    rt.set_radiation(st["N"], st["fr"] * cfg["c_red"])
    inside = np.ones(mesh.n_cells, bool)
    for c in (mesh.cx, mesh.cy, mesh.cz):
        inside &= (c > 3.5) & (c < 6.5)
    assert inside.any()
    return rt.gradients()[inside]


def test_infinite_box_is_refused():
    from paper_2404_17630_gb300.rt import RTError
    with pytest.raises(RTError, match="singular"):
        _inner(np.inf)


def test_infinite_box_marks_the_cells():
    from test_zz_no_alloc import _from_mesh, _noalloc
    mesh, cfg, st = voronoi_case(n=8, seed=5)
    G, bad = _noalloc(_from_mesh(mesh), st["N"], st["fr"], 3, 2, 1, 1e-5, np.inf)
    assert bad == 1 and (G == 0).all()


def test_huge_box():
    assert np.array_equal(_inner(1e308), _inner(0.0))
