"""A mesh that rt_init_mesh refuses (a bad face, a bad volume, a cell without faces, a
singular least-squares matrix) leaves no device memory with the context, which
takes a good mesh afterwards."""
import dataclasses

import numpy as np
import pytest

from _cases import voronoi_case

pytestmark = pytest.mark.gpu


def _bad(mesh, how):
    if how == "face":
        left = mesh.left.copy()
        left[7] = mesh.n_cells
        return dataclasses.replace(mesh, left=left)
    if how == "volume":
        return dataclasses.replace(mesh, volume=np.where(np.arange(mesh.n_cells) == 7, -1.0, mesh.volume))
    if how == "faces":   # every face of cell 7 goes to another cell
        l, r = (np.where(a == 7, np.where(b == 8, 9, 8), a).astype(np.int32) for a, b in
                ((mesh.left, mesh.right), (mesh.right, mesh.left)))
        return dataclasses.replace(mesh, left=l, right=r)
    return dataclasses.replace(mesh, area=np.where((mesh.left == 7) | (mesh.right == 7), 0.0, mesh.area))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("how,word", [("face", "face 7 joins"), ("volume", "cell 7 has volume"),
                                      ("faces", "cell 7 has no faces"), ("matrix", "singular")])
def test_no_memory_is_kept(how, word, precision):
    import torch
    from paper_2404_17630_gb300 import RT, make_config
    from paper_2404_17630_gb300.rt import RTError
    mesh, cfg, st = voronoi_case(n=24, seed=5)
    made = make_config(precision=precision, **cfg)
    good = RT(made, mesh)   # the library's kernels are loaded
    dt = 0.5 * good.max_dt()
    good.step(dt, 1)
    good.sync()
    rt = RT(made)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        with pytest.raises(RTError, match=word):
            rt.init_mesh(_bad(mesh, how))
        assert free - torch.cuda.mem_get_info()[0] < 4 << 20
    rt.init_mesh(mesh)
    rt.step(dt, 1)
    rt.sync()
