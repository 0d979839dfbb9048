"""Kernels that walk a grid by rows of x, at rows shorter than a warp, of a
whole warp, and longer, with the model's bad values found wherever they lie."""
import numpy as np
import pytest

from helpers import Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["v", "v2"])
@pytest.mark.parametrize("nx,ny,nz,nb", [
    (2, 3, 5, 1), (6, 1, 9, 1), (4, 7, 3, 6), (20, 5, 1, 4), (28, 6, 7, 2), (31, 9, 4, 10),
    (34, 8, 3, 1), (131, 5, 6, 2)])
def test_model_prep_is_exact(nx, ny, nz, nb, kind):
    import torch

    import paper_1603_03971_gb300 as rtm

    nx += -(nx + 2 * nb) % 4
    case = Case(nx=nx, ny=ny, nz=nz, nb=nb, src=(0, 0, 0))
    p = case.params()
    v = np.random.default_rng(nx).uniform(1500, 4500, (nz, ny, nx)).astype(np.float32)
    if kind == "v2":
        v = v * v
    ws = rtm.alloc_workspace(p)
    c = rtm.model_prep(p, torch.from_numpy(v).cuda(), ws, kind=kind).cpu().numpy()
    v2 = v if kind == "v2" else v * v
    ref = np.pad(v2 * np.float32(p.dt * p.dt), nb, mode="edge")
    assert np.array_equal(c, ref)
    for bad in (0, v.size // 2, v.size - 1):
        w = v.copy()
        w.flat[bad] = np.nan
        with pytest.raises(rtm.RtmError):
            rtm.model_prep(p, torch.from_numpy(w).cuda(), ws, kind=kind)
            rtm.check(ws)
