"""A padded y side of more rows than a grid of 8-row tiles has blocks for: the
automatic choice runs it, with the results of the 16-row tiles."""
import numpy as np
import pytest

from helpers import Case, DeviceShot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [4, 8])
@pytest.mark.parametrize("ny", [65535 * 8 + 1, 65535 * 16])
def test_long_y_side_runs(r, ny):
    import torch

    import paper_1603_03971_gb300 as rtm

    case = Case(nx=4, ny=4, nz=2, nb=0, r=r, nt=4, src=(1, 2, 1))
    g = DeviceShot(case)
    p = g.p.copy(ny=ny, nrec=3)
    vel = torch.from_numpy(np.random.default_rng(1).uniform(1500, 3000, (2, ny, 4))
                           .astype(np.float32)).cuda()
    ws = rtm.alloc_workspace(p)
    c = rtm.model_prep(p, vel, ws)
    rec = torch.tensor([[0, 0, 0], [2, 5, 1], [3, ny - 1, 1]], dtype=torch.int32, device="cuda")
    dobs = torch.ones((p.nt, 3), device="cuda")
    out = []
    for variant in (0, 2):
        rtm.set_tuning(r, 0, variant)
        try:
            img = torch.zeros(rtm.model_shape(p), device="cuda")
            data = torch.empty((p.nt, 3), device="cuda")
            rtm.shot(p, c, rec, dobs, ws, img, data=data)
            rtm.check(ws)
        finally:
            rtm.set_tuning(r, 0, 0)
        out.append((img.cpu().numpy(), data.cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert np.any(out[0][0] != 0)
