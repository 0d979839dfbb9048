"""Receivers that share a cell: the spans sum their data before they add it to
the field, the launch-per-step kernels add each by itself, so the images differ
by roundings only and the data (gathered, not summed) are equal."""
import numpy as np
import pytest

from helpers import Case, DeviceShot, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [4, 8])
@pytest.mark.parametrize("copies", [2, 5])
def test_receivers_of_one_cell(r, copies):
    import torch

    import paper_1603_03971_gb300 as rtm

    case = Case(r=r, nt=23)
    g = DeviceShot(case)
    rec = torch.from_numpy(np.repeat(g.rec_np, copies, axis=0)).cuda()
    p = g.p.copy(nrec=rec.shape[0])
    ws = rtm.alloc_workspace(p)
    dobs = torch.from_numpy(case.d_obs(p.nrec).astype(np.float32)).cuda()
    out = []
    for variant in (0, 3):
        rtm.set_tuning(r, 0, variant)
        try:
            img = torch.zeros(rtm.model_shape(p), device="cuda")
            data = torch.empty((p.nt, p.nrec), device="cuda")
            rtm.shot(p, g.c, rec, dobs, ws, img, data=data)
            rtm.check(ws)
        finally:
            rtm.set_tuning(r, 0, 0)
        out.append((img.cpu().numpy(), data.cpu().numpy()))
    assert np.array_equal(out[0][1], out[1][1])
    # per step up to `copies` roundings of the sums of each path, 23 steps
    assert rel_l2(out[0][0], out[1][0]) <= 2 * copies * 23 * 2.0 ** -24
