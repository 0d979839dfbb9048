"""Timeout paths of the kernels that take many steps per launch and of the
radius-8 stencil with two rows per thread, without a fault (as
test_gpu_stall.py for the other kernels): an armed wait runs out after about
2 s, the call's status word reads RTM_ERR_TIMEOUT, every block has left, and
the next call is exact."""
import time

import numpy as np
import pytest

from helpers import Case, DeviceShot

pytestmark = pytest.mark.gpu


def _stalled(kernel, plane, call, check):
    from paper_1603_03971_gb300 import _lib
    import paper_1603_03971_gb300 as rtm

    rtm.set_test_stall(kernel, plane)
    try:
        t0 = time.time()
        with pytest.raises(_lib.RtmError) as e:
            call()
            check()
        assert e.value.code == 5  # RTM_ERR_TIMEOUT
        assert 1.5 < time.time() - t0 < 60
    finally:
        rtm.set_test_stall(kernel, -1)


@pytest.mark.parametrize("r", [4, 8])
@pytest.mark.parametrize("plane", [0, 2, 100])  # the last step of a span, one before, the first
def test_span_wait_timeout_is_reported_not_hung(r, plane):
    import torch

    import paper_1603_03971_gb300 as rtm

    # several spans per call: those after the stalled one leave at once
    case = Case(r=r, nt=12, storage="ckpt", ckpt_every=4)
    g = DeviceShot(case)
    rd = torch.from_numpy(case.d_obs(g.nrec).astype(np.float32)).cuda()

    def forward():
        data = torch.empty((g.p.nt, g.nrec), device="cuda")
        rtm.forward(g.p, g.c, g.rec, g.ws, data=data)
        return data

    def backward():
        img = torch.zeros(rtm.model_shape(g.p), device="cuda")
        rtm.backward_image(g.p, g.c, g.rec, rd, g.ws, img)
        return img
    data, img = forward(), backward()
    rtm.check(g.ws)
    for call, want in ((forward, data), (backward, img)):
        forward()
        rtm.check(g.ws)
        _stalled(rtm.STALL_SPAN, plane, call, lambda: rtm.check(g.ws))
        assert torch.equal(forward(), data)
        assert torch.equal(backward(), img)
        rtm.check(g.ws)


@pytest.mark.parametrize("plane", [0, 1, 2, 9])
def test_two_row_stencil_wait_timeout_is_reported_not_hung(plane):
    import torch

    import paper_1603_03971_gb300 as rtm

    g = DeviceShot(Case(r=8, nt=6, storage="ckpt", ckpt_every=3))
    rtm.set_tuning(8, 0, 2)
    try:
        def forward():
            data = torch.empty((g.p.nt, g.nrec), device="cuda")
            rtm.forward(g.p, g.c, g.rec, g.ws, data=data)
            return data
        want = forward()
        rtm.check(g.ws)
        _stalled(rtm.STALL_ROWS, plane, forward, lambda: rtm.check(g.ws))
        assert torch.equal(forward(), want)
        rtm.check(g.ws)
    finally:
        rtm.set_tuning(8, 0, 0)
