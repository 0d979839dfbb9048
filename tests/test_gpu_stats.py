"""Counters of the stencil steps: many steps per launch book each step under
the mode that it ran in, as the launch-per-step kernels do."""
import numpy as np
import pytest

from helpers import Case, DeviceShot

pytestmark = pytest.mark.gpu


def _modes(r, variant, fn):
    import paper_1603_03971_gb300 as rtm

    rtm.set_tuning(r, 0, variant)
    try:
        rtm.reset_stats()
        fn()
        s = rtm.stats()
    finally:
        rtm.set_tuning(r, 0, 0)
    return s["launches"], {k: v["launches"] for k, v in s["stencil"].items()}


@pytest.mark.parametrize("storage,ckpt,every", [
    ("all", 0, 4), ("all", 0, 1), ("ckpt", 9, 4), ("revolve", 3, 3), ("decimated", 0, 3),
    ("decimated", 7, 2), ("boundary", 0, 2)])
@pytest.mark.parametrize("offgrid", [False, True])
def test_steps_are_booked_by_mode(storage, ckpt, every, offgrid):
    import torch

    import paper_1603_03971_gb300 as rtm

    case = Case(nt=22, storage=storage, ckpt_every=ckpt, image_every=every)
    g = DeviceShot(case)
    dobs = torch.from_numpy(case.d_obs(g.nrec).astype(np.float32)).cuda()
    img = torch.zeros(rtm.model_shape(g.p), device="cuda")
    pts = g.rec_np + 0.3
    taps = rtm.offgrid_taps(g.p, (13.6, 12.2, 3.5), pts, "cuda") if offgrid else None

    def run():
        if offgrid:
            rtm.shot_offgrid(g.p, g.c, taps, dobs, g.ws, img)
        else:
            rtm.shot(g.p, g.c, g.rec, dobs, g.ws, img)
        rtm.check(g.ws)
    few, spans = _modes(4, 0, run)
    many, steps = _modes(4, 3, run)
    assert few < many  # the automatic choice took the other path
    assert spans == steps


def test_gradient_steps_are_booked_by_mode():
    case = Case(nt=22, storage="ckpt", ckpt_every=6)
    g = DeviceShot(case, want_grad=True, squared=True)
    resid = case.d_obs(g.nrec)

    def run():
        g.forward()
        g.grad(resid)
    few, spans = _modes(4, 0, run)
    many, steps = _modes(4, 3, run)
    assert few < many and spans == steps
