"""Where many steps per launch are the automatic choice they are not slower
than the launch-per-step kernels (tuning variant 3), with few and with many
receivers."""
import time

import numpy as np
import pytest

from helpers import Case, DeviceShot

pytestmark = pytest.mark.gpu


def _best_ms(fn):
    import torch

    fn()
    best = float("inf")
    for _ in range(5):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        fn()
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t0)
    return best * 1e3


def _spans_and_launches(r, fn):
    import paper_1603_03971_gb300 as rtm

    out = []
    try:
        for variant in (0, 3):
            rtm.set_tuning(r, 0, variant)
            out.append(_best_ms(fn))
    finally:
        rtm.set_tuning(r, 0, 0)
    return out


# launches and waits of a few microseconds each on a shared machine: a quarter
# is well above their spread, and far below what a wrong choice costs (2 to 12 x)
SLACK = 1.25


def _off_grid(nx, ny, nz, nb, storage, ckpt, nrec):
    import torch

    import paper_1603_03971_gb300 as rtm

    case = Case(nx=nx, ny=ny, nz=nz, nb=nb, nt=60, storage=storage, ckpt_every=ckpt)
    g = DeviceShot(case)
    p = g.p.copy(nrec=nrec)
    ws = rtm.alloc_workspace(p)
    rng = np.random.default_rng(0)
    pts = rng.uniform((0.1, 0.1, 2.1), (nx - 1.1, ny - 1.1, 2.9), (nrec, 3))
    taps = rtm.offgrid_taps(p, (nx / 2 + 0.4, ny / 2 + 0.3, 3.5), pts, "cuda")
    dobs = torch.from_numpy(rng.normal(size=(60, nrec)).astype(np.float32)).cuda()
    img = torch.zeros(rtm.model_shape(p), device="cuda")
    data = torch.empty((60, nrec), device="cuda")
    return lambda: rtm.shot_offgrid(p, g.c, taps, dobs, ws, img, data=data)


@pytest.mark.parametrize("nrec", [1, 168, 672, 3969])
def test_off_grid_receivers_of_a_small_grid(nrec):
    spans, launches = _spans_and_launches(4, _off_grid(28, 24, 20, 6, "ckpt", 10, nrec))
    assert spans <= SLACK * launches


@pytest.mark.parametrize("grid", [(28, 24, 20, 6), (64, 64, 64, 20)])
@pytest.mark.parametrize("nrec", [256, 1024, 3969])
def test_off_grid_receivers_under_binomial_checkpointing(grid, nrec):
    spans, launches = _spans_and_launches(4, _off_grid(*grid, "revolve", 10, nrec))
    assert spans <= SLACK * launches
