"""Where many steps per launch are the automatic choice they are not slower
than the launch-per-step kernels (tuning variant 3), with few and with many
receivers; and what a step's receivers cost the launches."""
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


@pytest.mark.parametrize("nrec", [256, 1024])
def test_a_few_receivers_off_the_grid_hardly_cost_a_launch_per_step(nrec):
    """On a grid above the spans' sizes a step is two stencil launches of 30 us;
    1024 receivers are 0.5 M of its taps, 2 us at the L2 cache's rate."""
    one, many = (_best_ms(_off_grid(150, 131, 117, 21, "all", 0, n)) for n in (1, nrec))
    assert many <= SLACK * one


@pytest.mark.parametrize("grid", [(28, 24, 20, 6), (64, 64, 64, 20), (96, 90, 80, 16)])
@pytest.mark.parametrize("planes", [1, 6, 1000])
def test_receivers_on_the_grid(grid, planes):
    import torch

    import paper_1603_03971_gb300 as rtm

    nx, ny, nz, nb = grid
    g = DeviceShot(Case(nx=nx, ny=ny, nz=nz, nb=nb, nt=60, storage="ckpt", ckpt_every=20))
    z, y, x = np.meshgrid(np.arange(min(planes, nz)), np.arange(ny), np.arange(nx), indexing="ij")
    rec = torch.from_numpy(np.stack([x, y, z], axis=-1).reshape(-1, 3).astype(np.int32)).cuda()
    p = g.p.copy(nrec=rec.shape[0])
    ws = rtm.alloc_workspace(p)
    dobs = torch.randn((60, p.nrec), device="cuda")
    img = torch.zeros(rtm.model_shape(p), device="cuda")
    spans, launches = _spans_and_launches(4, lambda: rtm.shot(p, g.c, rec, dobs, ws, img))
    assert spans <= SLACK * launches


def test_a_brick_over_its_list_takes_all_receivers():
    import torch

    import paper_1603_03971_gb300 as rtm

    # 16250 receivers in a cube of 25 x 25 x 26 cells: several thousand in a
    # brick of 104^3, which lists 2048
    case = Case(nx=64, ny=64, nz=64, nb=20, nt=9, src=(32, 32, 40))
    g = DeviceShot(case)
    z, y, x = np.meshgrid(np.arange(26), np.arange(25), np.arange(25), indexing="ij")
    rec = torch.from_numpy(np.stack([x, y, z], axis=-1).reshape(-1, 3).astype(np.int32)).cuda()
    p = g.p.copy(nrec=rec.shape[0])
    ws = rtm.alloc_workspace(p)
    dobs = torch.from_numpy(case.d_obs(p.nrec).astype(np.float32)).cuda()
    out = []
    for variant in (0, 3):
        rtm.set_tuning(4, 0, variant)
        try:
            img = torch.zeros(rtm.model_shape(p), device="cuda")
            data = torch.empty((p.nt, p.nrec), device="cuda")
            rtm.shot(p, g.c, rec, dobs, ws, img, data=data)
            rtm.check(ws)
        finally:
            rtm.set_tuning(4, 0, 0)
        out.append((img.cpu().numpy(), data.cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert np.any(out[0][0] != 0)
