"""Several time steps per launch (grids whose bricks fit one per SM, the
automatic choice) against the launch-per-step kernels (tuning variant 3): the
same operations per cell in the same order, so every output is equal bit for
bit, at ragged and tiny grids, bricks with one and with several rounds of
items, all storages, receivers on and off the grid, and more receivers in a
brick than its list holds."""
import numpy as np
import pytest

from helpers import Case, DeviceShot, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _reset_tuning():
    import paper_1603_03971_gb300 as rtm

    yield
    for r in (4, 8):
        rtm.set_tuning(r, 0, 0)


def _both(r, fn):
    """fn() under the automatic choice and under the launch-per-step kernels."""
    import paper_1603_03971_gb300 as rtm

    rtm.set_tuning(r, 0, 0)
    rtm.reset_stats()
    a = fn()
    few = rtm.stats()["launches"]
    rtm.set_tuning(r, 0, 3)
    rtm.reset_stats()
    b = fn()
    many = rtm.stats()["launches"]
    rtm.set_tuning(r, 0, 0)
    assert few < many  # the automatic choice did take the other path
    return a, b


def _shot(case, rec=None):
    import torch

    import paper_1603_03971_gb300 as rtm

    g = DeviceShot(case)
    recs = g.rec if rec is None else torch.from_numpy(rec).cuda()
    p = g.p.copy(nrec=recs.shape[0])
    ws = rtm.alloc_workspace(p)
    dobs = torch.from_numpy(case.d_obs(p.nrec).astype(np.float32)).cuda()

    def run():
        img = torch.zeros(rtm.model_shape(p), device="cuda")
        data = torch.empty((p.nt, p.nrec), device="cuda")
        rtm.shot(p, g.c, recs, dobs, ws, img, data=data)
        rtm.check(ws)
        return img.cpu().numpy(), data.cpu().numpy()
    return run


SHAPES = {
    "tiny": dict(nx=28, ny=24, nz=20, nb=6),
    "thin": dict(nx=4, ny=3, nz=5, nb=8, src=(2, 1, 2), rec_stride=1),
    "ragged": dict(nx=102, ny=43, nz=37, nb=9),
    "rounds": dict(nx=110, ny=97, nz=88, nb=9),  # more items than threads in a brick (too large at r = 8)
}


@pytest.mark.parametrize("r,shape", [(r, s) for r in (4, 8) for s in SHAPES if (r, s) != (8, "rounds")])
@pytest.mark.parametrize("storage,ckpt,every", [
    ("all", 0, 1), ("all", 0, 3), ("ckpt", 9, 1), ("ckpt", 40, 2), ("revolve", 3, 2),
    ("decimated", 0, 3), ("decimated", 5, 2), ("boundary", 0, 2)])
def test_shot_equals_the_launches(r, shape, storage, ckpt, every):
    if storage == "boundary" and shape == "thin":
        pytest.skip("boundary storage needs model sides above 2 r")
    case = Case(r=r, nt=23, storage=storage, ckpt_every=ckpt, image_every=every, **SHAPES[shape])
    if storage == "boundary" and min(case.nx, case.ny, case.nz) <= 2 * r:
        pytest.skip("boundary storage needs model sides above 2 r")
    (img, data), (img_ref, data_ref) = _both(r, _shot(case))
    assert np.array_equal(data, data_ref)
    assert np.array_equal(img, img_ref)


@pytest.mark.parametrize("r", [4, 8])
@pytest.mark.parametrize("storage,ckpt", [("all", 0), ("ckpt", 7)])
def test_gradient_illumination_and_source_trace_equal_the_launches(r, storage, ckpt):
    import torch

    import paper_1603_03971_gb300 as rtm

    case = Case(r=r, nt=23, storage=storage, ckpt_every=ckpt, **SHAPES["ragged"])
    gg = DeviceShot(case, want_grad=True, squared=True)
    resid = case.d_obs(gg.nrec)

    def grad():
        data, last = gg.forward(keep_last=True)
        return gg.grad(resid).cpu().numpy(), data.cpu().numpy(), last.cpu().numpy()
    a, b = _both(r, grad)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    g = DeviceShot(case)
    rd = torch.from_numpy(resid.astype(np.float32)).cuda()

    def image():
        g.forward()
        img, adj = g.backward_image(resid, src_adj=True)
        img2, ill = torch.zeros_like(img), torch.zeros_like(img)
        g.forward()
        rtm.backward_image_illum(g.p, g.c, g.rec, rd, g.ws, img2, ill)
        return [t.cpu().numpy() for t in (img, adj, img2, ill)]
    a, b = _both(r, image)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def test_more_receivers_than_a_brick_lists():
    # every cell of six planes: about 3000 receivers in some bricks of 104^3
    z, y, x = np.meshgrid(np.arange(6), np.arange(64), np.arange(64), indexing="ij")
    rec = np.stack([x.ravel(), y.ravel(), z.ravel()], axis=1).astype(np.int32)
    case = Case(nx=64, ny=64, nz=64, nb=20, nt=12, src=(32, 32, 4))
    (img, data), (img_ref, data_ref) = _both(4, _shot(case, np.ascontiguousarray(rec)))
    assert np.array_equal(data, data_ref)
    assert np.array_equal(img, img_ref)


@pytest.mark.parametrize("r", [4, 8])
def test_off_grid_shot_matches_the_launches(r):
    import torch

    import paper_1603_03971_gb300 as rtm

    case = Case(r=r, nt=23, **SHAPES["ragged"])
    g = DeviceShot(case)
    pts = g.rec_np.astype(np.float64) + np.random.default_rng(3).uniform(-0.4, 0.9, g.rec_np.shape)
    taps = rtm.offgrid_taps(g.p, (50.3, 20.6, 3.5), pts, "cuda")
    dobs = torch.from_numpy(case.d_obs(g.nrec).astype(np.float32)).cuda()

    def run():
        img = torch.zeros(rtm.model_shape(g.p), device="cuda")
        data = torch.empty((g.p.nt, g.nrec), device="cuda")
        rtm.shot_offgrid(g.p, g.c, taps, dobs, g.ws, img, data=data)
        rtm.check(g.ws)
        return img.cpu().numpy(), data.cpu().numpy()
    (img, data), (img_ref, data_ref) = _both(r, run)
    # the taps of neighbouring receivers are summed in another order: each
    # cell adds at most 512 FP32 terms per step, sqrt(512 * 23) roundings
    assert rel_l2(data, data_ref) <= 7e-6
    assert rel_l2(img, img_ref) <= 7e-6


@pytest.mark.parametrize("r,storage,ckpt,nrec", [
    (4, "all", 0, 1), (4, "ckpt", 9, 6000), (4, "revolve", 3, 700), (8, "revolve", 3, 6000),
    (4, "boundary", 0, 700)])
def test_off_grid_receivers_beyond_a_blocks_tables(r, storage, ckpt, nrec):
    """One receiver, a few per block and more than a block keeps tap tables
    for (32), also where no padded fields are left to scatter into."""
    import torch

    import paper_1603_03971_gb300 as rtm

    case = Case(r=r, nt=23, storage=storage, ckpt_every=ckpt, nx=46, ny=43, nz=37, nb=9)
    rng = np.random.default_rng(5)
    pts = rng.uniform((0, 0, 1), (45, 42, 4.5), (nrec, 3))
    g = DeviceShot(case)
    p = g.p.copy(nrec=nrec)
    ws = rtm.alloc_workspace(p)
    taps = rtm.offgrid_taps(p, (20.3, 20.6, 3.5), pts, "cuda")
    dobs = torch.from_numpy(case.d_obs(nrec).astype(np.float32)).cuda()

    def run():
        img = torch.zeros(rtm.model_shape(p), device="cuda")
        data = torch.empty((p.nt, nrec), device="cuda")
        rtm.shot_offgrid(p, g.c, taps, dobs, ws, img, data=data)
        rtm.check(ws)
        return img.cpu().numpy(), data.cpu().numpy()
    (img, data), (img_ref, data_ref) = _both(r, run)
    # as above, with the terms of a cell: each of its 8^3 neighbours' receivers
    # (6000 over 45 x 42 x 3.5: about 0.9 per cell, 512 taps each way)
    assert rel_l2(data, data_ref) <= 7e-6
    assert rel_l2(img, img_ref) <= 7e-6


def test_receivers_outside_are_reported_and_skipped():
    import paper_1603_03971_gb300 as rtm

    case = Case(nt=12, extra_rec=np.array([[500, 1, 2], [-900, 0, 0]], np.int32))
    g = DeviceShot(case)
    with pytest.raises(rtm.RtmError) as e:
        g.forward()
    assert e.value.code == 1
