"""Shots on a stream that owns a few of the device's SMs (a green context):
grids that take many steps per launch on the whole device are tiled for those
SMs, or take the launches, with the same results."""
import ctypes
from types import SimpleNamespace

import numpy as np
import pytest

from helpers import Case, DeviceShot

pytestmark = pytest.mark.gpu

SM, DEFAULT_STREAM, NON_BLOCKING = 1, 1, 1


class Resource(ctypes.Structure):  # CUdevResource: a type and a union, 144 bytes
    _fields_ = [("type", ctypes.c_int), ("padding", ctypes.c_ubyte * 92),
                ("sm_count", ctypes.c_uint), ("rest", ctypes.c_ubyte * 44)]


def _few_sms(count):
    """(stream handle, its SMs, destroy) of a green context of about `count` SMs."""
    cu = ctypes.CDLL("libcuda.so.1")

    def call(name, *args):
        if getattr(cu, name)(*args) != 0:
            pytest.skip("%s: green contexts are not available here" % name)
    dev, res, group, rest = ctypes.c_int(), Resource(), Resource(), Resource()
    n, desc, ctx, stream = ctypes.c_uint(1), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    call("cuDeviceGet", ctypes.byref(dev), 0)
    call("cuDeviceGetDevResource", dev, ctypes.byref(res), SM)
    call("cuDevSmResourceSplitByCount", ctypes.byref(group), ctypes.byref(n), ctypes.byref(res),
         ctypes.byref(rest), ctypes.c_uint(0), ctypes.c_uint(count))
    call("cuDevResourceGenerateDesc", ctypes.byref(desc), ctypes.byref(group), ctypes.c_uint(1))
    call("cuGreenCtxCreate", ctypes.byref(ctx), desc, dev, ctypes.c_uint(DEFAULT_STREAM))
    call("cuGreenCtxStreamCreate", ctypes.byref(stream), ctx, ctypes.c_uint(NON_BLOCKING), 0)

    def destroy():
        cu.cuStreamDestroy_v2(stream)
        cu.cuGreenCtxDestroy(ctx)
    return stream.value, group.sm_count, destroy


@pytest.mark.parametrize("grid", [(28, 24, 20, 6), (64, 64, 64, 20)])
def test_shot_on_a_few_sms(grid):
    import torch

    import paper_1603_03971_gb300 as rtm

    nx, ny, nz, nb = grid
    case = Case(nx=nx, ny=ny, nz=nz, nb=nb, nt=20, storage="ckpt", ckpt_every=8)
    g = DeviceShot(case)
    dobs = torch.from_numpy(case.d_obs(g.nrec).astype(np.float32)).cuda()

    def shot(stream):
        img = torch.zeros(rtm.model_shape(g.p), device="cuda")
        data = torch.empty((g.p.nt, g.nrec), device="cuda")
        torch.cuda.synchronize()
        rtm.shot(g.p, g.c, g.rec, dobs, g.ws, img, data=data, stream=stream)
        rtm.check(g.ws, stream=stream)
        return img.cpu().numpy(), data.cpu().numpy()
    want = shot(None)
    handle, sms, destroy = _few_sms(16)
    assert 0 < sms < torch.cuda.get_device_properties(0).multi_processor_count
    try:
        got = shot(torch.cuda.ExternalStream(handle))
    finally:
        torch.cuda.synchronize()
        destroy()
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("handle", [0, 1, 2, None])  # NULL, legacy, per thread, a created one
def test_special_streams_take_many_steps_per_launch(handle):
    import torch

    import paper_1603_03971_gb300 as rtm

    g = DeviceShot(Case(nt=20, storage="all"))
    dobs = torch.from_numpy(g.case.d_obs(g.nrec).astype(np.float32)).cuda()
    img = torch.zeros(rtm.model_shape(g.p), device="cuda")
    stream = torch.cuda.Stream() if handle is None else SimpleNamespace(cuda_stream=handle)
    torch.cuda.synchronize()
    rtm.reset_stats()
    rtm.shot(g.p, g.c, g.rec, dobs, g.ws, img, stream=stream)
    torch.cuda.synchronize()
    assert rtm.stats()["launches"] < 20  # 2 x 20 steps
    rtm.check(g.ws)
