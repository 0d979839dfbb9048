"""The training kernels at the edges of their tiles and slabs: one latent
voxel, latent counts just below and above a 32-voxel slab and a 128-voxel
tile, sides of one latent voxel, and a batch whose samples start off a 16-byte
boundary; loss and gradient against the FP64 oracle with its bfloat16
roundings."""
import numpy as np
import pytest

import rtm_inputs
from helpers import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,offset", [
    ((4, 4, 4), 0), ((4, 4, 124), 0), ((4, 44, 12), 0), ((20, 20, 20), 0), ((16, 20, 28), 1),
    ((24, 28, 32), 0)])
def test_training_gradient_at_tile_edges(shape, offset):
    import torch

    from oracle import ae as oae
    from paper_1603_03971_gb300 import codec

    batch = rtm_inputs.standard_normal((2,) + shape, seed=3).astype(np.float32) * 1e-3
    params = rtm_inputs.ae_init_params(4)
    for k in ("b1", "b2", "b3", "b4"):
        params[k] = rtm_inputs.standard_normal(params[k].shape, seed=5) * 0.05
    P = torch.from_numpy(oae.flatten(params).astype(np.float32)).cuda()
    buf = torch.empty(batch.size + offset, device="cuda")  # `offset` floats off the boundary
    x = buf[offset:].view(batch.shape)
    x.copy_(torch.from_numpy(batch))
    grad = torch.zeros_like(P)
    loss = codec.train_step(P, None, None, 0, 0.0, x, codec.alloc_workspace(shape), grad_out=grad)
    L_ref, g_ref = 0.0, None
    ref = {k: v.astype(np.float32).astype(np.float64) for k, v in params.items()}
    for b in batch:
        s = b.astype(np.float64)
        L, g = oae.loss_and_grads(ref, s / oae.rms(s), bf16=True, bf16_grads=True, scale=0.5)
        L_ref += 0.5 * L
        g_ref = g if g_ref is None else {k: g_ref[k] + g[k] for k in g}
    assert float(loss.item()) == pytest.approx(L_ref, rel=1e-4)
    got = oae.unflatten(grad.cpu().numpy().astype(np.float64))
    for k in oae.PARAM_ORDER:  # the codec's gradient tolerance: stored bf16 values one step apart
        assert rel_l2(got[k], g_ref[k]) <= 5e-3, k
