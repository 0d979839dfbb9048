"""Encoding and decoding ask for no more workspace than before training kept
packed weights and normalised inputs in it."""
import numpy as np
import pytest

import rtm_inputs

pytestmark = pytest.mark.gpu


def _bytes(shape, training):
    """256 bytes of status and scalars, then 256-byte aligned parts: h1, latent,
    g1, y, gy, ga3, latent gradient, ga1, gradient; behind them xq and the packed weights."""
    n = int(np.prod(shape))
    nh, nl = n // 8, n // 64
    parts = [64 * nh, 32 * nl, 64 * nh, 4 * n, 2 * n, 64 * nh, 32 * nl, 64 * nh, 4 * 47185]
    if training:
        parts += [16 * nh, 16 * (27 * 64 + 32 * 128 + 64 * 64 + 14 * 128)]
    return 256 + sum(-(-p // 256) * 256 for p in parts)


def test_coding_runs_in_the_workspace_it_needs():
    import torch

    from paper_1603_03971_gb300 import _lib, codec

    shape = (24, 20, 28)
    P = torch.from_numpy(rtm_inputs.ae_flat(rtm_inputs.ae_init_params(3)).astype(np.float32)).cuda()
    s = torch.from_numpy(rtm_inputs.standard_normal(shape, 71, np.float32)).cuda()
    full = codec.alloc_workspace(shape)
    assert full.numel() == _bytes(shape, True)
    lat, scale = codec.encode(P, s, full)
    out = codec.decode(P, lat, scale, full)
    small = torch.empty(_bytes(shape, False), dtype=torch.uint8, device="cuda")
    lat2, scale2 = codec.encode(P, s, small)
    assert torch.equal(lat2, lat) and torch.equal(scale2, scale)
    assert torch.equal(codec.decode(P, lat, scale, small), out)
    for call in (lambda w: codec.encode(P, s, w), lambda w: codec.decode(P, lat, scale, w)):
        with pytest.raises(_lib.RtmError) as e:
            call(small[:-256])
        assert e.value.code == 3  # RTM_ERR_WORKSPACE
    with pytest.raises(_lib.RtmError) as e:
        codec.train_step(P, None, None, 0, 0.0, s[None].contiguous(), small)
    assert e.value.code == 3
