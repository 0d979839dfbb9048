"""The training loss keeps the bits and the range of float64 sums. With zero
weights the codec gives y = b4 everywhere, so the loss is the mean of
(b4 - x)^2 for the normalised samples x, and with a quarter's multiples of mean
square 1 as samples the normalisation is exact."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _loss(x, b4, offset=0):
    import torch

    from paper_1603_03971_gb300 import codec
    from paper_1603_03971_gb300._lib import lib

    n = int(lib().rtm_ae_param_count())
    P = torch.zeros(n, device="cuda")
    P[n - 1] = float(b4)  # the output layer's bias is the last parameter
    buf = torch.empty(x.size + offset, device="cuda")
    s = buf[offset:].view((1,) + x.shape)
    s.copy_(torch.from_numpy(x)[None])
    ws = codec.alloc_workspace(x.shape)
    loss = codec.train_step(P, None, None, 0, 0.0, s, ws)
    return float(loss.item())


def _samples(shape, seed):
    """+-0.5 and +-1.5, three of eight the larger: mean square 1 exactly."""
    rng = np.random.default_rng(seed)
    n = int(np.prod(shape))
    x = np.where(rng.permutation(n) < n * 3 // 8, 1.5, 0.5) * rng.choice([-1.0, 1.0], n)
    return x.reshape(shape).astype(np.float32)


@pytest.mark.parametrize("shape,offset", [((4, 4, 4), 0), ((8, 12, 16), 1), ((64, 60, 56), 0),
                                          ((128, 128, 124), 1)])
def test_loss_is_a_float64_sum(shape, offset):
    x = _samples(shape, 3)
    b4 = np.float32(0.123456789)
    d = (b4 - x).astype(np.float64)  # rounded to float, as the kernel's difference
    want = math.fsum((d * d).ravel().tolist()) / d.size
    # exact squares, then float64 sums: at most n / (304 x 256) values of a
    # thread, 13 levels of its block, one block after another (up to 1216)
    ulps = d.size / (304 * 256) + 13 + 1216
    assert abs(_loss(x, b4, offset) - want) <= ulps * 2.0 ** -53 * want


@pytest.mark.parametrize("b4", [1e-25, 3e-21, 2e18, 1e25, 1e37])
@pytest.mark.parametrize("offset", [0, 1])
def test_squares_beyond_a_floats_range_stay_finite(b4, offset):
    b4 = np.float32(b4)
    x = np.zeros((8, 12, 16), np.float32) if b4 < 1 else _samples((8, 12, 16), 5)
    d = (b4 - x).astype(np.float64)
    want = math.fsum((d * d).ravel().tolist()) / d.size
    got = _loss(x, b4, offset)
    assert abs(got - want) <= 1300 * 2.0 ** -53 * want
