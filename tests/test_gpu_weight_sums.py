"""The weight and bias gradients of a training step against float64 sums of the
bfloat16 operands that the step leaves in its workspace: sums over a volume
keep a float's bits, however long a block's share of them is."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [("W1", 256), ("b1", 32), ("W2", 16 * 864), ("b2", 16), ("W3", 32 * 1024), ("b3", 32),
         ("W4", 256), ("b4", 1)]


def _params(gen):
    import torch

    out = []
    for (name, n), fan in zip(SIZES, (8, 0, 864, 0, 128, 0, 32, 0)):
        a = torch.randn(n, device="cuda", generator=gen)
        out.append(a * (2.0 / fan) ** 0.5 if fan else 0.05 * a)
    return torch.cat(out).contiguous()


def _snapshot(shape, gen):
    """Band-limited noise, as a wavefield."""
    import torch

    nz, ny, nx = shape
    f = torch.fft.rfftn(torch.randn(shape, device="cuda", generator=gen))
    k2 = (torch.fft.fftfreq(nz, device="cuda")[:, None, None] ** 2
          + torch.fft.fftfreq(ny, device="cuda")[None, :, None] ** 2
          + torch.fft.rfftfreq(nx, device="cuda")[None, None, :] ** 2)
    u = torch.fft.irfftn(f * k2 * torch.exp(-k2 / 0.005), s=shape)
    return (1e-3 * u / u.std())[None].contiguous()


def _operands(ws, shape):
    """The activations and gradients kept in the workspace (256-byte aligned parts)."""
    import torch

    n = shape[0] * shape[1] * shape[2]
    nh, nl, at, out = n // 8, n // 64, 256, {}
    for name, count, dtype in [
            ("h1", nh * 32, torch.bfloat16), ("lat", nl * 16, torch.bfloat16),
            ("g1", nh * 32, torch.bfloat16), ("y", n, torch.float32), ("gy", n, torch.bfloat16),
            ("ga3", nh * 32, torch.bfloat16), ("glat", nl * 16, torch.bfloat16),
            ("ga1", nh * 32, torch.bfloat16)]:
        size = count * (4 if dtype == torch.float32 else 2)
        out[name] = ws[at:at + size].view(dtype).double()
        at += -(-size // 256) * 256
    inv_sigma = ws[76:80].view(torch.float32)
    return out, inv_sigma


def _reference(t, x, inv_sigma, shape):
    import torch
    import torch.nn.functional as F

    nz, ny, nx = shape
    h, q = (nz // 2, ny // 2, nx // 2), (nz // 4, ny // 4, nx // 4)

    def patch(v):  # the 8 voxels of each half-resolution voxel
        v = v.view(h[0], 2, h[1], 2, h[2], 2)
        return v.permute(0, 2, 4, 1, 3, 5).reshape(-1, 8)

    def taps(v, n, pad):  # rows at the n^3 taps of each quarter-resolution voxel
        v = F.pad(v.view(*h, 32), (0, 0) + pad * 3)
        for k in range(n ** 3):
            a, b, c = k // (n * n), k // n % n, k % n
            yield k, v[a:a + 2 * q[0]:2, b:b + 2 * q[1]:2, c:c + 2 * q[2]:2].reshape(-1, 32)
    xq = patch((x[0] * inv_sigma).bfloat16().double())
    ga1, g1, ga3 = (t[k].view(-1, 32) for k in ("ga1", "g1", "ga3"))
    glat, lat = t["glat"].view(-1, 16), t["lat"].view(-1, 16)
    W2 = torch.zeros(16, 27, 32, dtype=torch.float64, device="cuda")
    for k, v in taps(t["h1"], 3, (1, 1)):
        W2[:, k] = glat.T @ v
    W3 = torch.zeros(32, 64, 16, dtype=torch.float64, device="cuda")
    for k, v in taps(t["ga3"], 4, (1, 2)):
        W3[:, k] = v.T @ lat
    return {"W1": ga1.T @ xq, "b1": ga1.sum(0), "W2": W2, "b2": glat.sum(0), "W3": W3,
            "b3": ga3.sum(0), "W4": patch(t["gy"]).T @ g1, "b4": t["gy"].sum()}


@pytest.mark.parametrize("shape", [(40, 36, 44), (112, 120, 128), (192, 192, 192)])
def test_weight_gradients_are_sums_to_a_floats_bits(shape):
    import torch

    from paper_1603_03971_gb300 import codec

    gen = torch.Generator(device="cuda").manual_seed(7)
    P, x = _params(gen), _snapshot(shape, gen)
    ws = codec.alloc_workspace(shape)
    grad = torch.zeros_like(P)
    codec.train_step(P, None, None, 0, 0.0, x, ws, grad_out=grad)
    operands, inv_sigma = _operands(ws, shape)
    ref = _reference(operands, x, inv_sigma, shape)
    at = 0
    for name, n in SIZES:
        got, want = grad[at:at + n].double(), ref[name].reshape(-1)
        at += n
        # up to 4 truncated steps of 2^-23 within a turn, then at most 100 turns
        # and 304 blocks added with errors of either sign up to 2^-25 (b4: one
        # float sum per thread of up to 24 samples and 1216 blocks)
        bar = 4 * 2.0 ** -23 + (1240 if name == "b4" else 404) ** 0.5 * 2.0 ** -25
        assert float((got - want).norm() / want.norm()) <= bar, name
