"""The calls that a user of the framework makes, as measurable cases.

Each case is one pass through the public Python entry points on seeded inputs
that are made on the GPU: whole shots in the storage modes, the off-grid and
end-to-end shots, the velocity gradient, the imaging variants, the batched
launch and the snapshot codec. ``exact`` gives the same outputs in float64
from plain torch code. The stencil, the tables and the taps there are written
from the formulas of the method, not taken from the package.

``work`` counts the bytes of time stepping as one read of u^n, u^{n-1} and c
and one write of u^{n+1} per step (the fields of a step are the inputs and the
outputs of that step), plus the snapshots and the image of the imaging steps;
operations are those of the star stencil.
"""
import math
import random

import numpy as np
import torch

import paper_1603_03971_gb300 as rtm
from paper_1603_03971_gb300 import batch, codec

DX = 10.0
VMIN, VMAX = 1500.0, 4500.0
DT = 0.5 * DX / (VMAX * math.sqrt(3.0))


def _shot(name, nx, ny, nz, nb, radius, nt, storage, ckpt=0, every=1, stride=1, f0=25.0,
          kind="shot"):
    return dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, nb=nb, radius=radius, nt=nt,
                storage=storage, ckpt=ckpt, every=every, stride=stride, f0=f0)


def listed():
    return [
        # a unit-test or tutorial shot: all launches, hardly any work
        _shot("shot_smoke_28", 28, 24, 20, 6, 4, 60, "ckpt", ckpt=16, stride=2),
        # plain RTM of one shot with every snapshot kept (the two-layer workload's grid)
        _shot("shot_all_64", 64, 64, 64, 20, 4, 300, "all", f0=15.0),
        # the same grid with the source and 1024 receivers between grid points
        _shot("offgrid_64", 64, 64, 64, 20, 4, 80, "all", stride=2, kind="offgrid"),
        # a mid-size survey shot, odd sides, boundary storage with reverse stepping
        _shot("boundary_150", 150, 131, 117, 21, 4, 100, "boundary", stride=3),
        # the throughput workload's grid: checkpoints every 50 steps, all surface receivers
        _shot("shot_ckpt_512", 512, 512, 512, 32, 4, 100, "ckpt", ckpt=50, f0=20.0),
        # a 16th-order shot with ragged sides
        _shot("shot_r8_300", 300, 261, 230, 32, 8, 60, "ckpt", ckpt=20, stride=2),
        # several 16th-order shots on uneven apertures in one call
        dict(name="batch_r8_6", kind="batch", nx=480, ny=416, nz=320, nb=32, radius=8, nt=24,
             ckpt=8, every=1, shots=6, lo=96, hi=224, layout=1, f0=25.0),
        # one misfit and velocity-gradient evaluation of an inversion, through autograd
        _shot("gradient_256", 256, 256, 256, 32, 4, 50, "ckpt", ckpt=25, stride=2,
              kind="gradient"),
        # imaging every 4th step with source illumination, then both image filters
        _shot("illum_190", 192, 170, 149, 24, 4, 80, "all", every=4, stride=2, kind="illum"),
        # a whole shot from pinned host buffers: upload, model preparation, shot, download
        _shot("host_200", 200, 184, 160, 20, 4, 60, "ckpt", ckpt=20, kind="host"),
        # snapshot compression: encode and decode one snapshot of the learned workload
        dict(name="codec_384", kind="codec", nx=384, ny=384, nz=384),
        # one training step of the codec on the training workload's snapshots
        dict(name="train_192", kind="train", nx=192, ny=192, nz=192, batch=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, lo, hi, nb):
    """Three sides; the padded x extent has to be a multiple of 4."""
    nx, ny, nz = (_log_int(rng, lo, hi) for _ in range(3))
    return max(4, nx + (-(nx + 2 * nb)) % 4), ny, nz


def draw(rng):
    kind = rng.choice(["shot", "shot", "shot", "batch", "gradient", "illum", "offgrid", "host",
                       "codec", "train"])
    if kind in ("codec", "train"):
        nx, ny, nz = (4 * _log_int(rng, 10, 80 if kind == "codec" else 44) for _ in range(3))
        c = dict(kind=kind, nx=nx, ny=ny, nz=nz)
        if kind == "train":
            c["batch"] = rng.randint(1, 4)
        return c
    radius = rng.choice([4, 4, 8])
    nb = rng.randint(6, 32)
    nt = rng.randint(30, 90)
    if kind == "batch":
        nx, ny, nz = _sides(rng, 128, 400, nb)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, nb=nb, radius=radius,
                    nt=rng.randint(12, 30), ckpt=rng.randint(4, 12), every=rng.randint(1, 3),
                    shots=rng.randint(2, 7), lo=64, hi=rng.randint(96, 200),
                    layout=rng.randint(2, 1 << 20), f0=25.0)
    lo, hi = dict(shot=(24, 360), gradient=(24, 240), illum=(32, 256), offgrid=(24, 96),
                  host=(24, 240))[kind]
    nx, ny, nz = _sides(rng, lo, hi, nb)
    storage, ckpt, every = "ckpt", rng.randint(6, 30), 1
    if kind in ("shot", "offgrid"):
        storage = rng.choice(["all", "ckpt", "ckpt", "boundary", "decimated", "revolve"])
        every = rng.randint(1, 4)
        if storage == "revolve":
            ckpt = rng.randint(4, 12)
        elif storage == "decimated":
            ckpt = rng.choice([0, rng.randint(1, 20)])
    elif kind == "illum":
        storage, ckpt, every = "all", 0, rng.randint(2, 6)
    c = _shot("", nx, ny, nz, nb, radius, nt, storage, ckpt, every, rng.randint(1, 4),
              rng.uniform(20.0, 35.0), kind)
    del c["name"]
    return c


# ---- inputs ----------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _filtered(shape, gen, shape_of):
    """Seeded white noise with its spectrum shaped by shape_of(wavenumber in cycles per cell)."""
    nz, ny, nx = shape
    f = torch.fft.rfftn(torch.randn(shape, device="cuda", generator=gen))
    k2 = (torch.fft.fftfreq(nz, device="cuda")[:, None, None] ** 2
          + torch.fft.fftfreq(ny, device="cuda")[None, :, None] ** 2
          + torch.fft.rfftfreq(nx, device="cuda")[None, None, :] ** 2)
    f *= shape_of(k2)
    return torch.fft.irfftn(f, s=shape)


def _velocity(shape, gen):
    """Smooth random velocity: noise smoothed over 8 cells, scaled to [VMIN, VMAX]."""
    s = _filtered(shape, gen, lambda k2: torch.exp(-2.0 * (math.pi * 8.0) ** 2 * k2))
    lo, hi = s.min(), s.max()
    return (VMIN + (VMAX - VMIN) * (s - lo) / (hi - lo)).clamp_(VMIN, VMAX).contiguous()


def _ricker(t, f0):
    a = (math.pi * f0 * t) ** 2
    return (1.0 - 2.0 * a) * torch.exp(-a)


def _traces(nt, rec, src, f0, gen):
    """Recorded data: three events with hyperbolic moveout and weak noise."""
    t = torch.arange(nt, device="cuda", dtype=torch.float32)[:, None] * DT
    off = ((rec[:, :2].float() - torch.tensor(src[:2], device="cuda")) * DX).norm(dim=1)
    d = 2e-5 * torch.randn((nt, rec.shape[0]), device="cuda", generator=gen)
    for amp in (1e-3, 4e-4, -3e-4):
        depth = 40.0 + 400.0 * torch.rand((), device="cuda", generator=gen)
        v = 1800.0 + 1500.0 * torch.rand((), device="cuda", generator=gen)
        at = torch.sqrt(off * off + depth * depth) / v
        d += amp * _ricker(t - 0.4 * nt * DT - 0.2 * at[None, :], f0)
    return d.contiguous()


def _receivers(nx, ny, stride, z=2):
    y, x = torch.meshgrid(torch.arange(0, ny, stride), torch.arange(0, nx, stride),
                          indexing="ij")
    r = torch.stack([x.reshape(-1), y.reshape(-1), torch.full((x.numel(),), z)], dim=1)
    return r.to(torch.int32).cuda().contiguous()


def _source(case):
    return case["nx"] // 2, case["ny"] // 2, min(4, case["nz"] - 1)


def _points(case, seed):
    """Off-grid source and receivers (model coordinates in cells)."""
    r = np.random.RandomState(seed % (1 << 31))
    src = np.array(_source(case)) + np.array([0.4, -0.3, 0.5])
    ys, xs = np.meshgrid(np.arange(0, case["ny"] - 1, case["stride"]),
                         np.arange(0, case["nx"] - 1, case["stride"]), indexing="ij")
    rec = np.stack([xs.ravel(), ys.ravel(), np.full(xs.size, 2.0)], axis=1)
    return src, rec + r.uniform(0.1, 0.9, size=rec.shape)


def _shot_inputs(case, seed):
    g = _gen(seed)
    vel = _velocity((case["nz"], case["ny"], case["nx"]), g)
    rec = _receivers(case["nx"], case["ny"], case["stride"])
    if case["kind"] == "offgrid":
        src, pts = _points(case, seed)
        rec = torch.from_numpy(pts).cuda()
    dobs = _traces(case["nt"], rec, _source(case), case["f0"], g)
    return vel, rec, dobs


def _params(case, nrec):
    return rtm.make_params(case["nx"], case["ny"], case["nz"], case["nb"], case["radius"],
                           case["nt"], DX, DT, case["f0"], 1.0 / case["f0"], _source(case), nrec,
                           storage=case["storage"], ckpt_every=case["ckpt"],
                           image_every=case["every"], want_grad=case["kind"] == "gradient")


def _apertures(case):
    r = random.Random(case["layout"])
    out = []
    for _ in range(case["shots"]):
        nx, ny, nz = (min(n, _log_int(r, case["lo"], case["hi"]))
                      for n in (case["nx"], case["ny"], case["nz"]))
        nx -= (nx + 2 * case["nb"]) % 4
        ox, oy = r.randint(0, case["nx"] - nx), r.randint(0, case["ny"] - ny)
        out.append((ox, oy, 0, nx, ny, nz, nx // 2, ny // 2, 4, 2))
    return out


def _batch_inputs(case, seed):
    g = _gen(seed)
    vel = _velocity((case["nz"], case["ny"], case["nx"]), g)
    dobs = []
    for ap in _apertures(case):
        nx, ny = ap[3], ap[4]
        dobs.append(_traces(case["nt"], _receivers(nx, ny, 1), ap[6:9], case["f0"], g).reshape(-1))
    return vel, torch.cat(dobs)


AE_SHAPES = ((32, 8, 8), (32, 0, 0), (16, 27 * 32, 864), (16, 0, 0), (32, 64 * 16, 128),
             (32, 0, 0), (8, 32, 32), (1, 0, 0))  # rows, columns, fan-in of W1 b1 .. W4 b4


def _ae_params(gen):
    """He-style weights and small biases in the codec's order."""
    out = []
    for rows, cols, fan in AE_SHAPES:
        if cols:
            out.append(torch.randn(rows * cols, device="cuda", generator=gen)
                       * math.sqrt(2.0 / fan))
        else:
            out.append(0.05 * torch.randn(rows, device="cuda", generator=gen))
    return torch.cat(out).contiguous()


def _snapshots(count, shape, gen):
    """Wavefield-like snapshots: band-limited noise inside a spherical front, zero beyond it."""
    out = torch.empty((count,) + tuple(shape), device="cuda")
    ax = [torch.arange(n, device="cuda", dtype=torch.float32) for n in shape]
    for i in range(count):
        u = _filtered(shape, gen, lambda k2: k2 * torch.exp(-k2 / (2.0 * 0.05 ** 2)))
        at = torch.rand(3, device="cuda", generator=gen)
        r = torch.sqrt((ax[0][:, None, None] - at[0] * shape[0]) ** 2
                       + (ax[1][None, :, None] - at[1] * shape[1]) ** 2
                       + (ax[2][None, None, :] - at[2] * shape[2]) ** 2)
        front = 0.7 * max(shape)
        out[i] = 1e-3 * u / u.std() * (1.0 - r / front).clamp_(min=0.0) / (1.0 + 0.02 * r)
    return out


def _ae_inputs(case, seed):
    g = _gen(seed)
    P = _ae_params(g)
    shape = (case["nz"], case["ny"], case["nx"])
    s = _snapshots(case.get("batch", 1), shape, g)
    m = 1e-3 * torch.randn(P.numel(), device="cuda", generator=g)
    v = 1e-5 * (0.1 + torch.rand(P.numel(), device="cuda", generator=g))
    return P, s, m, v


# ---- the calls ---------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("codec", "train"):
        P, s, m, v = _ae_inputs(case, seed)
        st = dict(kind=kind, P=P, m=m, v=v)
        shape = (case["nz"], case["ny"], case["nx"])
        st["ws"] = codec.alloc_workspace(shape)
        if kind == "codec":
            st.update(s=s[0], out=torch.empty_like(s[0]),
                      lat=torch.empty(codec.latent_shape(shape), dtype=torch.bfloat16,
                                      device="cuda"),
                      scale=torch.empty(1, device="cuda"))
        else:
            st.update(s=s, grad=torch.empty_like(P),
                      loss=torch.empty(1, dtype=torch.float64, device="cuda"))
        return st
    shape = (case["nz"], case["ny"], case["nx"])
    if kind == "batch":
        vel, dobs = _batch_inputs(case, seed)
        p = rtm.make_params(case["nx"], case["ny"], case["nz"], case["nb"], case["radius"],
                            case["nt"], DX, DT, case["f0"], 1.0 / case["f0"], (0, 0, 0), 0,
                            storage="ckpt", ckpt_every=case["ckpt"], image_every=case["every"])
        aps = [batch.Aperture(*a) for a in _apertures(case)]
        return dict(kind=kind, p=p, aps=aps, vel=vel, dobs=dobs, data=torch.zeros_like(dobs),
                    image=torch.zeros(shape, device="cuda"), ws=batch.alloc_workspace(p, aps))
    vel, rec, dobs = _shot_inputs(case, seed)
    p = _params(case, rec.shape[0])
    st = dict(kind=kind, p=p, dobs=dobs)
    if kind == "host":
        st.update(vel=vel.cpu().pin_memory(), rec=rec.cpu().pin_memory(),
                  dobs=dobs.cpu().pin_memory(), image=torch.empty(shape).pin_memory(),
                  ws=rtm.alloc_workspace(p, host_io=True))
        return st
    st["ws"] = rtm.alloc_workspace(p)
    if kind == "gradient":
        st.update(v2=(vel * vel).requires_grad_(True), rec=rec)
        return st
    st["c"] = rtm.model_prep(p, vel, st["ws"])
    st["image"] = torch.zeros(shape, device="cuda")
    st["data"] = torch.empty((p.nt, p.nrec), device="cuda")
    if kind == "offgrid":
        st["taps"] = rtm.offgrid_taps(p, _points(case, seed)[0], rec.cpu().numpy(), "cuda")
    else:
        st["rec"] = rec
    if kind == "illum":
        st["illum"] = torch.zeros(shape, device="cuda")
    return st


def run(st):
    kind = st["kind"]
    if kind == "shot":
        rtm.shot(st["p"], st["c"], st["rec"], st["dobs"], st["ws"], st["image"], data=st["data"])
        return st["image"], st["data"]
    if kind == "offgrid":
        rtm.shot_offgrid(st["p"], st["c"], st["taps"], st["dobs"], st["ws"], st["image"],
                         data=st["data"])
        return st["image"], st["data"]
    if kind == "host":
        return rtm.shot_host(st["p"], st["vel"], st["rec"], st["dobs"], st["image"], st["ws"])
    if kind == "gradient":
        J = rtm.RtmMisfit.apply(st["v2"], st["p"], st["rec"], st["dobs"], st["ws"])
        return J.detach().float(), torch.autograd.grad(J, st["v2"])[0]
    if kind == "illum":
        rtm.forward(st["p"], st["c"], st["rec"], st["ws"], data=st["data"])
        rtm.backward_image_illum(st["p"], st["c"], st["rec"], st["dobs"], st["ws"], st["image"],
                                 st["illum"])
        norm, lap = rtm.image_filter(st["p"], st["image"], st["ws"], illum=st["illum"])
        return st["image"], st["illum"], norm, lap, st["data"]
    if kind == "batch":
        batch.run(st["p"], st["aps"], st["vel"], st["dobs"], st["image"], st["ws"],
                  data=st["data"])
        return st["image"], st["data"]
    if kind == "codec":
        codec.encode(st["P"], st["s"], st["ws"], latent=st["lat"], scale=st["scale"])
        codec.decode(st["P"], st["lat"], st["scale"], st["ws"], out=st["out"])
        return st["lat"], st["scale"], st["out"]
    codec.train_step(st["P"], st["m"], st["v"], 100, 1e-4, st["s"], st["ws"],
                     grad_out=st["grad"], loss=st["loss"])
    return st["loss"].float(), st["grad"], st["P"], st["m"], st["v"]


# ---- what a pass cannot do without --------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind in ("codec", "train"):
        n = case["nx"] * case["ny"] * case["nz"]
        enc = 2.0 * (n / 8 * 8 * 32 + n / 64 * 27 * 32 * 16)
        dec = 2.0 * (n / 8 * 8 * 16 * 32 + n * 32)
        if kind == "codec":
            return {"bytes": 2.0 * (4 * n + n / 2), "flops": enc + dec}
        return {"bytes": 4.0 * n * case["batch"] + 47185 * 4 * 7.0,
                "flops": 3.0 * (enc + dec) * case["batch"]}
    nt, nb, r = case["nt"], case["nb"], case["radius"]
    grids = ([a[3:6] for a in _apertures(case)] if kind == "batch"
             else [(case["nx"], case["ny"], case["nz"])])
    storage = "ckpt" if kind == "batch" else case["storage"]
    total = {"bytes": 0.0, "flops": 0.0}
    for nx, ny, nz in grids:
        N = float((nx + 2 * nb) * (ny + 2 * nb) * (nz + 2 * nb))
        M = float(nx * ny * nz)
        img = nt // case["every"]
        steps, b = 2.0 * nt, 0.0
        if kind == "gradient":
            b = 4.0 * N * nt + 12.0 * N * nt  # L u written, then read beside the gradient's sum
            steps += nt
        else:
            b = 12.0 * M * img + (8.0 * M * img if kind == "illum" else 0.0)
            if storage == "boundary":  # the reverse steps cover the model region
                b += 16.0 * M * nt
            elif storage != "decimated":
                b += 4.0 * M * img
            if storage in ("ckpt", "revolve"):
                steps += nt
        total["bytes"] += 16.0 * N * steps + b
        total["flops"] += (6.0 * r + 7.0) * N * steps
    return total


# ---- the same in 64 bits -------------------------------------------------------------

def _weights(r):
    f = math.factorial
    a = [0.0] + [2.0 * (-1) ** (k + 1) * f(r) ** 2 / (k * k * f(r - k) * f(r + k))
                 for k in range(1, r + 1)]
    a[0] = -2.0 * sum(a[1:])
    return a


def _star(u, r, out):
    """out = the star Laplacian of u with zeros outside."""
    a = [w / (DX * DX) for w in _weights(r)]
    torch.mul(u, 3.0 * a[0], out=out)
    for k in range(1, r + 1):
        for d in range(3):
            n = u.shape[d]
            if n > k:
                out.narrow(d, k, n - k).add_(u.narrow(d, 0, n - k), alpha=a[k])
                out.narrow(d, 0, n - k).add_(u.narrow(d, k, n - k), alpha=a[k])
    return out


class _Wave:
    """Leapfrog steps on the padded grid in float64."""

    def __init__(self, vel2, nb, r, nt, f0):
        self.nb, self.r = nb, r
        nz, ny, nx = vel2.shape
        self.model = (nz, ny, nx)
        at = [torch.arange(-nb, n + nb, device="cuda").clamp_(0, n - 1) for n in vel2.shape]
        self.c = (vel2.double() * (DT * DT))[at[0]][:, at[1]][:, :, at[2]].contiguous()
        self.shape = tuple(self.c.shape)
        prof = []
        for n in self.shape:
            i = torch.arange(n, device="cuda", dtype=torch.float64)
            d = torch.minimum(i, n - 1 - i)
            prof.append(torch.exp(-(0.015 * (nb - d).clamp_(min=0.0)) ** 2))
        self.g = prof[0][:, None, None] * prof[1][None, :, None] * prof[2][None, None, :]
        t = torch.arange(nt, dtype=torch.float64, device="cuda") * DT - 1.0 / f0
        self.w = _ricker(t, f0)
        self.lap = torch.empty_like(self.c)

    def zero(self):
        return torch.zeros_like(self.c)

    def step(self, cur, prev):
        """u^{n+1} in prev's memory, without the source."""
        lap = _star(cur, self.r, self.lap)
        lap.mul_(self.c).add_(cur, alpha=2.0).mul_(self.g)
        prev.mul_(self.g).mul_(self.g).neg_().add_(lap)
        return prev

    def inner(self, u):
        nz, ny, nx = self.model
        return u[self.nb:self.nb + nz, self.nb:self.nb + ny, self.nb:self.nb + nx]

    def add(self, u, idx, val):
        u.view(-1).index_add_(0, idx, val)


def _kaiser(x, n):
    """Indices and weights of one axis of a point at padded position x."""
    if x == math.floor(x):
        return [int(x)], [1.0]
    lo = int(math.floor(x)) - 3
    i = np.arange(lo, lo + 8)
    d = i - x
    w = np.sinc(d) * np.i0(4.14 * np.sqrt(np.clip(1.0 - (d / 4.0) ** 2, 0.0, None))) / np.i0(4.14)
    keep = (i >= 0) & (i < n)
    return i[keep].tolist(), w[keep].tolist()


def _taps(W, points):
    """(indices, weights, owner) of points at model coordinates."""
    NZ, NY, NX = W.shape
    pts = np.asarray(points)
    if pts.dtype.kind == "i":  # grid points: one tap of weight 1 each
        p = torch.from_numpy(pts.astype(np.int64)).cuda() + W.nb
        return ((p[:, 2] * NY + p[:, 1]) * NX + p[:, 0],
                torch.ones(len(pts), dtype=torch.float64, device="cuda"),
                torch.arange(len(pts), device="cuda"))
    idx, wt, own = [], [], []
    for j, p in enumerate(pts):
        (ix, wx), (iy, wy), (iz, wz) = (_kaiser(p[d] + W.nb, n) for d, n in enumerate((NX, NY, NZ)))
        lin = (np.array(iz)[:, None, None] * NY + np.array(iy)[None, :, None]) * NX \
            + np.array(ix)[None, None, :]
        idx.append(lin.ravel())
        wt.append((np.array(wz)[:, None, None] * np.array(wy)[None, :, None]
                   * np.array(wx)[None, None, :]).ravel())
        own.append(np.full(lin.size, j))
    return tuple(torch.from_numpy(np.concatenate(v)).cuda() for v in (idx, wt, own))


def _interpolated(u):
    """Every other sample per axis, then linear interpolation back."""
    for d, n in enumerate(u.shape):
        kept = u.index_select(d, torch.arange(0, n, 2, device="cuda"))
        right = torch.cat([kept.narrow(d, 1, kept.shape[d] - 1),
                           kept.narrow(d, kept.shape[d] - 1, 1)], dim=d)
        odd = 0.5 * (kept + right)
        u = torch.stack([kept, odd], dim=d + 1).flatten(d, d + 1).narrow(d, 0, n).contiguous()
    return u


def _exact_shot(vel2, nb, r, nt, f0, every, src, rec, dobs, grad=False, illum=False,
                coarse_after=None):
    """Data and image (and illumination), or data and the gradient for data - dobs."""
    W = _Wave(vel2, nb, r, nt, f0)
    s_idx, s_w, _ = _taps(W, [src])
    r_idx, r_w, r_own = _taps(W, rec)
    cv, gv = W.c.view(-1), W.g.view(-1)
    s_val = cv[s_idx] * s_w / DX ** 3
    nrec = len(rec)
    data = torch.zeros((nt, nrec), dtype=torch.float64, device="cuda")
    seg = 50
    starts = {}

    def forward(n0, n1, prev, cur, keep, record):
        for n in range(n0, n1):
            if grad and keep is not None:
                keep.append(cur.clone())
            nxt = W.step(cur, prev)
            W.add(nxt, s_idx, s_val * W.w[n])
            if record:
                data[n].index_add_(0, r_own, r_w * nxt.view(-1)[r_idx])
            prev, cur = cur, nxt
            if not grad and keep is not None:
                keep.append(W.inner(cur).clone() if (n + 1) % every == 0 else None)
        return prev, cur

    prev, cur = W.zero(), W.zero()
    for n0 in range(0, nt, seg):
        starts[n0] = (prev.clone(), cur.clone())
        prev, cur = forward(n0, min(nt, n0 + seg), prev, cur, None, True)
    prev = cur = None
    resid = data - dobs if grad else dobs
    r_val = cv[r_idx] * gv[r_idx] * r_w / DX ** 3
    image = torch.zeros(W.shape if grad else W.model, dtype=torch.float64, device="cuda")
    light = torch.zeros_like(image) if illum else None
    mu2, mu1 = W.zero(), W.zero()
    for n0 in reversed(range(0, nt, seg)):
        n1, keep = min(nt, n0 + seg), []
        forward(n0, n1, *starts.pop(n0), keep, False)
        for m in range(n1, n0, -1):
            mu = W.step(mu1, mu2)
            W.add(mu, r_idx, r_val * resid[m - 1][r_own])
            mu2, mu1 = mu1, mu
            u = keep.pop()
            if grad:
                _star(u, r, W.lap)
                W.add(W.lap, s_idx, s_w * W.w[m - 1] / (DX ** 3 * gv[s_idx]))
                image.addcmul_(W.lap, mu)
            elif u is not None:
                if coarse_after is not None and m > coarse_after:
                    u = _interpolated(u)
                image.addcmul_(u, W.inner(mu))
                if illum:
                    light.addcmul_(u, u)
    if grad:
        x = image.div_(W.c).mul_(DX ** 3 * DT * DT)
        for d, n in enumerate(W.model):  # the transpose of the edge padding
            y = x.narrow(d, nb, n).clone()
            if nb:
                y.select(d, 0).add_(x.narrow(d, 0, nb).sum(dim=d))
                y.select(d, n - 1).add_(x.narrow(d, nb + n, nb).sum(dim=d))
            x = y
        return data, x
    return (data, image, light) if illum else (data, image)


def _leaky(x):
    return torch.where(x > 0, x, 0.1 * x)


def _ae_split(P):
    out, o = [], 0
    for rows, cols, _ in AE_SHAPES:
        n = rows * max(cols, 1)
        out.append(P[o:o + n].view(rows, cols) if cols else P[o:o + n])
        o += n
    return out


def _ae_encode(P, x):
    """Normalised snapshot [nz][ny][nx] to the latent [nz/4][ny/4][nx/4][16]."""
    W1, b1, W2, b2 = _ae_split(P)[:4]
    nz, ny, nx = x.shape
    p = x.view(nz // 2, 2, ny // 2, 2, nx // 2, 2).permute(0, 2, 4, 1, 3, 5)
    h = _leaky(p.reshape(nz // 2, ny // 2, nx // 2, 8) @ W1.t() + b1)
    h = torch.nn.functional.pad(h, (0, 0, 1, 1, 1, 1, 1, 1))
    W2 = W2.view(16, 3, 3, 3, 32)
    lat = b2
    for kz in range(3):
        for ky in range(3):
            for kx in range(3):
                w = h[kz:kz + nz // 2:2, ky:ky + ny // 2:2, kx:kx + nx // 2:2]
                lat = lat + w @ W2[:, kz, ky, kx].t()
    return lat


def _ae_decode(P, lat):
    W3, b3, W4, b4 = _ae_split(P)[4:]
    W3 = W3.view(32, 4, 4, 4, 16)
    mz, my, mx = lat.shape[:3]
    lp = torch.nn.functional.pad(lat, (0, 0, 1, 1, 1, 1, 1, 1))
    taps = ([(0, 1), (-1, 3)], [(1, 0), (0, 2)])  # output parity: (input offset, kernel index)
    parts = []
    for q in range(8):
        acc = b3
        for tz, kz in taps[q >> 2]:
            for ty, ky in taps[(q >> 1) & 1]:
                for tx, kx in taps[q & 1]:
                    w = lp[1 + tz:1 + tz + mz, 1 + ty:1 + ty + my, 1 + tx:1 + tx + mx]
                    acc = acc + w @ W3[:, kz, ky, kx].t()
        parts.append(_leaky(acc) @ W4.t() + b4)  # [mz][my][mx][8]
    y = torch.stack(parts, dim=3).view(mz, my, mx, 2, 2, 2, 2, 2, 2)
    return y.permute(0, 3, 6, 1, 4, 7, 2, 5, 8).reshape(4 * mz, 4 * my, 4 * mx)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("codec", "train"):
        P, s, m, v = (t.double() for t in _ae_inputs(case, seed))
        if kind == "codec":
            scale = s[0].square().mean().sqrt()
            lat = _ae_encode(P, s[0] / scale)
            return lat, scale.view(1), scale * _ae_decode(P, lat)
        P.requires_grad_(True)
        loss, grad = 0.0, torch.zeros_like(P)
        for x in s:
            x = x / x.square().mean().sqrt()
            part = (_ae_decode(P, _ae_encode(P, x)) - x).square().mean() / len(s)
            grad += torch.autograd.grad(part, P)[0]
            loss = loss + part.detach()
        g = grad / max(1.0, float(grad.norm()))
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        step = 1e-4 * (m / (1 - 0.9 ** 100)) / ((v / (1 - 0.999 ** 100)).sqrt() + 1e-8)
        return loss.view(1), grad, P.detach() - step, m, v
    common = (case["nb"], case["radius"], case["nt"], case["f0"], case["every"] if "every" in case
              else 1)
    if kind == "batch":
        vel, dobs = _batch_inputs(case, seed)
        image = torch.zeros(vel.shape, dtype=torch.float64, device="cuda")
        datas, o = [], 0
        for ox, oy, oz, nx, ny, nz, sx, sy, sz, rz in _apertures(case):
            n = case["nt"] * nx * ny
            v = vel[oz:oz + nz, oy:oy + ny, ox:ox + nx].double()
            data, img = _exact_shot(v * v, *common, (sx, sy, sz),
                                    _receivers(nx, ny, 1, rz).cpu().numpy(),
                                    dobs[o:o + n].view(case["nt"], -1).double())
            image[oz:oz + nz, oy:oy + ny, ox:ox + nx] += img
            datas.append(data.reshape(-1))
            o += n
        return image, torch.cat(datas)
    vel, rec, dobs = _shot_inputs(case, seed)
    rec, dobs = rec.cpu().numpy(), dobs.double()
    src = _points(case, seed)[0] if kind == "offgrid" else _source(case)
    v2 = (vel * vel).double() if kind == "gradient" else vel.double() ** 2
    if kind == "gradient":
        data, grad = _exact_shot(v2, *common, src, rec, dobs, grad=True)
        return 0.5 * (data - dobs).square().sum(), grad
    if kind == "illum":
        data, image, light = _exact_shot(v2, *common, src, rec, dobs, illum=True)
        lap = _star(image, case["radius"], torch.empty_like(image)).neg_()
        return image, light, image / (light + 1e-3 * light.max()), lap, data
    after = case["ckpt"] if case["storage"] == "decimated" else None
    data, image = _exact_shot(v2, *common, src, rec, dobs, coarse_after=after)
    return image if kind == "host" else (image, data)
