"""The gradient's fold of the edge padding keeps the bits of float64 sums:
every model cell equals the float64 fold of the accumulator that the call
leaves in its workspace, rounded once, also where a quotient of an accumulated
value and a coefficient lies among the denormals or above the range of a float
(large and small grid spacings: c grows with dx^2, dx^3 dt^2 scales it back)."""
import numpy as np
import pytest

from helpers import Case, DeviceShot

pytestmark = pytest.mark.gpu


def _accumulator(g):
    """The padded accumulator of the last gradient call: the field behind the
    tables and the four fields of a workspace of 256-byte aligned parts."""
    import paper_1603_03971_gb300 as rtm

    NZ, NY, NX = rtm.padded_shape(g.p)

    def up(n):
        return -(-4 * n // 256) * 256
    off = 256 + up(g.p.nt) + up(NX) + up(NY) + up(NZ) + 4 * up(NX * NY * NZ)
    raw = g.ws.cpu().numpy().view(np.uint8)[off:off + 4 * NX * NY * NZ]
    return raw.view(np.float32).reshape(NZ, NY, NX)


def _fold(a, nb):
    """Sums of the padded cells copied from each model cell."""
    for axis in range(3):
        a = np.moveaxis(a, axis, 0)
        n = a.shape[0] - 2 * nb
        if n == 1:
            out = a.sum(axis=0, keepdims=True)
        else:
            out = a[nb:nb + n].copy()
            out[0] = a[:nb + 1].sum(axis=0)
            out[-1] = a[nb + n - 1:].sum(axis=0)
        a = np.moveaxis(out, 0, axis)
    return a


@pytest.mark.parametrize("dx,resid_scale", [(10.0, 1.0), (1000.0, 1.0), (1e-3, 1e30)])
@pytest.mark.parametrize("nx,ny,nz,nb", [(44, 40, 36, 0), (40, 36, 33, 12), (4, 1, 3, 16)])
def test_fold_equals_the_float64_fold(nx, ny, nz, nb, dx, resid_scale):
    case = Case(nx=nx, ny=ny, nz=nz, nb=nb, nt=16, dx=dx, f0=250.0 / dx, t0=0.004 * dx,
                src=(nx // 2, ny // 2, min(2, nz - 1)), rec_z=0, rec_stride=1, sigma=0.5)
    g = DeviceShot(case, want_grad=True, squared=True)
    g.forward()
    grad = g.grad(case.d_obs(g.nrec) * resid_scale).cpu().numpy()
    acc, c = _accumulator(g), g.c.cpu().numpy()
    assert np.isfinite(acc).all() and np.count_nonzero(acc) > 100
    q = acc.astype(np.float64) / c.astype(np.float64)
    scale = g.p.dx ** 3 * g.p.dt ** 2
    ref = _fold(q, nb) * scale
    assert np.abs(ref).max() < 1e38
    if dx > 100 and nz > 3:  # quotients among the denormals that the scale lifts out of them
        assert ((np.abs(q) < 1e-39) & (np.abs(q) * scale > 1e-37) & (q != 0)).any()
    if dx < 1:  # quotients above the float range
        assert np.abs(q).max() > 3.5e38
    # one rounding to float (half an ulp, a denormal step at the bottom), and
    # float64 sums in whatever order over a cell's padded cells
    cells = (2 * nb + 1) ** 3 + 8
    tol = (2.0 ** -24 * (1 + 1e-6) * np.abs(ref) + 2.0 ** -149
           + cells * 2.0 ** -52 * _fold(np.abs(q), nb) * scale)
    bad = np.abs(grad.astype(np.float64) - ref) > tol
    assert not bad.any(), (int(bad.sum()), grad[bad][:4], ref[bad][:4])
