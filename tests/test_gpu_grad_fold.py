"""The gradient's fold of the edge padding (one thread, a warp or a block per
model cell, by the padded cells it owns) against the FP64 oracle, at the sizes
where the owner changes: no sponge, single-cell model sides, and a sponge wide
enough that a corner's padded cells go to a block (21^3 > 4096)."""
import numpy as np
import pytest

from helpers import Case, DeviceShot, rel_l2

pytestmark = pytest.mark.gpu
TOL = 1e-4  # the wavefield tolerance: FP32 fields against FP64


@pytest.mark.parametrize("nx,ny,nz,nb", [
    (28, 24, 20, 0), (8, 5, 6, 20), (4, 1, 3, 8), (20, 6, 1, 16), (2, 3, 2, 17)])
def test_gradient_fold_matches_the_oracle(nx, ny, nz, nb):
    case = Case(nx=nx, ny=ny, nz=nz, nb=nb, nt=24, sigma=0.5, rec_stride=1,
                src=(nx // 2, ny // 2, min(2, nz - 1)), rec_z=0)
    vel = np.random.default_rng(5).uniform(1500.0, 3000.0, size=(nz, ny, nx))
    g = DeviceShot(case, want_grad=True, vel=vel * vel, squared=True)
    g.forward()
    resid = case.d_obs(g.nrec)
    grad = g.grad(resid).cpu().numpy()
    prob = case.oracle_problem(squared=True, vel=vel * vel)
    _, ref = prob.misfit_and_grad(prob.forward()["data"] - resid)
    assert rel_l2(grad, ref) <= TOL
    # no cell left out: each one within the same bar of the largest value
    assert np.max(np.abs(grad - ref)) <= TOL * np.max(np.abs(ref))
