"""Moments of a batch's instances on the device (lbm_batch_moments) against the oracle's moments of the
state that the batch hands out: FP64 sums over the same FP32 values, so 1e-13 of each moment's
largest term bounds the rounding.  Widths around whole strips of 32 columns, channels of one and of
several columns, both velocity-set sizes, and an instance that stopped in the odd buffer."""
import numpy as np
import pytest

from oracle.march import CAVITY, COUETTE, make_problem as oracle_problem
from paper_1308_0692_gb300 import lbm
from paper_1308_0692_gb300.inputs import random_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NAMES = ("rho", "ux", "uy", "pxx", "pxy", "pyy")


def _compare(b, i, p, stream):
    out = torch.empty((6, p.ncells), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    lbm.lbm_batch_moments(b, i, out.data_ptr())
    stream.synchronize()
    h = lbm.lbm_batch_get_state(b, i)
    ref = p.moments(h)
    # a moment is u_ref times a sum of at most n terms |xi_x^a xi_y^b h|
    worst = p.coeffs["u_ref"] * np.abs(h).sum(axis=0).max() * max(1.0, float(np.abs(p.xi_x).max()) ** 2)
    for k, name in enumerate(NAMES):
        got, want = out[k].cpu().numpy(), np.asarray(ref[name]).ravel()
        assert np.abs(got - want).max() <= 1e-13 * (1.0 + worst), (name, p.nx, p.ny)


@pytest.mark.parametrize("n_half", [2, 4])
@pytest.mark.parametrize("steps", [0, 1, 4])
def test_moments_match_oracle(n_half, steps):
    grids = [(CAVITY, 2, 2), (CAVITY, 31, 7), (CAVITY, 32, 5), (CAVITY, 33, 9), (CAVITY, 70, 3), (COUETTE, 1, 2),
             (COUETTE, 1, 61), (COUETTE, 5, 13)]
    stream = torch.cuda.Stream()
    b = lbm.lbm_batch_init(lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH, n_half),
                           [lbm.make_problem(g, nx, ny, 0.2, 0.004, -0.01, prec=lbm.LBM_FP32_PERTURB, residual_every=3)
                            for g, nx, ny in grids], stream=stream)
    probs = [oracle_problem("half", n_half, g, nx, ny, 0.2, 0.004, -0.01) for g, nx, ny in grids]
    for i, p in enumerate(probs):
        lbm.lbm_batch_set_state(b, i, random_state(p.n, p.ncells, seed=70 + i))
    if steps:
        lbm.lbm_batch_advance(b, steps, 0.0)
    for i, p in enumerate(probs):
        _compare(b, i, p, stream)
    b.close()


def test_moments_of_an_instance_that_stopped_in_the_odd_buffer():
    """One cavity and one channel converge at an odd residual check while a third instance marches on."""
    probs = [(CAVITY, 33, 9, 10.0), (COUETTE, 1, 8, 10.0), (CAVITY, 64, 64, 0.05)]
    stream = torch.cuda.Stream()
    b = lbm.lbm_batch_init(lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH, 2),
                           [lbm.make_problem(g, nx, ny, kn, 0.01, -0.01, prec=lbm.LBM_FP32_PERTURB, residual_every=5)
                            for g, nx, ny, kn in probs], stream=stream)
    tol = 1e-4
    lbm.lbm_batch_advance(b, 400, tol)
    lbm.lbm_batch_poll(b)
    stopped = [lbm.lbm_batch_status(b, i) for i in range(3)]
    assert all(s["converged"] for s in stopped[:2]) and not stopped[2]["converged"]
    assert all(s["steps"] % 2 for s in stopped[:2])
    for i, (g, nx, ny, kn) in enumerate(probs):
        _compare(b, i, oracle_problem("half", 2, g, nx, ny, kn, 0.01, -0.01), stream)
    b.close()
