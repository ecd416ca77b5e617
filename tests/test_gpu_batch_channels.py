"""One-column channels of a batch (batch_column_kernel) at the edges of a block's cells, against the
oracle: the states after an uneven split of steps (FP32: 2e-6 of max |h| per step, as for the
other batch kernels), the residual of the last check, and the freezing of a converged channel."""
import numpy as np
import pytest

from oracle.march import CAVITY, COUETTE, make_problem as oracle_problem, residual as oracle_residual
from paper_1308_0692_gb300 import lbm
from paper_1308_0692_gb300.inputs import random_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# one column of 2 to 512 cells on chip; longer or wider ones, and cavities, on the other kernels
INSTANCES = [(COUETTE, 1, ny) for ny in (2, 3, 31, 32, 33, 255, 512, 513)] + [(COUETTE, 3, 20), (CAVITY, 33, 5)]


@pytest.mark.parametrize("n_half", [2, 4])
def test_channels_match_oracle(n_half):
    vs = lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH, n_half)
    probs = [lbm.make_problem(g, nx, ny, 0.2, 0.004, -0.01, prec=lbm.LBM_FP32_PERTURB, residual_every=3)
             for g, nx, ny in INSTANCES]
    stream = torch.cuda.Stream()
    b = lbm.lbm_batch_init(vs, probs, stream=stream)
    start = []
    for i, (g, nx, ny) in enumerate(INSTANCES):
        h = random_state(4 * n_half * n_half, nx * ny, seed=50 + i).astype(np.float32).astype(np.float64)
        lbm.lbm_batch_set_state(b, i, h)
        start.append(h)
    lbm.lbm_batch_advance(b, 4, 0.0)
    lbm.lbm_batch_advance(b, 3, 0.0)
    lbm.lbm_batch_poll(b)
    for i, (g, nx, ny) in enumerate(INSTANCES):
        p = oracle_problem("half", n_half, g, nx, ny, 0.2, 0.004, -0.01)
        h5 = p.step(start[i], 5)
        h6 = p.step(h5, 1)
        ref = p.step(h6, 1)
        got = lbm.lbm_batch_get_state(b, i)
        assert np.abs(got - ref).max() <= 7 * 2e-6 * np.abs(ref).max(), (i, ny)
        st = lbm.lbm_batch_status(b, i)
        assert st["steps"] == 7 and abs(st["residual"] / oracle_residual(h6, h5) - 1) < 1e-4, (i, st)
    b.close()


def test_channels_freeze_at_the_residual_check():
    """A channel below the tolerance stops at its residual check, in either buffer, while the
    others march on."""
    vs = lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH, 2)
    probs = [lbm.make_problem(COUETTE, 1, ny, kn, 0.01, -0.01, prec=lbm.LBM_FP32_PERTURB, residual_every=5)
             for ny, kn in ((8, 10.0), (64, 0.05))]
    b = lbm.lbm_batch_init(vs, probs, stream=torch.cuda.Stream())
    lbm.lbm_batch_advance(b, 200, 1e-4)
    lbm.lbm_batch_poll(b)
    st = [lbm.lbm_batch_status(b, i) for i in range(2)]
    assert st[0]["converged"] and st[0]["steps"] < 200 and st[0]["residual"] < 1e-4
    p = oracle_problem("half", 2, COUETTE, 1, 8, 10.0, 0.01, -0.01)
    ref = p.step(p.zeros(), st[0]["steps"])
    assert np.abs(lbm.lbm_batch_get_state(b, 0) - ref).max() <= 2e-6 * st[0]["steps"] * np.abs(ref).max()
    assert st[1]["steps"] == 200 and not st[1]["converged"]
    b.close()
