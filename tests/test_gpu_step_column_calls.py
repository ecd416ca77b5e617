"""One-column channels: the state does not depend on how the steps are dealt to calls, nor on where
the residual checks fall, bit for bit; and the longest channels that each velocity set's cluster
takes, against the oracle (tolerances as in test_gpu_step_column.py)."""
import numpy as np
import pytest

from oracle.march import COUETTE, make_problem as oracle_problem
from paper_1308_0692_gb300 import lbm
from paper_1308_0692_gb300.inputs import random_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SETS = [("full", 3), ("half", 2), ("half", 3), ("half", 4), ("half", 6)]


def _sim(kind, n, ny, prec, h, every):
    vs = lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH if kind == "half" else lbm.LBM_FULL_RANGE_GH, n)
    prob = lbm.make_problem(COUETTE, 1, ny, 0.07, 0.004, -0.01, prec=prec, residual_every=every)
    return lbm.lbm_init(vs, prob, h, stream=torch.cuda.Stream())


@pytest.mark.parametrize("prec", [lbm.LBM_FP64, lbm.LBM_FP32_PERTURB])
@pytest.mark.parametrize("ny", [2, 17, 100, 300])
@pytest.mark.parametrize("kind,n", SETS)
def test_bits_do_not_depend_on_the_calls(kind, n, ny, prec):
    m = n if kind == "full" else 2 * n
    h = random_state(m * m, ny, seed=ny)
    got = []
    for calls, every in (((48,), 100), ((24, 24), 100), ((1, 5, 42), 100), ((48,), 7), ((48,), 1)):
        sim = _sim(kind, n, ny, prec, h, every)
        for k in calls:
            lbm.lbm_step(sim, k)
        got.append(lbm.lbm_get_state(sim))
        sim.close()
    assert all(np.array_equal(g, got[0]) for g in got[1:])


@pytest.mark.parametrize("prec", [lbm.LBM_FP64, lbm.LBM_FP32_PERTURB])
@pytest.mark.parametrize("kind,n", SETS)
def test_longest_channels_match_oracle(kind, n, prec):
    p = oracle_problem(kind, n, COUETTE, 1, 512, 0.07, 0.004, -0.01)
    h = random_state(p.n, p.ncells, seed=8)
    if prec == lbm.LBM_FP32_PERTURB:
        h = h.astype(np.float32).astype(np.float64)
    sim = _sim(kind, n, 512, prec, h, 3)
    lbm.lbm_step(sim, 8)
    ref = p.step(h, 8)
    tol = 1e-12 if prec == lbm.LBM_FP64 else 8 * 2e-6
    assert np.abs(lbm.lbm_get_state(sim) - ref).max() <= tol * np.abs(ref).max()
    sim.close()
