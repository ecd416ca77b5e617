"""One-column channels marched on a cluster (step_column.cu) against the oracle, and the unfolded
FP64 relaxation (1 - omega near zero) of the planar kernels.

Channels of one cell per CTA, of empty and half-filled CTAs, and the longest the kernel takes,
every velocity-set size, steps that end between, on and after residual checks.  Tolerances as in
test_gpu_step.py (FP64 1e-12 of max |h|, FP32 2e-6 per step): the update is the same."""
import math

import numpy as np
import pytest

from oracle.march import CAVITY, COUETTE, make_problem as oracle_problem, residual as oracle_residual
from paper_1308_0692_gb300 import lbm
from paper_1308_0692_gb300.inputs import random_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SETS = [("full", 3), ("half", 2), ("half", 3), ("half", 4), ("half", 6)]


def _run(kind, n, geom, nx, ny, kn, prec, calls, every, seed, splitting=0):
    p = oracle_problem(kind, n, geom, nx, ny, kn, 0.004, -0.01)
    h = random_state(p.n, p.ncells, seed=seed)
    if prec == lbm.LBM_FP32_PERTURB:
        h = h.astype(np.float32).astype(np.float64)
    vs = lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH if kind == "half" else lbm.LBM_FULL_RANGE_GH, n)
    sim = lbm.lbm_init(vs, lbm.make_problem(geom, nx, ny, kn, 0.004, -0.01, prec=prec, residual_every=every), h,
                       stream=torch.cuda.Stream())
    tol = 1e-12 if prec == lbm.LBM_FP64 else 2e-6
    done = 0
    for k in calls:
        lbm.lbm_step(sim, k)
        h = p.step(h, k - 1) if k > 1 else h
        h, before = p.step(h, 1), h
        done += k
        got = lbm.lbm_get_state(sim)
        assert np.abs(got - h).max() <= tol * (done if prec == lbm.LBM_FP32_PERTURB else 1) * np.abs(h).max(), (done,)
        if done % every == 0:
            r, step = lbm.lbm_residual(sim)
            assert step == done and abs(r / oracle_residual(h, before) - 1) <= (1e-9 if prec == lbm.LBM_FP64 else 1e-4)
    sim.close()


@pytest.mark.parametrize("prec", [lbm.LBM_FP64, lbm.LBM_FP32_PERTURB])
@pytest.mark.parametrize("ny", [2, 16, 17, 33, 300, 450, 513])
@pytest.mark.parametrize("kind,n", SETS)
def test_channel_matches_oracle(kind, n, ny, prec):
    _run(kind, n, COUETTE, 1, ny, 0.07, prec, (5, 1, 4, 2), 3, seed=ny)


@pytest.mark.parametrize("geom,nx,ny", [(COUETTE, 1, 21), (CAVITY, 19, 23)])
@pytest.mark.parametrize("kn", [1e-4, math.inf])
def test_relaxation_factors_at_both_ends(geom, nx, ny, kn):
    """dt = Kn (1 - omega = 0) and no collisions (omega = 0)."""
    _run("half", 4, geom, nx, ny, kn, lbm.LBM_FP64, (3, 3), 3, seed=5)
