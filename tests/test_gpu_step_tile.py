"""Default step kernel (step_tile.cuh) at the edges of its block shapes, against the oracle.

The block shape depends on the velocity set, the precision and the cell count: grids whose
rows and cell counts are no multiples of the block's places and rows, the smallest grids, and
both sides of every cell-count line of the choice.  Tolerances as in test_gpu_step.py (FP64
1e-12 of max |h|, FP32 2e-6 per step): the kernel evaluates the same update.
"""
import numpy as np
import pytest

from oracle.march import CAVITY, COUETTE, make_problem as oracle_problem, residual as oracle_residual
from paper_1308_0692_gb300 import lbm
from paper_1308_0692_gb300.inputs import random_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOTH = (lbm.LBM_FP64, lbm.LBM_FP32_PERTURB)
CASES = [
    # kind, n, geom, nx, ny, precisions
    ("full", 3, CAVITY, 33, 7, BOTH),            # two rows a block, odd row count
    ("full", 3, COUETTE, 1, 3, BOTH),            # one column, last block half empty in y
    ("half", 2, CAVITY, 3, 2, BOTH),
    ("half", 2, COUETTE, 5, 13, BOTH),
    ("half", 2, CAVITY, 63, 64, (lbm.LBM_FP32_PERTURB,)),      # 4032 cells: whole rows a thread
    ("half", 2, CAVITY, 251, 201, (lbm.LBM_FP32_PERTURB,)),    # 50451 cells: 32 places
    ("half", 3, CAVITY, 9, 11, BOTH),
    ("half", 3, CAVITY, 143, 141, (lbm.LBM_FP32_PERTURB,)),    # 20163 cells
    ("half", 4, CAVITY, 49, 53, (lbm.LBM_FP32_PERTURB,)),      # 2597 cells: two rows a thread
    ("half", 4, CAVITY, 7, 5, BOTH),
    ("half", 4, COUETTE, 1, 33, BOTH),
    ("half", 4, CAVITY, 158, 159, (lbm.LBM_FP64,)),            # 25122 cells: two rows a thread
    ("half", 4, CAVITY, 229, 219, (lbm.LBM_FP32_PERTURB,)),    # 50151 cells: 32 places
    ("half", 6, CAVITY, 5, 3, BOTH),
    ("half", 6, COUETTE, 2, 17, BOTH),
    ("half", 6, CAVITY, 317, 316, (lbm.LBM_FP64,)),            # 100172 cells: three rows a thread
]


@pytest.mark.parametrize("case", [c[:5] + (p,) for c in CASES for p in c[5]],
                         ids=lambda c: f"{c[0]}{c[1]}-{'cav' if c[2] else 'cou'}-{c[3]}x{c[4]}-{'f32' if c[5] else 'f64'}")
def test_default_step_matches_oracle(case):
    kind, n, geom, nx, ny, prec = case
    p = oracle_problem(kind, n, geom, nx, ny, 0.07, 0.004, -0.01)
    h0 = random_state(p.n, p.ncells, seed=nx + 7 * ny)
    if prec == lbm.LBM_FP32_PERTURB:
        h0 = h0.astype(np.float32).astype(np.float64)
    vs = lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH if kind == "half" else lbm.LBM_FULL_RANGE_GH, n)
    sim = lbm.lbm_init(vs, lbm.make_problem(geom, nx, ny, 0.07, 0.004, -0.01, prec=prec, residual_every=2), h0,
                       stream=torch.cuda.Stream())
    lbm.lbm_step(sim, 4)                         # one graph replay per buffer parity
    before = p.step(h0, 3)
    ref = p.step(before, 1)
    tol = 1e-12 if prec == lbm.LBM_FP64 else 4 * 2e-6
    assert np.abs(lbm.lbm_get_state(sim) - ref).max() <= tol * np.abs(ref).max()
    r, step = lbm.lbm_residual(sim)
    assert step == 4 and abs(r / oracle_residual(ref, before) - 1) <= (1e-9 if prec == lbm.LBM_FP64 else 1e-4)
    sim.close()
