"""Block shapes of the step kernel (step_tile.cuh) on grids beyond the L2 and at the lines between
them: against the oracle on both sides of a line where that is small enough, else against the
shape of explicitly chosen slices, which the small grids compare with the oracle.  Tolerances as in
test_gpu_step.py (FP64 1e-12 of max |h|, FP32 2e-6 per step)."""
import numpy as np
import pytest

from oracle.march import CAVITY, make_problem as oracle_problem
from paper_1308_0692_gb300 import lbm
from paper_1308_0692_gb300.inputs import random_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

F64, F32 = lbm.LBM_FP64, lbm.LBM_FP32_PERTURB


def _sim(kind, n, nx, ny, prec, h0, every=100):
    vs = lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH if kind == "half" else lbm.LBM_FULL_RANGE_GH, n)
    return lbm.lbm_init(vs, lbm.make_problem(lbm.LBM_CAVITY, nx, ny, 0.07, 0.004, -0.01, prec=prec, residual_every=every), h0,
                        stream=torch.cuda.Stream())


@pytest.mark.parametrize("kind,n,nx,ny,prec,slices", [
    ("full", 3, 143, 141, F32, None),       # 20163 cells
    ("half", 2, 251, 240, F64, None),       # 60240 cells: whole rows a thread
    ("half", 2, 251, 240, F64, 2),
    ("half", 3, 317, 316, F64, None),       # 100172 cells: two slices
    ("half", 6, 179, 168, F32, None),       # 30072 cells: four slices of 32 places
    ("half", 6, 61, 37, F32, 6),
    ("half", 6, 61, 37, F64, 3),
    ("half", 6, 61, 37, F64, 6),
    ("half", 4, 61, 37, F64, 2),
])
def test_shape_matches_oracle(kind, n, nx, ny, prec, slices):
    p = oracle_problem(kind, n, CAVITY, nx, ny, 0.07, 0.004, -0.01)
    h0 = random_state(p.n, p.ncells, seed=nx + 7 * ny).astype(np.float32).astype(np.float64)
    sim = _sim(kind, n, nx, ny, prec, h0)
    if slices:
        lbm.lbm_set_variant(sim, slices, 0)
    lbm.lbm_step(sim, 2)
    ref = p.step(h0, 2)
    assert np.abs(lbm.lbm_get_state(sim) - ref).max() <= (1e-12 if prec == F64 else 2 * 2e-6) * np.abs(ref).max()
    sim.close()


@pytest.mark.parametrize("n,slices", [(3, 1), (4, 2), (6, 3)])
def test_large_grid_matches_chosen_slices(n, slices):
    nx, ny = 1451, 1381                     # 2003831 cells: two rows of 32 places
    rng = np.random.default_rng(n)
    got = []
    h0 = rng.standard_normal((4 * n * n, nx * ny), dtype=np.float32)
    for g in (None, slices):
        sim = _sim("half", n, nx, ny, F32, None)
        lbm.lbm_set_state_f32(sim, h0)
        if g:
            lbm.lbm_set_variant(sim, g, 0)
        lbm.lbm_step(sim, 1)
        got.append(lbm.lbm_get_state_f32(sim))
        sim.close()
    assert np.abs(got[0] - got[1]).max() <= 2e-6 * np.abs(got[1]).max()


@pytest.mark.parametrize("n,nx,ny", [(2, 251, 240), (3, 317, 316), (6, 179, 168)])
def test_correction_continues_the_march(n, nx, ny):
    """The equation is linear: k correction steps from the defect of h are k steps of the FP64 march from h."""
    p = oracle_problem("half", n, CAVITY, nx, ny, 0.07, 0.004, -0.01)
    h0 = random_state(p.n, p.ncells, seed=n).astype(np.float32).astype(np.float64)
    plain, refined = (_sim("half", n, nx, ny, F32, h0, every=10) for _ in range(2))
    lbm.lbm_solve(plain, 1e-13, 10)
    info = lbm.lbm_solve(refined, 1e-13, 10, 1, 1e-13)
    k = info["correction_steps"]
    assert k == 10
    ref = p.step(lbm.lbm_get_state(plain), k)
    assert np.abs(lbm.lbm_get_state(refined) - ref).max() <= 2e-6 * (k + 1) * np.abs(ref).max()
    plain.close()
    refined.close()
