"""The variant that a simulation reports by itself, set again, changes nothing: the same kernels run
(the same bits), and it is the way back from a variant chosen in between."""
import numpy as np
import pytest

from paper_1308_0692_gb300 import lbm
from paper_1308_0692_gb300.inputs import random_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom,nx,ny,n,prec,other", [
    (lbm.LBM_COUETTE, 1, 100, 4, lbm.LBM_FP64, (2, 0)),
    (lbm.LBM_COUETTE, 1, 300, 6, lbm.LBM_FP32_PERTURB, (2, 0)),
    (lbm.LBM_CAVITY, 40, 33, 4, lbm.LBM_FP64, (2, 0)),
    (lbm.LBM_CAVITY, 40, 33, 4, lbm.LBM_FP32_PERTURB, (4, 0)),
    (lbm.LBM_CAVITY, 128, 40, 6, lbm.LBM_FP32_PERTURB, (6, 8)),
    (lbm.LBM_CAVITY, 40, 33, 2, lbm.LBM_FP64, (2, 0)),
])
def test_reported_variant_set_again_changes_nothing(geom, nx, ny, n, prec, other):
    vs = lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH, n)
    h = random_state(4 * n * n, nx * ny, seed=nx + ny)
    got = []
    for way in ("as it is", "set again", "there and back"):
        sim = lbm.lbm_init(vs, lbm.make_problem(geom, nx, ny, 0.07, 0.004, -0.01, prec=prec, residual_every=10), h,
                           stream=torch.cuda.Stream())
        first = lbm.lbm_get_variant(sim)
        if way == "there and back":
            lbm.lbm_set_variant(sim, *other)
            assert lbm.lbm_get_variant(sim) == other
        if way != "as it is":
            lbm.lbm_set_variant(sim, *first)
        assert lbm.lbm_get_variant(sim) == first
        lbm.lbm_step(sim, 25)
        got.append((lbm.lbm_get_state(sim), lbm.lbm_residual(sim)))
        sim.close()
    for state, resid in got[1:]:
        assert np.array_equal(state, got[0][0]) and resid == got[0][1]
