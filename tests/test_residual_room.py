"""Room for the residual's partial sums in a simulation's buffer: as much as the finest launch on its
grid writes, no more, and every variant and the refinement fit in it."""
import numpy as np
import pytest

from paper_1308_0692_gb300 import lbm

SETS = [(lbm.LBM_FULL_RANGE_GH, 3), (lbm.LBM_HALF_RANGE_GH, 2), (lbm.LBM_HALF_RANGE_GH, 3), (lbm.LBM_HALF_RANGE_GH, 4),
        (lbm.LBM_HALF_RANGE_GH, 6)]


@pytest.mark.parametrize("prec", [lbm.LBM_FP64, lbm.LBM_FP32_PERTURB])
@pytest.mark.parametrize("kind,n", SETS)
def test_buffer_is_the_states_and_the_diagnostics_and_little_more(kind, n, prec):
    """Two FP64 or four FP32 states and eight FP64 fields a cell; partial sums of a block of at least
    eight cells take two bytes a cell."""
    vs = lbm.lbm_make_velocity_set(kind, n)
    nx, ny = 1000, 900
    nv = len(lbm.lbm_vset_query(vs)[0])
    total = lbm.lbm_sim_bytes(vs, lbm.make_problem(lbm.LBM_CAVITY, nx, ny, 0.1, 0.0, 0.01, prec=prec))
    assert total - (16 * nv + 64) * nx * ny <= 2 * nx * ny + 100_000


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [lbm.LBM_FP64, lbm.LBM_FP32_PERTURB])
@pytest.mark.parametrize("kind,n", SETS)
def test_every_variant_fits(kind, n, prec):
    torch = pytest.importorskip("torch")
    vs = lbm.lbm_make_velocity_set(kind, n)
    for geom, nx, ny in [(lbm.LBM_CAVITY, 2, 3), (lbm.LBM_CAVITY, 3, 301), (lbm.LBM_CAVITY, 301, 2), (lbm.LBM_COUETTE, 1, 777),
                         (lbm.LBM_COUETTE, 2, 2), (lbm.LBM_CAVITY, 157, 159), (lbm.LBM_CAVITY, 320, 333)]:
        sim = lbm.lbm_init(vs, lbm.make_problem(geom, nx, ny, 0.1, 0.0, 0.01, prec=prec, residual_every=1),
                           stream=torch.cuda.Stream())
        steps = 0
        for g in [None] + list(range(1, 13)):
            for path in (0, 1):
                if g is not None:
                    try:
                        lbm.lbm_set_variant(sim, g, path)
                    except lbm.LBMError as e:
                        assert e.status == lbm.LBM_EUNSUPPORTED, (g, path, nx, ny)
                        continue
                lbm.lbm_step(sim, 2)
                steps += 2
                r, at = lbm.lbm_residual(sim)
                assert at == steps and np.isfinite(r)
        if prec == lbm.LBM_FP32_PERTURB:
            lbm.lbm_solve(sim, 1e-3, 20, 1, 1e-4)
        sim.close()
