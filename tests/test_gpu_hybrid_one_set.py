"""Hybrid cavities whose cells all carry one velocity set (no interface cells): each step lets the next
one's blocks be set up at its end.  Steps in flight against the oracle (tolerances as in
test_gpu_hybrid_order.py) and, bit for bit, against steps that the host waits for; grids of fewer and
of more blocks than SMs, and on both sides of two and a half blocks an SM."""
import numpy as np
import pytest

from oracle import hybrid as hy
from paper_1308_0692_gb300 import lbm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# n_half, nx, ny, layer (0: full-range, 1000: half-range)
CASES = [(2, 33, 31, 0), (3, 70, 66, 1000), (4, 128, 128, 0), (4, 65, 63, 1000), (6, 120, 100, 0), (3, 210, 224, 0), (2, 120, 120, 1000),
         (5, 161, 158, 1000)]


def _cavity(case, prec, h):
    n, nx, ny, layer = case
    hb = lbm.lbm_hybrid_init(lbm.LBM_CAVITY, n, nx, ny, 0.1, 0.0, 0.01, layer, stream=torch.cuda.Stream())
    lbm.lbm_hybrid_set_state(hb, h)
    lbm.lbm_hybrid_set_precision(hb, prec)
    return hb


@pytest.mark.parametrize("prec", [lbm.LBM_FP64, lbm.LBM_FP32_PERTURB])
@pytest.mark.parametrize("case", CASES)
def test_steps_of_one_velocity_set(case, prec):
    n, nx, ny, layer = case
    p = hy.HybridCavity(n, nx, ny, 0.1, 0.0, 0.01, layer)
    rng = np.random.default_rng(nx + layer)
    h0 = [(rng.standard_normal(p.vset(c).n) * 1e-2).astype(np.float32).astype(np.float64) for c in range(p.ncells)]
    packed = np.concatenate(h0)
    hb = _cavity(case, prec, packed)
    lbm.lbm_hybrid_step(hb, 2)
    want = np.concatenate([np.asarray(v) for v in p.step(h0, 2)])
    tol = 1e-12 if prec == lbm.LBM_FP64 else 2 * 2e-6
    assert np.abs(lbm.lbm_hybrid_get_state(hb) - want).max() <= tol * np.abs(want).max()
    hb.close()
    got = []
    for calls in ((40,), (1,) * 40):
        hb = _cavity(case, prec, packed)
        for k in calls:
            lbm.lbm_hybrid_step(hb, k)
            if len(calls) > 1:
                torch.cuda.synchronize()
        got.append(lbm.lbm_hybrid_get_state(hb))
        hb.close()
    assert np.isfinite(got[0]).all() and np.array_equal(got[0], got[1])
