"""Hybrid cavities of more than four blocks per SM, whose interface blocks alternate with the
tile blocks, and one with more interface than tile blocks, whose order stays: every cell is
stepped once, against the FP64 numpy oracle (oracle/hybrid.py) from a seeded random state, at the
tolerances of the smaller cavities (1e-12 in FP64, 2e-6 a step in FP32, of the largest value)."""
import numpy as np
import pytest

from oracle import hybrid as hy
from paper_1308_0692_gb300 import lbm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [
    # n_half, nx, ny, layer (kn 0.1, lid 0.01)
    (3, 200, 190, 8),       # 357 interface blocks, 391 others
    (2, 211, 203, 3),       # ragged tiles, 401 and 568
    (5, 180, 171, 20),      # 270 and 403
    (4, 230, 220, 1),       # 445 and 436: interface blocks first
]


@pytest.mark.parametrize("prec", [lbm.LBM_FP64, lbm.LBM_FP32_PERTURB])
@pytest.mark.parametrize("case", CASES)
def test_every_cell_of_a_large_cavity_is_stepped(case, prec):
    from paper_1308_0692_gb300 import build
    build.build()
    n, nx, ny, layer = case
    p = hy.HybridCavity(n, nx, ny, 0.1, 0.0, 0.01, layer)
    rng = np.random.default_rng(nx + layer)
    h0 = [(rng.standard_normal(p.vset(c).n) * 1e-2).astype(np.float32).astype(np.float64) for c in range(p.ncells)]
    hb = lbm.lbm_hybrid_init(lbm.LBM_CAVITY, n, nx, ny, 0.1, 0.0, 0.01, layer, stream=torch.cuda.Stream())
    lbm.lbm_hybrid_set_state(hb, np.concatenate(h0))
    lbm.lbm_hybrid_set_precision(hb, prec)
    lbm.lbm_hybrid_step(hb, 2)
    got = lbm.lbm_hybrid_get_state(hb)
    want = np.concatenate([np.asarray(v) for v in p.step(h0, 2)])
    tol = 1e-12 if prec == lbm.LBM_FP64 else 2 * 2e-6
    assert np.abs(got - want).max() <= tol * np.abs(want).max()
    hb.close()
