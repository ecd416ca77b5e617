"""Second-order column march where its strips fill the chip and every block takes one chunk of rows
(1024 and 512 columns, rows of which the chunks do not divide), against the oracle's stored-state
steps at the tolerance of the narrower cavities (2e-6 a step of the largest value), with the residual
of a residual step."""
import math

import numpy as np
import pytest

from oracle.march import CAVITY, make_problem as oracle_problem
from paper_1308_0692_gb300 import lbm
from paper_1308_0692_gb300.inputs import random_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", [8, 9])
@pytest.mark.parametrize("n,nx,ny", [(6, 1024, 97), (4, 1024, 173), (6, 512, 179)])
def test_one_chunk_a_block_matches_oracle(n, nx, ny, path):
    p = oracle_problem("half", n, CAVITY, nx, ny, 0.05, 0.003, 0.01)
    refs = [p.relax_exp(random_state(p.n, p.ncells, seed=83), 0.5).astype(np.float32).astype(np.float64)]
    for _ in range(3):
        refs.append(p.relax_exp(p.transport2(refs[-1]), 1.0))
    vs = lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH, n)
    prob = lbm.make_problem(CAVITY, nx, ny, 0.05, 0.003, 0.01, prec=lbm.LBM_FP32_PERTURB, residual_every=2)
    sim = lbm.lbm_init(vs, prob, refs[0], stream=torch.cuda.Stream())
    lbm.lbm_set_transport(sim, 2)
    lbm.lbm_set_splitting(sim, lbm.LBM_SPLIT_STRANG_EXACT)
    lbm.lbm_set_variant(sim, n, path)
    lbm.lbm_step(sim, 3)
    got = lbm.lbm_get_state(sim)
    assert np.abs(got - refs[-1]).max() <= 3 * 2e-6 * np.abs(refs[-1]).max()
    r, at = lbm.lbm_residual(sim)
    want = math.sqrt(float(np.sum((refs[2] - refs[1]) ** 2)) / float(np.sum(refs[2] ** 2)))
    assert at == 2 and abs(r - want) <= 1e-3 * want
    sim.close()
