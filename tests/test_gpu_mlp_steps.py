"""Training steps of the warm-start network one behind another: nothing may depend on whether the
host waits between them."""
import numpy as np
import pytest

from paper_1308_0692_gb300 import lbm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_steps_in_flight_equal_steps_waited_for():
    """Parameters after steps of changing row counts, bit for bit (every sum has a fixed order)."""
    rng = np.random.default_rng(3)
    rows = [700, 9000, 1, 128, 9000, 129, 2048, 9000] * 4
    x = torch.from_numpy(rng.uniform(-1, 1, (9000, 4)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.standard_normal((9000, 6)).astype(np.float32)).cuda()
    torch.cuda.synchronize()
    got = []
    for wait in (False, True, False):
        stream = torch.cuda.Stream()
        m = lbm.lbm_mlp_create(9000, seed=2, stream=stream)
        for r in rows:
            lbm.lbm_mlp_train_step(m, x.data_ptr(), t.data_ptr(), r, 1e-2)
            if wait:
                stream.synchronize()
        got.append(lbm.lbm_mlp_get_params(m))
        m.close()
    assert np.isfinite(got[0]).all()
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[2], got[1])
