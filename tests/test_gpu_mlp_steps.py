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


def test_weight_gradients_of_many_rows():
    """128 rows over and over: the row's factor 2 / (6 M) falls by a power of two, so the exact
    gradients are those of the 128 rows and the difference is what the FP32 accumulation loses.  An
    addition of a chain loses half an ulp, 2^-24 of its value then, at most on average; in chains of
    1024 rows (64 additions of 16 rows' products, the partial sum half the final one on average)
    that is 64 * 2^-25 of the sum."""
    rows = 32768
    for seed in range(2):
        rng = np.random.default_rng(seed)
        x = rng.uniform(-1, 1, (128, 4)).astype(np.float32)
        t = rng.standard_normal((128, 6)).astype(np.float32)
        grads = []
        for times in (1, rows // 128):
            m = lbm.lbm_mlp_create(128 * times, seed=4 + seed)
            xd, td = torch.from_numpy(np.tile(x, (times, 1))).cuda(), torch.from_numpy(np.tile(t, (times, 1))).cuda()
            torch.cuda.synchronize()
            grads.append(lbm.mlp_unflatten(lbm.lbm_mlp_loss_grad(m, xd.data_ptr(), td.data_ptr(), 128 * times)[1]))
            m.close()
        for (one, _), (many, _) in zip(*grads):
            one, many = np.asarray(one, dtype=np.float64), np.asarray(many, dtype=np.float64)
            assert np.linalg.norm(many - one) <= 64 * 2.0 ** -25 * np.linalg.norm(one)
