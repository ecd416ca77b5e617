"""The network's forward pass with its output laid over its input: the bits of a pass into memory of
its own, whichever rows of the two overlap."""
import numpy as np
import pytest

from paper_1308_0692_gb300 import lbm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 129, 12001])
def test_output_over_input(rows):
    x = torch.from_numpy(np.random.default_rng(rows).uniform(-1, 1, (rows, 4)).astype(np.float32)).cuda()
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    m = lbm.lbm_mlp_create(rows, seed=3, stream=stream)
    want = torch.empty((rows, 6), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    lbm.lbm_mlp_forward(m, x.data_ptr(), rows, want.data_ptr())
    stream.synchronize()
    # y before x by some rows (y[0] .. on x[-a]), at x, and behind its first row
    for y_at, x_at in ((0, 0), (0, 8), (4, 0), (0, 4 * (rows // 2)), (4 * (rows - 1), 0)):
        buf = torch.zeros(12 * rows + 64, dtype=torch.float32, device="cuda")
        buf[x_at:x_at + 4 * rows] = x.reshape(-1)
        torch.cuda.synchronize()
        lbm.lbm_mlp_forward(m, buf.data_ptr() + 4 * x_at, rows, buf.data_ptr() + 4 * y_at)
        stream.synchronize()
        assert torch.equal(buf[y_at:y_at + 6 * rows].view(rows, 6), want), (y_at, x_at)
    m.close()
