"""Calls that a capture of one of their streams into a CUDA graph refuses: before they enqueue
anything, so that the capture stays usable and the call works afterwards."""
import numpy as np
import pytest

from paper_1308_0692_gb300 import lbm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _refused_under_capture(stream, call):
    junk = torch.ones(1000, device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        junk.add_(1)
        with pytest.raises(lbm.LBMError) as e:
            call()
        assert e.value.status == lbm.LBM_ECUDA
        junk.add_(1)
    graph.replay()
    torch.cuda.synchronize()
    assert bool((junk == 3).all())


def _problem(nx=32, ny=32):
    return lbm.make_problem(lbm.LBM_CAVITY, nx, ny, 0.1, 0.0, 0.01, prec=lbm.LBM_FP32_PERTURB, residual_every=5)


@pytest.mark.parametrize("captured", ["object", "network"])
@pytest.mark.parametrize("kind", ["simulation", "batch"])
def test_warm_start_with_either_stream_under_capture(kind, captured):
    stream, net_stream = torch.cuda.Stream(), torch.cuda.Stream()
    vs = lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH, 4)
    net = lbm.lbm_mlp_create(1024, seed=0, stream=net_stream)
    if kind == "simulation":
        obj = lbm.lbm_init(vs, _problem(), stream=stream)
        call, state = (lambda: lbm.lbm_warm_start(obj, net, 0.1, 0.01)), (lambda: lbm.lbm_get_state(obj))
    else:
        obj = lbm.lbm_batch_init(vs, [_problem()], stream=stream)
        call, state = (lambda: lbm.lbm_batch_warm_start(obj, 0, net, 0.1, 0.01)), (lambda: lbm.lbm_batch_get_state(obj, 0))
    call()
    h = state()
    _refused_under_capture(stream if captured == "object" else net_stream, call)
    call()
    assert np.array_equal(state(), h)


def test_batch_moments_under_capture():
    stream = torch.cuda.Stream()
    b = lbm.lbm_batch_init(lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH, 4), [_problem()], stream=stream)
    lbm.lbm_batch_advance(b, 3, 0.0)
    out = torch.full((6, 32, 32), -7.0, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    _refused_under_capture(stream, lambda: lbm.lbm_batch_moments(b, 0, out.data_ptr()))
    assert bool((out == -7.0).all())
    lbm.lbm_batch_moments(b, 0, out.data_ptr())
    stream.synchronize()
    assert bool((out[0] > 0.5).all())
