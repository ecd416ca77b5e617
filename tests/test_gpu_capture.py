"""Calls made while the caller captures the object's stream into a CUDA graph: steps go into the
graph and replay to the same bits as direct launches, a warm start (which synchronises) is refused
before it enqueues anything, so that the capture stays usable."""
import numpy as np
import pytest

from paper_1308_0692_gb300 import lbm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _captured(stream, call):
    from paper_1308_0692_gb300 import build
    build.build()
    junk = torch.empty(1000, device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        junk.zero_()                       # nodes that are not kernels of the library around the call
        call()
        junk.zero_()
    graph.replay()
    torch.cuda.synchronize()


def _sim(geom, nx, ny, prec, stream):
    vs = lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH, 4)
    return lbm.lbm_init(vs, lbm.make_problem(geom, nx, ny, 0.1, 0.0, 0.01, prec=prec, residual_every=5), stream=stream)


@pytest.mark.parametrize("prec", [lbm.LBM_FP64, lbm.LBM_FP32_PERTURB])
@pytest.mark.parametrize("geom,nx,ny", [(lbm.LBM_COUETTE, 1, 40), (lbm.LBM_CAVITY, 40, 33)])
def test_captured_steps_equal_direct_ones(geom, nx, ny, prec):
    stream = torch.cuda.Stream()
    a, b = _sim(geom, nx, ny, prec, stream), _sim(geom, nx, ny, prec, stream)
    for k in (3, 12):
        lbm.lbm_step(a, k)
        _captured(stream, lambda: lbm.lbm_step(b, k))
    assert np.array_equal(lbm.lbm_get_state(a), lbm.lbm_get_state(b))
    assert lbm.lbm_residual(a) == lbm.lbm_residual(b)


@pytest.mark.parametrize("prec", [lbm.LBM_FP64, lbm.LBM_FP32_PERTURB])
def test_captured_hybrid_steps_equal_direct_ones(prec):
    stream = torch.cuda.Stream()
    pair = [lbm.lbm_hybrid_init(lbm.LBM_CAVITY, 4, 48, 40, 0.1, 0.0, 0.01, 4, stream=stream) for _ in range(2)]
    for hb in pair:
        lbm.lbm_hybrid_set_precision(hb, prec)
    for k in (1, 6):
        lbm.lbm_hybrid_step(pair[0], k)
        _captured(stream, lambda: lbm.lbm_hybrid_step(pair[1], k))
    assert np.array_equal(lbm.lbm_hybrid_get_state(pair[0]), lbm.lbm_hybrid_get_state(pair[1]))


def test_warm_start_is_refused_under_capture():
    stream = torch.cuda.Stream()
    sim = _sim(lbm.LBM_CAVITY, 32, 32, lbm.LBM_FP32_PERTURB, stream)
    net = lbm.lbm_mlp_create(1024, seed=0, stream=torch.cuda.Stream())
    lbm.lbm_warm_start(sim, net, 0.1, 0.01)
    h = lbm.lbm_get_state(sim)

    def call():
        with pytest.raises(lbm.LBMError) as e:
            lbm.lbm_warm_start(sim, net, 0.1, 0.01)
        assert e.value.status == lbm.LBM_ECUDA
    _captured(stream, call)
    lbm.lbm_warm_start(sim, net, 0.1, 0.01)
    assert np.array_equal(lbm.lbm_get_state(sim), h)
