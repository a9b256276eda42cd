"""jkcals_mttkrp of an FP64 handle into device memory is only enqueued, on the products' route as on
the CUDA-core kernel: it returns while earlier work of the stream still runs, and it can be
captured into a caller's graph, whose replays follow the handle's factors."""
import numpy as np
import pytest

from paper_2112_03985_gb300 import api

pytestmark = pytest.mark.gpu

DIMS, C = (40, 33, 61), 205


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _handle(stream, native):
    rng = np.random.default_rng(3)
    kw = dict(max_device_bytes=1 << 46) if native else {}
    U = [rng.random((I, C)) for I in DIMS]
    return api.JKCALS(rng.random(DIMS), 0, [5] * 41, [[] for _ in range(41)], U, stream=stream.cuda_stream, **kw), U


@pytest.mark.parametrize("native", [False, True], ids=["products", "cuda-cores"])
def test_returns_while_the_stream_is_busy(native):
    torch = _torch()
    s = torch.cuda.Stream()
    h, _ = _handle(s, native)
    with h, torch.cuda.stream(s):
        outs = [torch.empty((I, C), dtype=torch.float64, device="cuda") for I in DIMS]
        want = [h.mttkrp(n) for n in range(3)]
        done = torch.cuda.Event()
        torch.cuda._sleep(400_000_000)          # a fifth of a second
        for n in range(3):
            h.mttkrp(n, out=outs[n])
        done.record()
        assert not done.query()
        h.sync()
        for n in range(3):
            np.testing.assert_array_equal(outs[n].cpu().numpy(), want[n])


@pytest.mark.parametrize("native", [False, True], ids=["products", "cuda-cores"])
def test_captured_into_a_callers_graph(native):
    torch = _torch()
    s = torch.cuda.Stream()
    h, U = _handle(s, native)
    with h:
        outs = [torch.empty((I, C), dtype=torch.float64, device="cuda") for I in DIMS]
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            for n in range(3):
                h.mttkrp(n, out=outs[n])
        for scale in (1.0, 2.0):
            h.set_factors([scale * u for u in U])
            want = [h.mttkrp(n) for n in range(3)]
            for o in outs:
                o.zero_()
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            for n in range(3):
                np.testing.assert_array_equal(outs[n].cpu().numpy(), want[n])
        h.sync()
