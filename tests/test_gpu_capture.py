"""GPU: a step given to a stream that is being captured leaves later steps as they would have been without it."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from helpers import MU  # noqa: E402
from paper_2504_05295_b200 import binding  # noqa: E402

THREAD_LOCAL = 1      # cudaStreamCaptureModeThreadLocal


def problem(m, n, r):
    g = torch.Generator(device="cuda"); g.manual_seed(5)
    rn = lambda *s: torch.randn(*s, generator=g, device="cuda")
    return rn(m, n) * 0.02, rn(m, n) * 0.3, rn(m, n) * 0.1, rn(n, r) / n ** 0.5


@pytest.mark.parametrize("rate", [0.01, 0.02])
def test_learning_rate_after_a_capture(rate):
    # a matrix small enough to be stepped by replaying a graph that reads the rate from memory; the runtime may refuse to
    # record that replay, and then nothing of the call has run
    cudart = ctypes.CDLL("libcudart.so.12")
    rates = [0.01, 0.02, 0.01]
    X, M, G, Q = problem(512, 384, 64)
    with binding.Dion(mu=MU) as opt:
        for lr in rates:
            opt.step(X, M, G, Q, lr)
        want = [t.clone() for t in (X, M, Q)]
    X, M, G, Q = problem(512, 384, 64)
    side = torch.cuda.Stream()
    graph, replay = ctypes.c_void_p(), ctypes.c_void_p()
    with binding.Dion(mu=MU) as opt:
        opt.step(X, M, G, Q, rates[0])
        torch.cuda.synchronize()
        assert cudart.cudaStreamBeginCapture(ctypes.c_void_p(side.cuda_stream), THREAD_LOCAL) == 0
        try:
            opt.step(X, M, G, Q, rate, stream=side)
            recorded = True
        except binding.DionError:
            recorded = False
        recorded = cudart.cudaStreamEndCapture(ctypes.c_void_p(side.cuda_stream), ctypes.byref(graph)) == 0 and recorded
        cudart.cudaGetLastError()
        for lr in rates[1:]:
            opt.step(X, M, G, Q, lr)
        assert opt.get_status() == (0, 0)
        for name, a, b in zip("XMQ", (X, M, Q), want):
            assert torch.equal(a, b), name
        if recorded:      # the recorded step keeps its rate, and a direct step after it its own
            Y = [t.clone() for t in (X, M, Q)]
            assert cudart.cudaGraphInstantiate(ctypes.byref(replay), graph, ctypes.c_ulonglong(0)) == 0
            torch.cuda.synchronize()
            assert cudart.cudaGraphLaunch(replay, ctypes.c_void_p(side.cuda_stream)) == 0
            side.synchronize()
            opt.step(X, M, G, Q, rates[0])
            torch.cuda.synchronize()
            with binding.Dion(mu=MU) as other:
                for lr in (rate, rates[0]):
                    other.step(Y[0], Y[1], G, Y[2], lr)
                torch.cuda.synchronize()
            for name, a, b in zip("XMQ", (X, M, Q), Y):
                assert torch.equal(a, b), name
    # (the thread's own generator and allocator know nothing of the capture)
    assert torch.isfinite(torch.randn(4, device="cuda")).all()
