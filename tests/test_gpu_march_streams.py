"""Several contexts stepping at once, each on its own stream and host thread, beside other work on the GPU:
the launches of the multi-step kernel start when their blocks fit together, none gives up a wait, and
every context ends in the bits of a run alone."""
import threading

import pytest
import torch

from paper_2608_23786_gb300 import Ensemble, mclbm

pytestmark = pytest.mark.gpu

SHAPES = [(64, 4, "fp32", "pull", 60), (32, 3, "fp32", "aa", 150), (32, 2, "fp16", "pull", 150), (32, 1, "fp64", "aa", 40),
          (16, 5, "fp32", "pull", 150), (64, 4, "fp32", "aa", 61)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    mclbm.load(build_if_missing=True)


def _run(shape, calls, stream=None, limit=0):
    N, M, precision, pattern, steps = shape
    e = Ensemble(N, M, Re=12.5 * N, Ma=1.6 / 64, precision=precision, pattern=pattern, stream=stream).init()
    mclbm.mclbm_set_step_limit(e.ctx, limit)
    for _ in range(calls):
        e.step(steps)
    return e


@pytest.mark.parametrize("calls", [1, 4])
def test_contexts_on_streams_of_their_own(calls):
    alone = [_run(s, calls, limit=1) for s in SHAPES]
    torch.cuda.synchronize()
    a = torch.randn(4096, 4096, device="cuda")
    busy = torch.cuda.Stream()
    out = [None] * len(SHAPES)

    def work(k):
        out[k] = _run(SHAPES[k], calls, torch.cuda.Stream())

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(SHAPES))]
    for t in threads:
        t.start()
    with torch.cuda.stream(busy):
        for _ in range(20):
            a = torch.tanh(a @ a)
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for got, ref in zip(out, alone):
        mclbm.mclbm_device_status(got.ctx)
        assert mclbm.mclbm_get_step_launches(got.ctx)[0] == calls
        assert all(torch.equal(got.populations(m), ref.populations(m)) for m in range(ref.M))


@pytest.mark.parametrize("precision,N,M,pattern", [("fp32", 32, 7, "pull"), ("fp32", 64, 9, "aa"), ("fp16", 32, 2, "aa"),
                                                   ("fp64", 32, 2, "pull")])
def test_a_captured_call_replays(precision, N, M, pattern):
    """A call of an even number of steps inside a CUDA graph capture, replayed: the bits of the same steps
    taken one at a time."""
    stream = torch.cuda.Stream()
    e = Ensemble(N, M, Re=12.5 * N, Ma=1.6 / 64, precision=precision, pattern=pattern, stream=stream).init()
    e.step(20)
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        e.step(20)
    assert mclbm.mclbm_get_step_launches(e.ctx) == (2, 40)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    mclbm.mclbm_device_status(e.ctx)
    ref = Ensemble(N, M, Re=12.5 * N, Ma=1.6 / 64, precision=precision, pattern=pattern).init()
    mclbm.mclbm_set_step_limit(ref.ctx, 1)
    ref.step(80)
    assert all(torch.equal(e.populations(m), ref.populations(m)) for m in range(M))
