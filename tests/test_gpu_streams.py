"""GPU tests of StencilFn from several streams and threads: every call has its own
plan's workspace and exchange grids, and its own weights."""
import threading

import pytest

from paper_2605_07954_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07954_gb300 import build
    build.build()


def _step(x, W, T):
    """u_T and both gradients."""
    from paper_2605_07954_gb300 import StencilFn
    u, w = x.detach().clone().requires_grad_(True), W.clone().requires_grad_(True)
    y = StencilFn.apply(u, w, T)
    return (y.detach(),) + torch.autograd.grad(y, (u, w), torch.ones_like(y))


# a small grid (cluster-resident size), one of one tile per SM, and one of several waves of tiles
@pytest.mark.parametrize("shape", [(130, 517), (1000, 1022), (1801, 1804)])
def test_one_shape_on_two_streams(shape):
    W = torch.from_numpy(inputs.pattern_weights("star13"))
    xs = [torch.from_numpy(inputs.field(*shape, stream=60 + i)).cuda() for i in range(2)]
    want = [_step(x, W, 40) for x in xs]
    streams = [torch.cuda.Stream() for _ in xs]
    torch.cuda.synchronize()
    for _ in range(6):
        got = []
        for x, s in zip(xs, streams):
            with torch.cuda.stream(s):
                got.append(_step(x, W, 40))
        torch.cuda.synchronize()
        for g, w in zip(got, want):
            assert all(torch.equal(a, b) for a, b in zip(g, w))


@pytest.mark.parametrize("own_stream", [True, False])
def test_one_shape_from_two_threads(own_stream):
    """Two threads with different weights, on streams of their own and on one stream."""
    Ws = [torch.from_numpy(inputs.random_weights("star", 3, stream=70 + i)) for i in range(2)]
    x = torch.from_numpy(inputs.field(300, 420)).cuda()
    want = [_step(x, W, 24) for W in Ws]
    torch.cuda.synchronize()
    wrong = []

    def work(i):
        s = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
        with torch.cuda.stream(s):
            for _ in range(20):
                got = _step(x, Ws[i], 24)
                s.synchronize()
                if not all(torch.equal(a, b) for a, b in zip(got, want[i])):
                    wrong.append(i)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


def test_captured_after_a_warm_up_on_another_stream():
    from paper_2605_07954_gb300 import StencilFn
    W = torch.from_numpy(inputs.pattern_weights("heat5"))
    x = torch.from_numpy(inputs.field(260, 264)).cuda()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        want = StencilFn.apply(x, W, 30)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        y = StencilFn.apply(x, W, 30)
    for _ in range(3):
        y.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, want)
