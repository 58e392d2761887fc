"""The network's calls in stream order: a handle created while the default
stream is busy, and a handle whose stream changes while work is queued."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPE = (5, 64, 2, 9)
BUSY = 400_000_000  # cycles: about 0.2 s


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _theta(n, seed=0):
    return (0.3 * np.random.default_rng(seed).standard_normal(n)).astype(np.float32)


def _data(rows=48):
    import torch
    rng = np.random.default_rng(1)
    x = torch.from_numpy(rng.standard_normal((rows, SHAPE[0])).astype(np.float32))
    t = torch.from_numpy(rng.standard_normal((rows, SHAPE[3])).astype(np.float32))
    return x.cuda(), t.cuda()


def test_parameters_set_while_the_default_stream_is_busy():
    import torch
    from paper_1309_6726_gb300 import mlp
    x, t = _data()
    first = mlp.Mlp(*SHAPE, max_batch=48)  # (the kernels are loaded by now)
    theta = _theta(first.param_count)
    first.set_params(theta)
    want = first.forward(x).cpu()
    torch.cuda.synchronize()
    torch.cuda._sleep(BUSY)
    net = mlp.Mlp(*SHAPE, max_batch=48)
    net.set_params(theta)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(net.params(), theta)
    assert torch.equal(net.forward(x).cpu(), want)
    net.close()
    first.close()


def test_calls_on_another_stream_follow_the_queued_ones():
    import torch
    from paper_1309_6726_gb300 import mlp
    x, t = _data()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    got = []
    for switch in (False, True):
        net = mlp.Mlp(*SHAPE, max_batch=48)
        net.set_params(_theta(net.param_count))
        torch.cuda.synchronize()
        with torch.cuda.stream(a):
            net.forward(x)
            torch.cuda._sleep(BUSY if switch else 1)
            for _ in range(3):
                net.train_step(x, t, 1e-2)
        with torch.cuda.stream(b if switch else a):
            y = net.forward(x)
            g, loss = net.grad(x, t)
            y, g = y.cpu(), g.cpu()
        torch.cuda.synchronize()
        got.append((y, g, loss, net.params()))
        net.close()
    assert torch.equal(got[0][0], got[1][0])
    assert torch.equal(got[0][1], got[1][1])
    assert got[0][2] == got[1][2]
    np.testing.assert_array_equal(got[0][3], got[1][3])


def test_a_captured_pass_follows_passes_on_other_streams():
    # the capturing stream cannot wait for work outside the capture; the
    # caller orders the replay, as with any captured work
    import torch
    from paper_1309_6726_gb300 import mlp
    x, t = _data()
    net = mlp.Mlp(*SHAPE, max_batch=48)
    net.set_params(_theta(net.param_count))
    want = net.forward(x)
    out = torch.empty_like(want)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        net.forward(x, out)
    out.zero_()
    graph.replay()
    assert torch.equal(out, want)
    assert torch.equal(net.forward(x), want)
    net.close()
