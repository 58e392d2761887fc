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
