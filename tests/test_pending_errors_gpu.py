"""A refused allocation is that call's error alone: the handles that exist and
those created after it work as before."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_calls_after_a_refused_allocation():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1309_6726_gb300 import inputs as I, lbm, mlp
    x, t = torch.randn(32, 5, device="cuda"), torch.randn(32, 9, device="cuda")
    net = mlp.Mlp(5, 64, 2, 9, max_batch=32)
    net.set_params(np.full(net.param_count, 0.01, np.float32))
    want, loss = net.grad(x, t)
    for _ in range(2):
        with pytest.raises(lbm.LbmError):
            mlp.Mlp(256, 1024, 8, 1024, max_batch=1 << 24)  # 600 GB at least
        g, again = net.grad(x, t)
        assert torch.equal(g, want) and again == loss
    geom, mp, _ = I.config_small()
    with pytest.raises(lbm.LbmError):
        mlp.Mlp(256, 1024, 8, 1024, max_batch=1 << 24)
    with lbm.Solver(geom, mp) as s:
        s.step(3)
        assert s.observables()[0]["step"] == 3
    net.close()
