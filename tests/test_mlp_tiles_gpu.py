"""Edges of the network kernels against the FP64 reference with the same BF16
operand rounding: batches around the 16-, 32- and 64-row blocks, more row
tiles than blocks, one and many outputs, unit counts that are not multiples of
the 32-unit word, several 256-unit passes, one and eight hidden layers.

Tolerances: FP32 accumulation leaves the median output within 1e-6 of the
output scale and the median gradient within 1e-5 of the gradient scale; an
activation that FP32 and FP64 round to neighbouring BF16 values moves its row
by up to a BF16 unit (2^-8) of one operand, and the layers above pass it on."""
import numpy as np
import pytest

from oracle import mlp_ref as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,n_hidden,n_layers,n_out,batch", [
    (5, 256, 3, 65, 1), (5, 256, 3, 65, 17), (1, 16, 1, 1, 15),
    (33, 48, 2, 97, 2433), (5, 80, 1, 31, 4865), (256, 1024, 1, 300, 40),
    (3, 16, 8, 2, 40000), (7, 272, 2, 257, 129)])
def test_block_and_tile_edges(n_in, n_hidden, n_layers, n_out, batch):
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1309_6726_gb300 import mlp
    rng = np.random.default_rng(n_hidden + batch)
    shapes = mlp.layer_shapes(n_in, n_hidden, n_layers, n_out)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)  # noqa: E731
    ws = [f32(rng.uniform(-1, 1, s) * np.sqrt(6.0 / (s[0] + s[1]))) for s in shapes]
    bs = [f32(rng.uniform(-0.1, 0.1, s[0])) for s in shapes]
    x = rng.uniform(-1, 1, (batch, n_in)).astype(np.float32)
    t = rng.standard_normal((batch, n_out)).astype(np.float32)
    t[1::7, -1] = np.nan
    net = mlp.Mlp(n_in, n_hidden, n_layers, n_out, max_batch=batch)
    net.set_params(mlp.pack(ws, bs))
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    y = net.forward(xd).cpu().numpy().astype(np.float64)
    _, ref = R.forward(ws, bs, x, bf16=True)
    err, scale = np.abs(y - ref), np.abs(ref).max()
    assert np.median(err) < 1e-6 * scale
    assert np.median(err[-16:]) < 1e-5 * scale  # the last, ragged block
    assert err.max() < 2.0 ** -8 * scale * n_layers
    g, loss = net.grad(xd, td)
    g = g.cpu().numpy().astype(np.float64)
    loss_ref, g_ref = R.loss_grad(ws, bs, x, t, bf16=True)
    assert loss == pytest.approx(loss_ref, rel=1e-4)
    gs = np.abs(g_ref).max()
    gerr = np.abs(g - g_ref)
    assert np.median(gerr) < 1e-5 * gs
    assert gerr.max() < 2.0 ** -8 * gs * n_layers
    # the same from a training step: Adam's first update has the gradient's sign
    net.train_step(xd, td, 1e-3)
    moved = net.params().astype(np.float64) - mlp.pack(ws, bs)
    big = np.abs(g_ref) > 1e-3 * gs
    assert np.array_equal(np.sign(moved[big]), -np.sign(g_ref[big]))
    net.close()
