"""Device memory of a network's handle: the largest batch that fits is set by
what a row of the batch takes, and large batches go through the buffers that
the blocks share between their row tiles."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,row_bytes", [
    # every hidden activation, two gradients of a layer, the output and its
    # gradient, in FP32
    ((256, 1024, 8, 1024), 4 * (8 * 1024 + 2 * 1024 + 2 * 1024)),
    ((5, 256, 3, 65), 4 * (3 * 256 + 2 * 256 + 2 * 65))])
def test_memory_per_row_of_the_batch(shape, row_bytes):
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1309_6726_gb300 import mlp
    used = []
    for rows in (100_000, 400_000):
        mlp.Mlp(*shape, max_batch=rows).close()
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        net = mlp.Mlp(*shape, max_batch=rows)
        used.append(free - torch.cuda.mem_get_info()[0])
        net.close()
    per_row = (used[1] - used[0]) / 300_000
    print("%s: %.0f bytes per row (%d)" % (shape, per_row, row_bytes))
    assert per_row < row_bytes
    # and no more than that in all, but for the weights and what is kept per
    # block (weights: FP32, two moments, two BF16 copies, sixteen parts)
    weights = sum(r * c + r for r, c in mlp.layer_shapes(*shape))
    assert used[1] < 400_000 * row_bytes + weights * 4 * (3 + 1 + 16) + (64 << 20)


def test_rows_that_share_a_block_s_buffers():
    # 100,000 rows: every block carries several row tiles through the network
    import __graft_entry__
    __graft_entry__.build()
    import torch
    from oracle import mlp_ref as R
    from paper_1309_6726_gb300 import mlp
    shape, rows = (5, 32, 3, 7), 100_003
    rng = np.random.default_rng(3)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)  # noqa: E731
    shapes = mlp.layer_shapes(*shape)
    ws = [f32(rng.uniform(-1, 1, s) * np.sqrt(6.0 / (s[0] + s[1]))) for s in shapes]
    bs = [f32(rng.uniform(-0.1, 0.1, s[0])) for s in shapes]
    x = rng.uniform(-1, 1, (rows, shape[0])).astype(np.float32)
    t = rng.standard_normal((rows, shape[3])).astype(np.float32)
    net = mlp.Mlp(*shape, max_batch=rows)
    net.set_params(mlp.pack(ws, bs))
    g, loss = net.grad(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    net.close()
    loss_ref, g_ref = R.loss_grad(ws, bs, x, t, bf16=True)
    err = np.abs(g.cpu().numpy().astype(np.float64) - g_ref)
    scale = np.abs(g_ref).max()
    # FP32 sums over the batch leave the median at 1e-5 of the gradient's
    # scale; an operand that rounds to the other of two BF16 values moves its
    # row by 2^-8 of one of 100,003 terms
    assert loss == pytest.approx(loss_ref, rel=1e-4)
    assert np.median(err) < 1e-5 * scale
    assert err.max() < 2.0 ** -8 * scale
