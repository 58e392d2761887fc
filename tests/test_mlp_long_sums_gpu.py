"""Weight gradients of large batches on wide networks: the sum over the batch
is kept in at least eight parts whatever the network's size, so that the
rounding of a part's running sum stays short of the gradient's last digits.

With zero weights the outputs are 0, dz[b][n] = -2 t[b][n] / (rows outputs) in
FP32, then BF16, and the hidden activations are the same in every row, so that
the sum of exact products is known; with targets t = -(1 + i / 128) all terms
are positive.

Tolerance: a part of 65536 / 8 rows takes 512 steps of 16 rows on the tensor
cores; a step that truncates its FP32 sum loses up to 2^-23 of it, and the sum
grows evenly, so half of 512 times 2^-23 of the result at most, and 2^-24 for
each of the eight additions of the parts."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

OUT = 64
TOL = 256 * 2.0 ** -23 + 8 * 2.0 ** -24


def _bf16(a):
    import torch
    return torch.from_numpy(np.asarray(a, np.float32)).bfloat16().float().numpy()


@pytest.mark.parametrize("hidden,layers,rows", [
    (64, 1, 65536), (256, 3, 65536), (512, 2, 65536), (1024, 1, 65536),
    (1024, 2, 65536), (1024, 2, 65499), (1024, 8, 64 * 1017 + 1)])
def test_sums_over_a_large_batch(hidden, layers, rows):
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1309_6726_gb300 import mlp
    rng = np.random.default_rng(hidden + layers)
    t = -(1 + rng.integers(0, 128, (rows, OUT)) / 128.0)
    bias = rng.uniform(0.2, 1.5, hidden).astype(np.float32)
    h = np.tanh(bias.astype(np.float64))
    # units whose activation could round to either of two BF16 values are left out
    sure = _bf16(h * (1 - 1e-5)) == _bf16(h * (1 + 1e-5))
    assert sure.sum() > hidden // 2
    shapes = mlp.layer_shapes(3, hidden, layers, OUT)
    ws = [np.zeros(s) for s in shapes]
    bs = [np.zeros(s[0]) for s in shapes]
    bs[-2] = bias
    net = mlp.Mlp(3, hidden, layers, OUT, max_batch=rows)
    net.set_params(mlp.pack(ws, bs))
    x = torch.zeros(rows, 3, device="cuda")
    g, _ = net.grad(x, torch.from_numpy(t.astype(np.float32)).cuda())
    net.close()
    got = mlp.unpack(g.cpu().numpy(), 3, hidden, layers, OUT)[0][-1]
    dz = np.float32(-2.0) * t.astype(np.float32) * (np.float32(1) / np.float32(rows * OUT))
    want = np.outer(_bf16(dz).astype(np.float64).sum(0), _bf16(h).astype(np.float64))
    err = np.abs(got / want - 1.0)[:, sure].max()
    print("hidden %d layers %d rows %d: %.3g (tolerance %.3g)" % (hidden, layers, rows, err, TOL))
    assert err < TOL
