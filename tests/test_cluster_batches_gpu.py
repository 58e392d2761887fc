"""Steps kept on chip for batches of unequal lattices (blocks of a cluster
without a tile among them) and with each tile, against single launches of the
tile kernel, bit for bit; and batches whose clusters do not all fit the device,
which take single launches."""
import numpy as np
import pytest

from paper_1309_6726_gb300 import inputs as I
from paper_1309_6726_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _run(sizes, precision, calls, chip):
    geoms = [I.random_lattice(nx, ny, seed=nx * ny + k) for k, (nx, ny) in enumerate(sizes)]
    mps = [I.ModelParams(tau_a=0.9 + 0.1 * (k % 3), g_ads=I.G_ADS_30, k_r=5e-2,
                         m_threshold=0.4, inlet=k % 2) for k in range(len(sizes))]
    with lbm.Solver(geoms, mps, precision) as s:
        assert s.on_chip() == chip
        for k, (g, (nx, ny)) in enumerate(zip(geoms, sizes)):
            f, sol = I.random_populations(g, 7 + k, spread=0.05)
            s.set_populations(np.concatenate([f.reshape(18, ny, nx), sol]), k)
        out = []
        for n in calls:
            s.step(n)
            out.append([s.populations(k) for k in range(s.count)]
                       + [s.deposit(k) for k in range(s.count)] + s.solid_masks()
                       + [s.observables_array(allow_nan=True)[c]
                          for c in ("closure_step", "step", "nonfinite")])
    grown = sum(int(m.sum()) for m in out[-1][2 * len(sizes):3 * len(sizes)])
    assert grown > sum(int(g.solid.sum()) for g in geoms)
    return out


@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("sizes,tile,blocks", [
    ([(40, 10), (100, 14), (6, 6)], "32x4", 16),
    ([(66, 6), (34, 10), (30, 4)], "32x4", 8),
    ([(40, 10), (131, 14), (6, 6)], "64x4", 16),
    ([(256, 16)], "64x4", 16), ([(1024, 4), (66, 6)], "64x4", 16),
    ([(256, 32), (66, 6), (512, 16)], "64x8", 16), ([(66, 6), (200, 20)], "64x8", 16)],
    ids=lambda v: "+".join("%dx%d" % q for q in v) if isinstance(v, list) else str(v))
def test_batches_on_chip(sizes, tile, blocks, precision, monkeypatch):
    calls = (24, 31, 600)
    chip = _run(sizes, precision, calls, (tile, blocks))
    monkeypatch.setenv("LBM_TILE", "64x4")
    single = _run(sizes, precision, calls, None)
    for a, b in zip(chip, single):
        for u, v in zip(a, b):
            np.testing.assert_array_equal(u, v)


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
def test_more_clusters_than_the_device_holds(precision):
    sizes = [(256, 32 - 2 * (k % 3)) for k in range(20)]  # 20 x 16 blocks, one per SM
    one = _run(sizes[:1], precision, (26,), ("64x8", 16))
    many = _run(sizes, precision, (26,), None)
    np.testing.assert_array_equal(one[0][0], many[0][0])
