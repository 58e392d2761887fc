"""Steps kept on chip (one thread block cluster per lattice) against single
launches of the tile kernel, bit for bit: lattices around the tile edges, last
tiles of two nodes, one tile with itself as neighbour, random solids, growth in
the middle of a launch, calls longer than one launch, several lattices of
unequal size, all storages.  The general path is the same handle with its tile
named, which keeps it off the cluster."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [[(4, 4)], [(32, 4)], [(34, 6)], [(130, 10)], [(66, 13)], [(131, 13)],
         [(256, 32)], [(254, 31)], [(512, 16)], [(1024, 8)],
         [(40, 9), (131, 13), (6, 5)]]


@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("sizes", SIZES, ids=lambda s: "+".join("%dx%d" % q for q in s))
def test_on_chip_steps_equal_single_launches(sizes, precision, monkeypatch):
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1309_6726_gb300 import inputs as I, lbm
    geoms, params, pops = [], [], []
    for k, (nx, ny) in enumerate(sizes):
        g = I.random_lattice(nx, ny, seed=nx * ny + k)
        geoms.append(g)
        params.append(I.ModelParams(tau_a=0.9 + 0.1 * k, g_ads=I.G_ADS_30, k_r=5e-2,
                                    m_threshold=0.4, inlet=1))
        f, s = I.random_populations(g, 7 + k, spread=0.05)
        pops.append(np.concatenate([f.reshape(18, ny, nx), s]))
    got = []
    for tile in (None, "64x4"):
        if tile:
            monkeypatch.setenv("LBM_TILE", tile)
        with lbm.Solver(geoms, params, precision) as s:
            for k, f in enumerate(pops):
                s.set_populations(f, k)
            out = []
            for n in (4, 5, 1, 31, 600):  # 600: more than one launch
                s.step(n)
                o = s.observables_array(allow_nan=True)
                out.append([s.populations(k) for k in range(s.count)]
                           + [s.deposit(k) for k in range(s.count)] + s.solid_masks()
                           + [o["closure_step"], o["step"], o["nonfinite"]])
                led = np.stack([o["ledger_" + c] for c in "abcm"])
                out[-1].append(led)
        got.append(out)
    grown = sum(int(m.sum()) for m in got[0][-1][2 * len(sizes):3 * len(sizes)])
    assert grown > sum(int(g.solid.sum()) for g in geoms)
    for a, b in zip(*got):
        for u, v in zip(a[:-1], b[:-1]):
            np.testing.assert_array_equal(u, v)
        # the ledgers are FP64 sums in no fixed order: 64 additions' rounding
        np.testing.assert_allclose(a[-1], b[-1], rtol=64 * 2.0 ** -52, atol=1e-300,
                                   equal_nan=True)
