"""The tile a handle picks by size, storage and solid share, and its results
against the direct-load kernel, bit for bit (no arithmetic differs)."""
import numpy as np
import pytest

from paper_1309_6726_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _solids(nx, ny, share):
    g = I.random_lattice(nx, ny, seed=nx + ny, solid_fraction=share)
    return g


@pytest.mark.parametrize("nx,ny,share,precision,tile", [
    (256, 32, 0.05, "fp32", "32x4"), (256, 32, 0.05, "fp16", "32x4"),
    (999, 61, 0.05, "fp32", "64x4"), (999, 61, 0.05, "bf16", "64x4"),
    (1001, 701, 0.05, "fp32", "64x8"), (1001, 701, 0.4, "fp32", "32x8"),
    (1001, 701, 0.4, "fp16", "64x4"), (2047, 740, 0.4, "fp32", "64x8")])
def test_default_tile_and_its_results(nx, ny, share, precision, tile, monkeypatch):
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1309_6726_gb300 import lbm
    g = _solids(nx, ny, share)
    p = I.ModelParams(g_ads=0.3, k_r=1e-2, m_threshold=0.05, inlet=1)
    got = []
    for kernel in ("", "direct"):
        if kernel:
            monkeypatch.setenv("LBM_KERNEL", kernel)
        with lbm.Solver(g, p, precision) as s:
            if not kernel:
                assert s.tuning()["tile"] == tile
            s.step(7)
            got.append((s.populations(), s.deposit(), s.solid_mask()))
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
