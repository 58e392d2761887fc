"""Steps with each kind of schedule (runs, strips, evened strips) against the
direct-load kernel, bit for bit: a tile that is left out, done twice or takes
its top row from the wrong neighbour shows."""
import numpy as np
import pytest

from paper_1309_6726_gb300 import inputs as I
from paper_1309_6726_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("sizes,kind", [
    ([(3001, 97)], "runs"), ([(3001, 97), (700, 31)], "runs"),
    ([(2999, 99)] * 3, "strips"), ([(4096, 128)] * 3, "evened"),
    ([(4096, 128)] * 2 + [(4050, 127)], "evened")])
def test_schedules_give_the_same_steps(sizes, kind, precision, monkeypatch):
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    grid = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    tiles = sum(-(-nx // 64) * -(-ny // 4) for nx, ny in sizes)
    even = not np.array_equal(lbm.plan_schedule(sizes, 64, 4, grid),
                              lbm.plan_tiles(sizes, 64, 4, grid))
    assert kind == ("runs" if tiles <= 8 * grid else "evened" if even else "strips")
    geoms = [I.random_lattice(nx, ny, seed=k, solid_fraction=0.01)
             for k, (nx, ny) in enumerate(sizes)]
    mps = [I.ModelParams(g_ads=0.3, k_r=1e-2, m_threshold=0.05, inlet=1)] * len(sizes)
    got = []
    for kernel in ("", "direct"):
        if kernel:
            monkeypatch.setenv("LBM_KERNEL", kernel)
        with lbm.Solver(geoms, mps, precision) as s:
            assert s.tuning()["tile"] == "64x4"
            s.step(9)
            got.append([s.populations(k) for k in range(s.count)]
                       + [s.deposit(k) for k in range(s.count)] + s.solid_masks())
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
