"""The tile of FP32 batches by the solid nodes inside their lattices, whatever
memory the arrays are in, and its results against the direct-load kernel, bit
for bit."""
import ctypes as C

import numpy as np
import pytest

from paper_1309_6726_gb300 import inputs as I
from paper_1309_6726_gb300 import lbm

pytestmark = pytest.mark.gpu

MP = I.ModelParams(g_ads=0.3, k_r=1e-2, m_threshold=0.05, inlet=1)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _batch(sizes, share):
    return [I.random_lattice(nx, ny, seed=k, solid_fraction=share)
            for k, (nx, ny) in enumerate(sizes)]


@pytest.mark.parametrize("sizes,share,precision,tile", [
    ([(790, 800)] * 2, 0.05, "fp32", "64x8"), ([(790, 800)] * 2, 0.005, "fp32", "64x4"),
    ([(790, 800)] * 2, 0.05, "fp16", "64x4"), ([(513, 509)] * 4, 0.3, "fp32", "64x4"),
    ([(131, 13), (1500, 200), (999, 3), (1201, 801)], 0.1, "fp32", "64x8"),
    ([(790, 800)], 0.3, "fp32", "64x4")])
def test_tile_of_a_batch_and_its_results(sizes, share, precision, tile, monkeypatch):
    geoms = _batch(sizes, share)
    got = []
    for kernel in ("", "direct"):
        if kernel:
            monkeypatch.setenv("LBM_KERNEL", kernel)
        with lbm.Solver(geoms, [MP] * len(geoms), precision) as s:
            if not kernel:
                assert s.tuning()["tile"] == tile
            s.step(5)
            got.append([s.populations(k) for k in range(s.count)]
                       + [s.deposit(k) for k in range(s.count)] + s.solid_masks())
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)


def test_walls_are_not_inside():
    # capillaries: solid rows along both edges only
    geoms = [I.capillary(4096, 128, 256, 128)] * 3
    with lbm.Solver(geoms, [MP] * 3) as s:
        assert s.tuning()["tile"] == "64x4"


@pytest.mark.parametrize("count,nx,ny", [(2, 790, 800), (60, 301, 83)])
@pytest.mark.parametrize("share,tile", [(0.05, "64x8"), (0.0, "64x4")])
def test_device_arrays_give_the_same_tile(count, nx, ny, share, tile):
    import torch
    geoms = _batch([(nx, ny)] * count, share)
    with lbm.Solver(geoms, [MP] * count) as s:
        assert s.tuning()["tile"] == tile
    lib = lbm.load_library()
    G, P = (lbm.Geometry * count)(), (lbm.Params * count)()
    keep = []
    for k, g in enumerate(geoms):
        a = [torch.from_numpy(np.ascontiguousarray(getattr(g, f))).cuda()
             for f in ("solid", "rho_a", "rho_b", "conc")]
        keep += a
        G[k] = lbm.Geometry(nx, ny, *(v.data_ptr() for v in a), int(g.cap_x0),
                            int(g.cap_x1))
        P[k] = lbm._params(MP, lbm.LBM_FP32)
    torch.cuda.synchronize()
    h = C.c_void_p()
    assert lib.lbm_create_batch(G, P, count, C.byref(h)) == lbm.LBM_OK
    t = lbm.Tuning()
    assert lib.lbm_get_tuning(h, C.byref(t)) == lbm.LBM_OK
    assert t.as_dict()["tile"] == tile
    lib.lbm_destroy(h)
