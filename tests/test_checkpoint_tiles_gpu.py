"""A checkpoint holds the state, not how a handle launches: handles of the same
sizes and parameters load one another's, whatever tiles they use."""
import numpy as np
import pytest

from paper_1309_6726_gb300 import inputs as I

pytestmark = pytest.mark.gpu

MP = I.ModelParams(g_ads=0.3, k_r=1e-2, m_threshold=0.05, inlet=1)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("tile", ["32x8", "64x8", "128x4"])
def test_load_under_another_tile(tile, precision, tmp_path, monkeypatch):
    from paper_1309_6726_gb300 import lbm
    geoms = [I.random_lattice(300, 40, seed=1), I.random_lattice(131, 33, seed=2)]
    path = str(tmp_path / "state")
    with lbm.Solver(geoms, [MP] * 2, precision) as a:
        a.step(30)
        a.save(path)
        a.step(31)
        monkeypatch.setenv("LBM_TILE", tile)
        with lbm.Solver(geoms, [MP] * 2, precision) as b:
            assert b.tuning()["tile"] == tile != a.tuning()["tile"]
            b.load(path)
            b.step(31)
            for k in range(2):
                np.testing.assert_array_equal(a.populations(k), b.populations(k))
                np.testing.assert_array_equal(a.deposit(k), b.deposit(k))
                np.testing.assert_array_equal(a.solid_mask(k), b.solid_mask(k))


def test_load_with_another_initial_solid(tmp_path):
    # (FP32, 700k nodes: the default tile depends on the solid share)
    from paper_1309_6726_gb300 import lbm
    full = I.random_lattice(1001, 701, seed=5, solid_fraction=0.4)
    thin = I.random_lattice(1001, 701, seed=6, solid_fraction=0.05)
    path = str(tmp_path / "state")
    with lbm.Solver(full, MP) as a, lbm.Solver(thin, MP) as b:
        assert a.tuning()["tile"] != b.tuning()["tile"]
        a.step(5)
        a.save(path)
        b.load(path)
        a.step(6)
        b.step(6)
        np.testing.assert_array_equal(a.populations(), b.populations())
        np.testing.assert_array_equal(a.solid_mask(), b.solid_mask())


def test_load_refuses_other_parameters(tmp_path):
    from paper_1309_6726_gb300 import lbm
    import dataclasses
    g = I.random_lattice(300, 40, seed=1)
    path = str(tmp_path / "state")
    with lbm.Solver(g, MP) as a:
        a.save(path)
    for other in (dataclasses.replace(MP, g_ads=0.31), dataclasses.replace(MP, inlet=0)):
        with lbm.Solver(g, other) as b, pytest.raises(lbm.LbmError):
            b.load(path)
    with lbm.Solver(I.random_lattice(296, 40, seed=1), MP) as b, \
            pytest.raises(lbm.LbmError):
        b.load(path)


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_steps_queued_right_after_a_load(precision, tmp_path):
    # nothing but the stream's order stands between the upload and the steps
    # (the step counter is the last thing uploaded), with other work around
    import torch
    from paper_1309_6726_gb300 import lbm
    g = I.random_lattice(300, 40, seed=1)
    path = str(tmp_path / "state")
    x = torch.ones(1 << 24, device="cuda")
    with lbm.Solver(g, MP, precision) as a, lbm.Solver(g, MP, precision) as b:
        a.step(17)
        a.save(path)
        a.step(9)
        want, mask = a.populations(), a.solid_mask()
        for _ in range(10):
            b.step(3)
            x.add_(1.0)
            b.load(path)
            b.step(9)
            assert b.observables_array(allow_nan=True)["step"][0] == 26
            np.testing.assert_array_equal(b.populations(), want)
            np.testing.assert_array_equal(b.solid_mask(), mask)
