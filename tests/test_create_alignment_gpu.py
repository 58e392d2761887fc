"""Input arrays that start anywhere: views into byte buffers, behind odd
headers, as ``numpy.frombuffer`` and memory maps give them.  They hold the
same values as the aligned arrays, so the state after creation and the
trajectory are the same bit for bit."""
import dataclasses

import numpy as np
import pytest

from paper_1309_6726_gb300 import inputs as I
from paper_1309_6726_gb300 import lbm

pytestmark = pytest.mark.gpu


def _shifted(a, dtype, offset, pinned):
    """The values of ``a`` in an array that starts ``offset`` bytes behind a
    64-byte boundary."""
    import torch
    a = np.ascontiguousarray(a, dtype)
    n = a.nbytes + 128
    buf = (torch.empty(n, dtype=torch.uint8, pin_memory=True).numpy() if pinned
           else np.empty(n, np.uint8))
    at = -buf.ctypes.data % 64 + offset
    out = buf[at:at + a.nbytes].view(dtype).reshape(a.shape)
    out[...] = a
    assert out.ctypes.data % 64 == offset
    return out


@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("offsets", [(1, 1, 1, 1), (3, 2, 6, 13), (8, 4, 0, 5)])
def test_inputs_at_any_address(offsets, pinned):
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    geoms = [I.random_lattice(131, 13, seed=3), I.random_lattice(37, 21, seed=4)]
    mps = [I.ModelParams(g_ads=0.3, k_r=1e-2, m_threshold=0.05, inlet=1)] * 2
    kinds = (("rho_a", np.float32), ("rho_b", np.float32), ("conc", np.float32),
             ("solid", np.uint8))
    moved = [dataclasses.replace(g, **{
        k: _shifted(getattr(g, k), t, o, pinned)
        for (k, t), o in zip(kinds, offsets)}) for g in geoms]
    got = []
    for gs in (geoms, moved):
        with lbm.Solver(gs, mps) as s:
            out = [s.populations(k) for k in range(2)]
            s.step(7)
            got.append(out + [s.populations(k) for k in range(2)] + s.solid_masks())
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
