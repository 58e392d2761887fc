"""The arrays that read-backs return: any shape and type, and what making one
costs beside the plain array (no GPU needed)."""
import mmap
import time

import numpy as np
import pytest

from paper_1309_6726_gb300 import lbm


@pytest.mark.parametrize("shape,dtype", [
    ((1, 1), np.uint8), ((3, 13, 131), np.float32), ((16, 64), np.float64),
    ((mmap.PAGESIZE,), np.uint8), ((mmap.PAGESIZE + 1,), np.uint8),
    ((22, 257, 129), np.float32), ((1023, 1025), np.float64),
    ((32 << 20,), np.uint8), (((32 << 20) + 1,), np.uint8)])
def test_shape_type_and_ownership(shape, dtype):
    a = lbm._fresh(shape, dtype)
    assert a.shape == shape and a.dtype == dtype
    assert a.flags.c_contiguous and a.flags.writeable and a.flags.owndata
    a[...] = 1
    assert (a == 1).all()


def _fastest(f, n):
    best = 1e9
    for _ in range(n):
        t = time.perf_counter()
        f()
        best = min(best, time.perf_counter() - t)
    return best


@pytest.mark.parametrize("shape,factor,n", [((3, 16, 64), 3.5, 2000), ((22, 1024, 1024), 20, 10)])
def test_no_dearer_than_a_cleared_array(shape, factor, n):
    # a few hundred nanoseconds for small ones; large ones are not touched
    # (clearing 92 MB takes thousands of times the mapping of it)
    fresh = _fastest(lambda: lbm._fresh(shape, np.float32), n)
    plain = _fastest(lambda: np.zeros(shape, np.float32), n)
    print("%s: %.2f us, plain %.2f us" % (shape, fresh * 1e6, plain * 1e6))
    assert fresh < factor * plain
