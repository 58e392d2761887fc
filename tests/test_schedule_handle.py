"""Host logic of the schedule that a handle uses (``lbm_plan_schedule``):
every tile exactly once whatever the batch, one run of consecutive tiles per
block up to 8 tiles per block, strips from there on, evened out for 16 to 32
tiles per block where that shortens the longest list by a sixteenth.  No GPU
needed."""
import heapq
import math
import random

import numpy as np
import pytest

from paper_1309_6726_gb300 import lbm


def _tiles(sizes, tx, ty):
    return [(l, x, y) for l, (nx, ny) in enumerate(sizes)
            for x in range(0, nx, tx) for y in range(0, ny, ty)]


def _lists(sched):
    """Tiles of each block, in order; nothing follows an end marker."""
    out = []
    for b in range(sched.shape[1]):
        col = sched[:, b]
        n = int((col[:, 0] >= 0).sum())
        assert (col[n:] == (-1, 0, 0)).all()
        out.append([tuple(int(v) for v in t) for t in col[:n]])
    return out


def _evened(sizes, tx, ty, grid):
    """The longest list's length and the lists, columns cut into equal pieces
    of the length 3 to 8 that leaves the longest list the shortest."""
    best = None
    for seg in range(8, 2, -1):
        strips = []
        for l, (nx, ny) in enumerate(sizes):
            rows = -(-ny // ty)
            n = -(-rows // seg)
            for x in range(0, nx, tx):
                for k in range(n):
                    r0, r1 = k * rows // n, (k + 1) * rows // n
                    strips.append([(l, x, r * ty) for r in range(r0, r1)])
        heap = [(0, b, []) for b in range(grid)]
        for s in sorted(strips, key=lambda s: -len(s)):
            load, b, tiles = heapq.heappop(heap)
            heapq.heappush(heap, (load + len(s), b, tiles + s))
        top = max(h[0] for h in heap)
        if best is None or top < best[0]:
            best = (top, [h[2] for h in sorted(heap, key=lambda h: h[1])])
    return best


def _check(sizes, tx, ty, grid):
    lists = _lists(lbm.plan_schedule(sizes, tx, ty, grid))
    tiles = _tiles(sizes, tx, ty)
    assert sorted(t for b in lists for t in b) == tiles
    total, loads = len(tiles), [len(b) for b in lists]
    if total <= 8 * grid:
        assert [t for b in lists for t in b] == tiles  # runs, in order
        assert max(loads) - min(loads) <= 1
        return "runs"
    strips = _lists(lbm.plan_tiles(sizes, tx, ty, grid))
    plain = max(len(b) for b in strips)
    if 16 * grid < total <= 32 * grid and max(-(-ny // ty) for _, ny in sizes) <= 64:
        top, want = _evened(sizes, tx, ty, grid)
        if 16 * top <= 15 * plain:
            assert lists == want
            return "evened"
    assert lists == strips
    return "strips"


@pytest.mark.parametrize("sizes,tx,ty,grid,kind", [
    ([(4096, 128)], 64, 4, 304, "runs"), ([(4096, 128)] * 3, 64, 4, 304, "evened"),
    ([(4096, 128)] * 4, 64, 4, 304, "strips"), ([(4600, 160)] * 3, 64, 4, 304, "evened"),
    ([(1024, 1024)], 64, 8, 152, "strips"), ([(1024, 1024)], 32, 8, 304, "strips"),
    ([(2048, 2048)], 64, 8, 152, "strips"), ([(256, 32)], 32, 4, 304, "runs"),
    ([(1, 3)], 32, 4, 304, "runs"), ([(64, 5), (300, 255), (64, 1)], 64, 4, 20, "evened"),
    ([(300, 256)], 64, 4, 18, "strips"), ([(300, 260)], 64, 4, 18, "strips")])
def test_kinds_of_schedule(sizes, tx, ty, grid, kind):
    assert _check(sizes, tx, ty, grid) == kind


@pytest.mark.parametrize("per", [1, 8, 16, 32])
@pytest.mark.parametrize("grid", [1, 7, 152])
@pytest.mark.parametrize("rows", [1, 5, 32, 64, 65])
def test_totals_around_the_limits(per, grid, rows):
    # per - 1, per, per + 1 tiles more or less than `per` per block
    for total in sorted({per * grid - 1, per * grid, per * grid + 1}):
        if total < 1:
            continue
        cols, rest = divmod(total, rows)
        sizes = ([(32 * cols - 5, 4 * rows - 1)] if cols else []) + \
            ([(7, 4 * rest - 2)] if rest else [])
        assert len(_tiles(sizes, 32, 4)) == total
        _check(sizes, 32, 4, grid)


def test_random_batches():
    rng = random.Random(5)
    kinds = set()
    for _ in range(150):
        tx, ty = rng.choice([(32, 4), (64, 4), (64, 8), (32, 8)])
        grid = rng.choice([1, 2, 13, 40, 152])
        sizes = [(rng.randint(1, 900), int(math.exp(rng.uniform(0, 5.9))))
                 for _ in range(rng.randint(1, 12))]
        kinds.add(_check(sizes, tx, ty, grid))
    assert kinds == {"runs", "strips", "evened"}


@pytest.mark.parametrize("count", [4, 5, 8, 10])
def test_evened_strips_cost_no_more_than_a_few_plain_ones(count):
    # a handle's schedule is part of every create: choosing among six lengths
    # must not deal the batch six times (measured 6 to 8 times plan_tiles then)
    import time
    from paper_1309_6726_gb300 import inputs as I
    sizes = [(m.length + 96, m.width + 2) for m in I.sweep_members(512)[:count]]

    def fastest(f):
        best = math.inf
        for _ in range(40):
            t = time.perf_counter()
            f(sizes, 64, 4, 304)
            best = min(best, time.perf_counter() - t)
        return best
    ratio = fastest(lbm.plan_schedule) / fastest(lbm.plan_tiles)
    print("%d lattices: %.2f" % (count, ratio))
    assert ratio < 3


def test_rejects_what_plan_tiles_rejects():
    for args in (([], 64, 8, 152), ([(64, 8)], 0, 8, 152), ([(64, 8)], 64, 8, 0),
                 ([(0, 8)], 64, 8, 4)):
        with pytest.raises(lbm.LbmError):
            lbm.plan_schedule(*args)
