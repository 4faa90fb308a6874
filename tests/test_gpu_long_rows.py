"""Rows whose columns span more than a warp's bitmap (131,072 points apart) take the block row sort:
its bitmap, its radix sort with both buffers in shared memory and with passes that alternate between
the row and the buffer, and its sorting network in place, each against the rows known from the
input.  The kernel is left out of a shape's builds while no row is left to it and comes back."""
import numpy as np
import pytest

from paper_1409_8112_gb300 import rtg

pytestmark = pytest.mark.gpu

D, R = 3, 0.01


def _points(n, spot, spread, seed=5):
    """n points of which `spot` lie within r of one another (spread over all indices, the first and
    the last among them, or the first ones) and no others do; the identity grid, shifted so that
    the spot is inside a cell."""
    rng = np.random.default_rng(seed)
    pts = rng.uniform(10.0, 1000.0, (n, D)).astype(np.float32)
    idx = np.unique(np.linspace(0, n - 1, spot).astype(np.int64)) if spread else np.arange(spot)
    pts[idx] = rng.uniform(0.0, 1e-3, (spot, D))
    T = np.concatenate([np.eye(D).reshape(-1), np.full(D, R / 2)])[None]
    return pts, T, idx


def _check(ctx, n, spot, spread, symmetric=False):
    pts, T, idx = _points(n, spot, spread)
    res = ctx.all_pairs(pts, R, T, R, symmetric=symmetric)
    rp, col = res.download()
    attempts = res.stats["attempts"]
    res.release()
    want = np.zeros(n + 1, dtype=np.int64)
    want[idx + 1] = spot - 1 if symmetric else spot - 1 - np.arange(spot)
    assert np.array_equal(rp, np.cumsum(want))
    if symmetric:
        rows = [np.delete(idx, k) for k in range(spot)]
    else:
        rows = [idx[k + 1:] for k in range(spot)]
    assert np.array_equal(col, np.concatenate(rows))
    return attempts


@pytest.mark.parametrize("n,spot,symmetric", [
    (140000, 300, False), (140000, 300, True),    # radix sort, both buffers in shared memory
    (140000, 3000, False), (140000, 2600, True),  # one bitmap per block
    (700000, 9000, False),                        # radix sort, the row is one of the buffers
    (700000, 16700, False),                       # the network, in place
])
def test_rows_that_span_more_than_a_bitmap(n, spot, symmetric):
    with rtg.Context(0) as ctx:
        for _ in range(2):
            _check(ctx, n, spot, True, symmetric)


def test_block_row_sort_comes_back():
    # long rows that fit the bitmaps let the shape leave the block sort out; rows that do not are
    # flagged and the build runs again with it
    n, spot = 140000, 300
    with rtg.Context(0) as ctx:
        _check(ctx, n, spot, False)
        assert _check(ctx, n, spot, False) == 1
        assert _check(ctx, n, spot, True) == 2
        assert _check(ctx, n, spot, True) == 1
        for _ in range(17):
            assert _check(ctx, n, spot, False) == 1
        assert _check(ctx, n, spot, True) == 2


def test_bitmaps_come_back():
    # and so for the bitmaps and the warp sorts, with no long row at all before
    n = 140000
    with rtg.Context(0) as ctx:
        for spot, spread, attempts in ((20, True, None), (20, True, 1), (40, True, 2), (40, True, 1),
                                       (300, False, 2), (300, False, 1), (300, True, 1)):
            a = _check(ctx, n, spot, spread)
            assert attempts is None or a == attempts, (spot, spread)
