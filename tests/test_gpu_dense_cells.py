"""Cells of more than 32 points (32 x 32 member tiles): block edges, short last blocks, several
jobs per cell, the largest tiled cell and the first beyond it, every key-row layout and output
form, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1409_8112_gb300 import gen, rtg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = rtg.Context(0)
    yield c
    c.close()


def _same(ctx, pts, r, T, c, **kw):
    ref = oracle.rtg(pts, r, T, c)
    for _ in range(2):  # first build, then the shape's second
        res = ctx.all_pairs(pts, r, T, c, **kw)
        rp, col = res.download()
        st = res.stats
        res.release()
        if kw.get("symmetric"):
            i = np.repeat(np.arange(len(rp) - 1), np.diff(rp))
            up = i < col
            assert 2 * up.sum() == len(col) == 2 * ref.csr.nnz
            rp, col = np.concatenate([[0], np.cumsum(np.bincount(i[up], minlength=len(rp) - 1))]), col[up]
        assert np.array_equal(rp, ref.csr.row_ptr) and np.array_equal(col, ref.csr.col)
        assert st["max_cell"] == max(s["max_cell"] for s in ref.stats)
        if not kw.get("bitset"):
            assert st["candidates"] == [s["candidates"] for s in ref.stats]
    return st


@pytest.mark.parametrize("n,d,dtype", [(33, 2, np.float64), (64, 6, np.float32), (65, 7, np.float32),
                                       (96, 4, np.float64), (97, 12, np.float32),
                                       (513, 13, np.float64), (4097, 3, np.float32),
                                       (8192, 2, np.float32), (8193, 2, np.float64)])
def test_one_cell(ctx, n, d, dtype):
    # cells far larger than the points: (nearly always) one cell of n points per grid
    pts = gen.points_uniform(n + d, n, d, dtype)
    r = gen.radius_for_degree(n, d, 9.0)
    st = _same(ctx, pts, r, gen.transforms(n, d, 2, 40.0), 40.0)
    assert st["large_cells"] >= 1


@pytest.mark.parametrize("form", ["plain", "symmetric", "two_pass", "bitset"])
@pytest.mark.parametrize("m,cf", [(1, 1.0), (5, 1.0), (8, 1.3), (20, 1.0), (37, 1.5)])
def test_forms_and_key_rows(ctx, m, cf, form):
    # key rows in place (m = 37), by the key (m = 1, 5) and in 16-byte blocks (m = 8, 20)
    pts = gen.points_mixture(90 + m, 1500, 3, k=4, sigma=0.05, dtype=np.float32)
    r = 0.11
    kw = {} if form == "plain" else {form: True}
    st = _same(ctx, pts, r, gen.transforms(90 + m, 3, m, cf * r), cf * r, **kw)
    assert st["large_cells"] > 0


def test_wide_keys(ctx):
    # 64-bit composite keys next to dense cells
    pts = np.vstack([gen.points_mixture(5, 1200, 9, k=3, sigma=0.02, dtype=np.float64),
                     gen.points_uniform(6, 300, 9) * 6.0])
    r = 0.3
    st = _same(ctx, pts, r, gen.transforms(5, 9, 6, r), r)
    assert st["large_cells"] > 0 and st["key_bits"] > 32
