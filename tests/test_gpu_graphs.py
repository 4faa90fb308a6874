"""Replayed launch sequences (CUDA graphs): later builds of a shape replay the sequence
captured on an earlier one.  New points and transforms of the same shape, host or device
inputs, symmetric output and timing must all give the oracle's CSR bit for bit, and the
same results as direct launches."""
import os

import numpy as np
import pytest

import oracle
from paper_1409_8112_gb300 import gen, rtg

pytestmark = pytest.mark.gpu


def _context(graphs: bool):
    old = os.environ.get("RTG_GRAPHS")
    os.environ["RTG_GRAPHS"] = "1" if graphs else "0"
    try:
        return rtg.Context(0)
    finally:
        if old is None:
            os.environ.pop("RTG_GRAPHS", None)
        else:
            os.environ["RTG_GRAPHS"] = old


def _case(seed, n=9001, d=5, m=6, dtype=np.float64):
    r = gen.radius_for_degree(n, d)
    pts = gen.points_uniform(seed, n, d, dtype)
    T = gen.transforms(seed, d, m, r)
    return pts, r, T


@pytest.mark.parametrize("graphs", [True, False])
def test_repeated_shape_new_data(graphs):
    import torch
    ctx = _context(graphs)
    try:
        for k, seed in enumerate([40, 41, 42, 43, 44]):
            pts, r, T = _case(seed)
            arg = torch.from_numpy(pts).cuda() if k % 2 else pts
            res = ctx.all_pairs(arg, r, T, r, timing=(k == 3))
            rp, col = res.download()
            st = res.stats
            res.release()
            ref = oracle.rtg(pts, r, T, r)
            assert np.array_equal(rp, ref.csr.row_ptr) and np.array_equal(col, ref.csr.col)
            assert st["candidates"] == [s["candidates"] for s in ref.stats]
            assert st["near_wall"] == sum(s["near_wall"] for s in ref.stats)
            assert st["attempts"] == 1
            if k == 3:
                assert st["phase_us"]["total"] > 0 and st["phase_us"]["sort"] > 0
    finally:
        ctx.close()


def test_symmetric_and_fp32_shapes_interleaved():
    ctx = _context(True)
    try:
        for k in range(4):
            pts, r, T = _case(50 + k, n=7000, d=4, m=5, dtype=np.float32 if k % 2 else np.float64)
            res = ctx.all_pairs(pts, r, T, r, symmetric=True)
            rp, col = res.download()
            res.release()
            ref = oracle.rtg(pts, r, T, r)
            p = ref.csr.pairs()
            both = np.concatenate([p, p[:, ::-1]])
            both = both[np.lexsort((both[:, 1], both[:, 0]))]
            want_rp = np.zeros(len(pts) + 1, dtype=np.int64)
            np.add.at(want_rp, both[:, 0] + 1, 1)
            assert np.array_equal(rp, np.cumsum(want_rp))
            assert np.array_equal(col, both[:, 1].astype(np.int32))
    finally:
        ctx.close()


def test_pair_buffer_growth_falls_back_and_recaptures():
    # a shape whose second input has far more pairs: the guessed pair buffer overflows, the
    # build re-runs directly, and the next replay uses the grown buffer
    ctx = _context(True)
    try:
        n, d, m = 6000, 3, 4
        r = 0.05
        T = gen.transforms(60, d, m, r)
        sparse = gen.points_uniform(60, n, d)
        dense = gen.points_mixture(61, n, d, k=2, sigma=0.02, dtype=np.float64)
        for pts in (sparse, sparse, dense, dense, sparse):
            res = ctx.all_pairs(pts, r, T, r)
            rp, col = res.download()
            res.release()
            ref = oracle.rtg(pts, r, T, r)
            assert np.array_equal(rp, ref.csr.row_ptr) and np.array_equal(col, ref.csr.col)
    finally:
        ctx.close()


def test_overflow_after_a_replay_with_an_even_pass_count():
    # a replayed build whose pairs overflow its buffer writes the columns by a second
    # enumeration, which has to read the buffer the sort ended in (the second one for an even
    # number of passes)
    d, n, m, r = 3, 6000, 6, 0.06
    corners = np.array([[0.0] * d, [1.0] * d])
    loose = np.vstack([gen.points_mixture(21, n - 2, d, k=8, sigma=0.08, dtype=np.float64), corners])
    tight = np.vstack([gen.points_mixture(21, n - 2, d, k=8, sigma=0.05, dtype=np.float64), corners])
    T = gen.transforms(21, d, m, r)
    ctx = rtg.Context(0)
    for k in range(5):
        pts = loose if k < 3 else tight
        res = ctx.all_pairs(pts, r, T, r)
        st, (rp, col) = res.stats, res.download()
        res.release()
        assert st["sort_passes"] % 2 == 0 and st["max_cell"] > 24
        assert st["attempts"] == (2 if k == 3 else 1) or k == 0
        ref = oracle.rtg(pts, r, T, r).csr
        assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col), k
    ctx.close()


def test_inputs_that_alternate_settle():
    # two inputs of one shape whose pair counts, cells and rows differ: once both were built, no
    # build runs twice, and each still equals the oracle's
    d, n, m, r = 3, 4000, 6, 0.06
    a = gen.points_uniform(31, n, d)  # light cells and short rows
    b = gen.points_mixture(31, n, d, k=8, sigma=0.05, dtype=np.float64)
    T = gen.transforms(31, d, m, r)
    refs = [oracle.rtg(p, r, T, r).csr for p in (a, b)]
    ctx = rtg.Context(0)
    for k in range(10):
        which = k % 2
        res = ctx.all_pairs((a, b)[which], r, T, r)
        st, (rp, col) = res.stats, res.download()
        res.release()
        assert np.array_equal(rp, refs[which].row_ptr) and np.array_equal(col, refs[which].col), k
        assert k < 4 or st["attempts"] == 1, (k, st["attempts"])
    ctx.close()


@pytest.mark.parametrize("symmetric", [False, True])
def test_more_columns_than_recent_builds(symmetric):
    # the pairs fit the shape's pair buffer (16 a point at first) but not the column array, which
    # follows the pairs of recent builds: they are scattered again
    n, d, m, r = 6000, 3, 4, 0.05
    T = gen.transforms(63, d, m, r)
    few = gen.points_uniform(63, n, d)
    more = gen.points_uniform(64, n, d) * 0.7  # (no dense cells or long rows either)
    refs = {id(p): oracle.rtg(p, r, T, r).csr for p in (few, more)}
    assert 2 * refs[id(few)].nnz + 4096 < refs[id(more)].nnz < 16 * n
    with rtg.Context(0) as ctx:
        for k, pts in enumerate((few, few, few, more, more, few, more)):
            res = ctx.all_pairs(pts, r, T, r, symmetric=symmetric)
            st, (rp, col) = res.stats, res.download()
            res.release()
            ref = refs[id(pts)]
            if symmetric:
                i = np.repeat(np.arange(n), np.diff(rp))
                assert len(col) == 2 * ref.nnz
                assert np.array_equal(np.sort(i * n + col), np.sort(col * np.int64(n) + i))
                up = i < col
                rp, col = np.concatenate([[0], np.cumsum(np.bincount(i[up], minlength=n))]), col[up]
            assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col), k
            assert st["attempts"] == (2 if k == 3 else 1), k


def test_stored_results_hold_the_memory_of_their_pairs():
    # results kept after a much denser input of their shape: each holds its own columns (as much
    # again and 256 KB at most) and not the capacity the dense one needed
    import torch
    n, d, m, r = 20000, 3, 4, 0.05
    T = gen.transforms(65, d, m, r)
    few = gen.points_uniform(65, n, d)
    dense = gen.points_mixture(66, n, d, k=8, sigma=0.06, dtype=np.float64)
    with rtg.Context(0) as ctx:
        for pts in (few, dense, dense):
            res = ctx.all_pairs(pts, r, T, r)
            pairs = res.nnz
            res.release()
        assert 500000 < pairs < 1200000
        ref = oracle.rtg(few, r, T, r).csr
        ctx.all_pairs(few, r, T, r).release()
        before = torch.cuda.mem_get_info()[0]
        kept = [ctx.all_pairs(few, r, T, r) for _ in range(100)]
        held = before - torch.cuda.mem_get_info()[0]
        for res in (kept[0], kept[50], kept[99]):
            rp, col = res.download()
            assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col)
        each = 2 * 4 * ref.nnz + (4 << 16) + 8 * (n + 1)
        # and room for one build's full capacity, and the pool's rounding
        assert held <= 100 * each + 8 * pairs + (64 << 20), (held, each)
        for res in kept:
            res.release()


def test_key_width_settles():
    # keys wider than 32 bits once: the shape's builds keep that width while narrower keys come, give
    # it up after a number of them, and take it again, each with the oracle's pairs
    n, d, m = 3000, 6, 5
    pts = gen.points_uniform(67, n, d)
    small, wide = 0.03, 0.3
    grids = {r: gen.transforms(67, d, m, r) for r in (small, wide)}
    refs = {r: oracle.rtg(pts, r, grids[r], r).csr for r in grids}
    passes = []
    with rtg.Context(0) as ctx:
        for r in (small, small, *[wide] * 20, small, small):
            res = ctx.all_pairs(pts, r, grids[r], r)
            st, (rp, col) = res.stats, res.download()
            res.release()
            assert np.array_equal(rp, refs[r].row_ptr) and np.array_equal(col, refs[r].col)
            assert (st["key_bits"] > 32) == (r == small)
            passes.append(st["sort_passes"])
    assert passes[2] == passes[1] > passes[21] and passes[22] == passes[23] == passes[1], passes


def test_wide_keys_are_given_up_soon():
    # one build with keys of more than 32 bits does not leave the shape's next ones on 64-bit keys
    # for long, and narrower ones now and then do not make every wide build run twice
    n, d, m = 3000, 6, 5
    pts = gen.points_uniform(68, n, d)
    grids = {r: gen.transforms(68, d, m, r) for r in (0.03, 0.3)}

    def build(r):
        res = ctx.all_pairs(pts, r, grids[r], r)
        st = res.stats
        res.release()
        return st

    with rtg.Context(0) as ctx:
        wide = [build(0.03) for _ in range(2)][1]["sort_passes"]
        passes = [build(0.3)["sort_passes"] for _ in range(8)]
        assert passes[:4] == [wide] * 4 and max(passes[4:]) < wide, (wide, passes)
        assert build(0.03)["attempts"] == 2
        for _ in range(3):
            assert [build(r)["attempts"] for r in (0.3, 0.3, 0.3, 0.03)] == [1] * 4
