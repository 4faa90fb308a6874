"""Tensor-core brute force (tcgen05 tiles, FP16 / BF16 hi-lo split, FP32 accumulation, FP64
band check): the pair set equals the FP64 definition exactly, and the observed tile error
stays inside the band."""
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


@pytest.mark.parametrize("tensor", ["fp16", "bf16"])
@pytest.mark.parametrize("d,n,dtype", [(1, 700, np.float64), (3, 3001, np.float64),
                                       (6, 4099, np.float32), (9, 2500, np.float64),
                                       (16, 1300, np.float32)])
def test_tc_brute_matches_oracle(ctx, tensor, d, n, dtype):
    pts = gen.points_uniform(50 + d, n, d, dtype)
    r = gen.radius_for_degree(n, d, 20.0)
    res = ctx.brute_force(pts, r, tensor=tensor)
    rp, col = res.download()
    ex = oracle.brute(pts, r)
    assert np.array_equal(rp, ex.row_ptr) and np.array_equal(col, ex.col)
    st = res.stats
    assert st["band"] >= 1e-3 * r * r * (1 - 1e-12)
    assert st["max_abs_err_d2"] < st["band"]
    res.release()


def test_tc_offset_coordinates(ctx):
    pts = gen.points_uniform(8, 3000, 4) * 2.0 + 5.0  # centring keeps the split accurate
    r = 0.25
    for tensor in ("fp16", "bf16"):
        res = ctx.brute_force(pts, r, tensor=tensor)
        rp, col = res.download()
        ex = oracle.brute(pts, r)
        assert np.array_equal(rp, ex.row_ptr) and np.array_equal(col, ex.col)


@pytest.mark.parametrize("tensor", ["fp16", "bf16"])
@pytest.mark.parametrize("sigma,n,d,dtype", [(0.01, 6000, 3, np.float32),
                                             (0.02, 8000, 6, np.float64),
                                             (0.05, 9000, 6, np.float32),
                                             (0.05, 5000, 12, np.float32)])
def test_dense_cells_on_tensor_cores_match_oracle(ctx, tensor, sigma, n, d, dtype):
    # clustered points (8 Gaussians): cells of hundreds to thousands of points, whose pairs go
    # through the tensor-core tiles; the set must equal the oracle's and the build without
    # the tiles, candidate counts included
    pts = gen.points_mixture(70 + d, n, d, k=8, sigma=sigma, dtype=dtype)
    r = gen.radius_for_degree(n, d, 6.0)
    T = gen.transforms(70 + d, d, 4, r)
    res = ctx.all_pairs(pts, r, T, r, tensor=tensor)
    rp, col = res.download()
    st = res.stats
    res.release()
    ref = oracle.rtg(pts, r, T, r)
    assert np.array_equal(rp, ref.csr.row_ptr) and np.array_equal(col, ref.csr.col)
    assert st["candidates"] == [s["candidates"] for s in ref.stats]
    assert st["large_cells"] > 0 and st["max_cell"] > 256


@pytest.mark.parametrize("two_pass_by_overflow", [True, False])
def test_tc_brute_writes_columns_of_dense_graphs(ctx, two_pass_by_overflow):
    # more pairs than a first build's buffer holds (16 a point): the columns come from a second
    # enumeration; the shape's next build holds them all
    n, d = (1500, 3) if two_pass_by_overflow else (400, 2)
    pts = gen.points_uniform(77, n, d, np.float32)
    r = gen.radius_for_degree(n, d, 150.0)
    ex = oracle.brute(pts, r)
    assert ex.nnz > 16 * n
    own = rtg.Context(0)
    for k in range(2):
        res = own.brute_force(pts, r, tensor="fp16")
        rp, col = res.download()
        assert res.stats["attempts"] == (2 if k == 0 else 1)
        res.release()
        assert np.array_equal(rp, ex.row_ptr) and np.array_equal(col, ex.col)
    own.close()


@pytest.mark.parametrize("n,d,dtype,scale,shift,degree,tiles", [
    (4095, 6, np.float64, 1.0, 0.0, 20.0, False),   # below the size rule
    (4096, 6, np.float64, 1.0, 0.0, 20.0, True),
    (4223, 1, np.float32, 1.0, 0.0, 9.0, None),
    (4225, 4, np.float32, 1.0, 0.0, 12.0, True),    # one K = 16 part
    (4099, 5, np.float64, 1.0, 0.0, 12.0, True),    # two parts
    (5000, 9, np.float32, 1.0, 0.0, 12.0, True),
    (4500, 10, np.float64, 1.0, 0.0, 12.0, True),   # norms in the hi block
    (4300, 13, np.float32, 1.0, 0.0, 12.0, True),   # norms added afterwards
    (4111, 3, np.float64, 1e-3, 0.0, 12.0, None),
    (4111, 3, np.float64, 1e-7, 0.0, 12.0, False),  # the halves cannot resolve such points
    (4111, 6, np.float32, 1e3, 0.0, 12.0, False),   # norms beyond the half range
    (4111, 6, np.float64, 1.0, 1e4, 12.0, True),    # far from the origin: the tiles are centred
    (4111, 2, np.float64, 1.0, 0.0, 0.02, False),   # r far below the points' extent
])
def test_default_brute_force_by_either_kernel(ctx, n, d, dtype, scale, shift, degree, tiles):
    # the default brute force takes tensor-core tiles where their error bound is narrow against
    # r^2; the set is the oracle's whichever kernel decided it
    pts = (gen.points_uniform(n + d, n, d) * scale + shift).astype(dtype)
    r = gen.radius_for_degree(n, d, degree) * scale
    ex = oracle.brute(pts, r)
    for kw in ({}, {"count_only": True}, {"symmetric": True}):
        res = ctx.brute_force(pts, r, **kw)
        st = res.stats
        assert st["pairs"] == ex.nnz
        if tiles is not None:
            assert (st["band"] > 0) == tiles
        if not kw:
            rp, col = res.download()
            assert np.array_equal(rp, ex.row_ptr) and np.array_equal(col, ex.col)
        res.release()


def _cuda_cores():
    # a context with a memory budget keeps the default brute force to the CUDA cores
    return rtg.Context(0, 8 << 30)


@pytest.mark.parametrize("n,d,dtype,degree", [(4096, 6, np.float64, 20.0), (5001, 9, np.float32, 12.0),
                                              (4500, 12, np.float64, 12.0), (4300, 16, np.float32, 40.0),
                                              (4097, 3, np.float32, 300.0), (4096, 0, np.float64, 0.0)])
def test_default_brute_force_counts_as_on_cuda_cores(ctx, n, d, dtype, degree):
    # the pairs the tiles leave are decided by the filter of the CUDA-core kernel, so its counters
    # are the same; the last case is a lattice with many pairs at exactly r
    if d:
        pts = gen.points_uniform(60 + d, n, d, dtype)
        r = gen.radius_for_degree(n, d, degree)
    else:
        pts = np.stack(np.meshgrid(*[np.arange(16) / 32.0] * 3), -1).reshape(-1, 3)
        r = 3.0 / 32.0
    with _cuda_cores() as plain:
        for kw in ({}, {"count_only": True}, {"symmetric": True}):
            a, b = ctx.brute_force(pts, r, **kw), plain.brute_force(pts, r, **kw)
            assert a.stats["band"] > 0 or (degree > 100.0 and "count_only" in kw)
            assert b.stats["band"] == 0
            for key in ("pairs", "owned_candidates", "dist_rechecks", "near_r"):
                assert a.stats[key] == b.stats[key], key
            assert a.stats["owned_candidates"] >= a.stats["pairs"] > 0
            assert d or a.stats["near_r"] > 0
            a.release()
            b.release()


@pytest.mark.parametrize("share,emit_tiles,count_tiles", [(0.002, True, True), (0.2, True, False),
                                                          (0.6, False, False), (1.0, False, False)])
def test_default_brute_force_of_dense_graphs(ctx, share, emit_tiles, count_tiles):
    # many pairs within r: the tiles' candidates would cost more than they save
    n, d = 4200, 6
    pts = gen.points_uniform(61, n, d, np.float32)
    k = np.random.default_rng(62).integers(0, n, (2, 20000))
    k = k[:, k[0] != k[1]]
    s = np.sort(((pts[k[0]].astype(np.float64) - pts[k[1]]) ** 2).sum(1))
    r = float(np.sqrt(s[int(share * (len(s) - 1))])) * (3.0 if share == 1.0 else 1.0)
    ex = oracle.brute(pts, r)
    for kw, tiles in (({}, emit_tiles), ({"count_only": True}, count_tiles)):
        res = ctx.brute_force(pts, r, **kw)
        assert res.stats["pairs"] == ex.nnz
        assert (res.stats["band"] > 0) == tiles
        if not kw:
            rp, col = res.download()
            assert np.array_equal(rp, ex.row_ptr) and np.array_equal(col, ex.col)
        res.release()


def test_default_brute_force_does_not_ask_refused_tiles_again():
    # a shape whose tiles were refused at a radius launches two kernels less for a while; another
    # radius asks at once, the same one after 16 builds
    n, d = 4300, 2
    wide = gen.points_uniform(64, n, d)
    r = gen.radius_for_degree(n, d, 0.02)
    narrow = wide * (20.0 * r)  # the same radius, an extent the tiles resolve
    with rtg.Context(0) as own:
        def call(pts, radius):
            res = own.brute_force(pts, radius)
            ex, (rp, col), st = oracle.brute(pts, radius), res.download(), res.stats
            assert np.array_equal(rp, ex.row_ptr) and np.array_equal(col, ex.col)
            res.release()
            return st["launches"], st["band"] > 0
        asked = call(wide, r)
        assert not asked[1]
        for _ in range(3):
            assert call(wide, r) == (asked[0] - 2, False)
        assert call(wide, 8.0 * gen.radius_for_degree(n, d))[1]
        assert call(wide, r) == asked
        for _ in range(16):
            assert not call(narrow, r)[1]
        for _ in range(2):
            assert call(narrow, r)[1]


def _tile_error_bound(M, d, bf16):
    """|tile d^2 - d^2| for coordinates within M of the centre: half-precision hi + lo of the
    coordinates (and of the norms, for d <= 12) with unit roundoff u, FP32 sums of 48 or 52 terms
    in any order."""
    u, u32 = (2.0 ** -8 if bf16 else 2.0 ** -11), 2.0 ** -24
    e = 16.0 * d * u32 * M * M + 2.0 * (2.0 * d * M * M * (2.0 * u * u + 2.0 ** -22) + d * 2.0 ** -24 * M)
    if d <= 12:
        return e + 2.0 * (d * u32 * d * M * M + u * u * d * M * M + 2.0 ** -25) + 2080.0 * u32 * d * M * M
    return e + 768.0 * u32 * d * M * M + 2.0 * d * u32 * d * M * M + 12.0 * u32 * d * M * M


@pytest.mark.parametrize("tensor", ["fp16", "bf16"])
@pytest.mark.parametrize("d", [1, 2, 4, 5, 6, 9, 10, 12, 13, 16])
@pytest.mark.parametrize("kind,scale", [("uniform", 1.0), ("corners", 1.0), ("mixed", 1.0),
                                        ("uniform", 60.0), ("corners", 1e-3)])
def test_tile_error_of_every_pair_is_within_its_bound(ctx, tensor, d, kind, scale):
    # rejections rely on the error bound of the tiles.  With every pair within r none is rejected,
    # and the largest error over all pairs is reported
    n = 900
    rng = np.random.default_rng(100 * d + len(kind))
    pts = rng.uniform(-1.0, 1.0, (n, d))
    if kind == "corners":  # halves of the same sign, all terms near their largest
        pts = np.sign(pts) * (1.0 - rng.random((n, d)) * 2.0 ** -9)
    elif kind == "mixed":  # large and tiny magnitudes next to each other
        pts *= 2.0 ** -rng.integers(0, 24, (n, d)).astype(np.float64)
    pts = np.vstack([pts, np.full((1, d), 1.0), np.full((1, d), -1.0)]) * scale
    r = 4.0 * scale * np.sqrt(d)
    res = ctx.brute_force(pts, r, tensor=tensor, count_only=True)
    assert res.stats["pairs"] == (n + 2) * (n + 1) // 2
    assert res.stats["max_abs_err_d2"] <= _tile_error_bound(scale, d, tensor == "bf16")
    res.release()
