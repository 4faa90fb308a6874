"""Failure detection without a GPU fault: bounded device waits that run out return
RTG_E_TIMEOUT and leave the context usable; a failed device allocation returns RTG_E_NOMEM;
a host wait with a short limit returns RTG_E_TIMEOUT and the ticket still completes.

Each hook (rtg_set_test_hooks) only makes a bounded wait wait for something that never
happens, or one allocation give up: nothing traps, faults or hangs.  After every failure the
next build on the same context is compared element by element with the CPU oracle."""
import numpy as np
import pytest

import oracle
from paper_1409_8112_gb300 import gen, rtg

pytestmark = pytest.mark.gpu


def workload(n=100000, d=6, m=8, seed=0):
    pts = gen.points_uniform(seed, n, d)
    r = gen.radius_for_degree(n, d)
    T = gen.transforms(seed, d, m, r)
    return pts, r, T


_REF = {}


def reference(n=100000, d=6, m=8, seed=0):
    key = (n, d, m, seed)
    if key not in _REF:
        pts, r, T = workload(n, d, m, seed)
        _REF[key] = oracle.rtg(pts, r, T, r).csr
    return _REF[key]


def assert_exact(ctx, pts, r, T):
    res = ctx.all_pairs(pts, r, T, r)
    rp, col = res.download()
    res.release()
    ref = reference(pts.shape[0], pts.shape[1], len(T))
    assert np.array_equal(rp, ref.row_ptr)
    assert np.array_equal(col, ref.col)


@pytest.mark.parametrize("hook", [rtg.RTG_INJECT_SORT_WAIT, rtg.RTG_INJECT_SCAN_WAIT],
                         ids=["sort_lookback", "csr_scan"])
def test_bounded_wait_times_out_and_context_stays_usable(hook, monkeypatch):
    # the look-back sort strategy (the one with inter-block waits) for this context
    monkeypatch.setenv("RTG_SORT_VARIANT", "8,12,0")
    monkeypatch.setenv("RTG_AUTOTUNE", "0")
    pts, r, T = workload()
    with rtg.Context(0) as ctx:
        assert_exact(ctx, pts, r, T)  # the shape's launch plan (and graph) exists
        rtg.rtg_set_test_hooks(ctx.handle, hook, 64, 0)
        with pytest.raises(rtg.RTGError) as e:
            ctx.all_pairs(pts, r, T, r)
        assert e.value.status == rtg.RTG_E_TIMEOUT
        assert "wait" in rtg.lib().rtg_last_error(ctx.handle).decode()
        rtg.rtg_set_test_hooks(ctx.handle, 0, 0, 0)
        assert_exact(ctx, pts, r, T)
        assert_exact(ctx, pts, r, T)


def test_tensor_core_wait_times_out_and_context_stays_usable():
    import torch

    n, d = 5000, 6
    pts = gen.points_uniform(4, n, d)
    r = gen.radius_for_degree(n, d, 30.0)
    ref = oracle.brute(pts, r)
    dev = torch.from_numpy(pts).cuda()
    with rtg.Context(0) as ctx:
        rtg.rtg_set_test_hooks(ctx.handle, rtg.RTG_INJECT_TC_WAIT, 1024, 0)
        with pytest.raises(rtg.RTGError) as e:
            ctx.brute_force(dev, r, tensor="fp16")
        assert e.value.status == rtg.RTG_E_TIMEOUT
        rtg.rtg_set_test_hooks(ctx.handle, 0, 0, 0)
        res = ctx.brute_force(dev, r, tensor="fp16")
        rp, col = res.download()
        res.release()
        assert np.array_equal(rp, ref.row_ptr)
        assert np.array_equal(col, ref.col)


@pytest.mark.parametrize("after", [1, 2, 5])
def test_allocation_failure_returns_nomem(after):
    pts, r, T = workload()
    with rtg.Context(0) as ctx:
        # a fresh context: the first build allocates its workspace, then its outputs
        rtg.rtg_set_test_hooks(ctx.handle, 0, 0, after)
        with pytest.raises(rtg.RTGError) as e:
            ctx.all_pairs(pts, r, T, r)
        assert e.value.status == rtg.RTG_E_NOMEM
        assert_exact(ctx, pts, r, T)
        # a warm context: the next allocation is the output CSR's
        rtg.rtg_set_test_hooks(ctx.handle, 0, 0, 1)
        with pytest.raises(rtg.RTGError) as e:
            ctx.all_pairs(pts, r, T, r)
        assert e.value.status == rtg.RTG_E_NOMEM
        assert_exact(ctx, pts, r, T)


def test_host_wait_with_a_short_limit_times_out_and_the_ticket_completes():
    pts, r, T = workload()
    with rtg.Context(0) as ctx:
        ticket = rtg.rtg_submit(ctx.handle, pts, r, T, r)
        with pytest.raises(rtg.RTGError) as e:
            rtg.rtg_wait(ctx.handle, ticket, 1)
        assert e.value.status == rtg.RTG_E_TIMEOUT
        res = ctx.wait(ticket, -1, m=len(T))
        rp, col = res.download()
        res.release()
        ref = reference()
        assert np.array_equal(rp, ref.row_ptr)
        assert np.array_equal(col, ref.col)


def test_fp64_coordinates_beyond_the_fp32_range_are_decided_in_fp64():
    # points in the unit cube plus a few far beyond the FP32 range (two of them close to
    # each other); cells wide enough that every cell index fits a key
    rng = np.random.default_rng(9)
    base = rng.random((3000, 3))
    far = np.array([[1e39, 0.1, 0.2], [1e39, 0.15, 0.2], [-4e38, 0.5, 0.5], [0.3, 7e300, 0.1]])
    pts = np.concatenate([base[:1000], far, base[1000:]])
    r, c, m = 0.3, 1e301, 3
    T = gen.transforms(9, 3, m, c)
    ref = oracle.rtg(pts, r, T, c).csr
    assert ref.nnz > 0
    with rtg.Context(0) as ctx:
        res = ctx.all_pairs(pts, r, T, c)
        rp, col = res.download()
        st = res.stats
        res.release()
    assert np.array_equal(rp, ref.row_ptr)
    assert np.array_equal(col, ref.col)
    assert st["key_rechecks"] > 0 and st["dist_rechecks"] > 0


def subnormal_scaled_rotation(n=400, d=8, m=3):
    """Points, radius, transforms and cell side with R / c below the smallest normal FP32 number:
    the first axis is near zero for all points (its terms cancel), on either side of the cell wall
    there, and the roundings of R / c (multiples of 2^-149) add up over its terms."""
    c = 2.0 ** 120
    rng = np.random.default_rng(17)
    sign = np.where(np.arange(d) % 2 == 0, 1.0, -1.0)
    T = np.zeros((m, d * d + d))
    for t in range(m):
        T[t, :d] = 2.0 ** -29 * (512.0 + 3 * np.arange(d) + 7 * t + 0.5 + 0.04 * sign)
    big = 2.0 ** 127 * rng.uniform(0.6, 0.9, (n, d)) * sign
    y = big @ T[0, :d]
    big[:, -1] -= (y - 2.0 ** 120 * rng.normal(0.0, 4e-7, n)) / T[0, d - 1]
    return big, 2.0 ** 129, T, c


def test_cells_whose_scaled_rotation_is_subnormal():
    # the FP32 cell index is off by far more than its relative error bound: every such coordinate
    # has to be decided in FP64
    pts, r, T, c = subnormal_scaled_rotation()
    ref = oracle.rtg(pts, r, T, c).csr
    assert 0 < ref.nnz < len(pts) * (len(pts) - 1) // 2
    with rtg.Context(0) as ctx:
        res = ctx.all_pairs(pts, r, T, c)
        rp, col = res.download()
        res.release()
    assert np.array_equal(rp, ref.row_ptr)
    assert np.array_equal(col, ref.col)


def _same(res, ref):
    rp, col = res.download()
    band = res.stats["band"]
    res.release()
    assert np.array_equal(rp, ref.row_ptr)
    assert np.array_equal(col, ref.col)
    return band


def test_scratch_kept_for_speed_refuses_no_call():
    # the answer slots of index queries and the tiles of the default brute force are given back
    # when an allocation fails; what then still fails is refused as before
    n, d, m = 5000, 6, 8
    pts = gen.points_uniform(21, n, d)
    r = gen.radius_for_degree(n, d, 20.0)
    T = gen.transforms(21, d, m, r)
    q = gen.points_uniform(22, 700, d)
    pairs, exact = oracle.rtg(pts, r, T, r).csr, oracle.brute(pts, r)
    answers = oracle.rtg_query(pts, r, T, r, q)
    with rtg.Context(0) as ctx:
        ix = ctx.index(pts, r, T, r)
        calls = {"query": (lambda: ix.query(q), answers), "pairs": (lambda: ctx.all_pairs(pts, r, T, r), pairs),
                 "exact": (lambda: ctx.brute_force(pts, r), exact)}
        for call, ref in calls.values():  # warm: only outputs are allocated from here on
            for _ in range(2):
                _same(call(), ref)
        for name in ("pairs", "query", "exact"):
            for after in (1, 2):  # the row pointers, then the columns
                for warm, ref in (calls["query"], calls["exact"]):
                    _same(warm(), ref)
                rtg.rtg_set_test_hooks(ctx.handle, 0, 0, after)
                _same(calls[name][0](), calls[name][1])
                rtg.rtg_set_test_hooks(ctx.handle, 0, 0, 0)
        for _ in range(2):  # the first failure takes what was kept, the second has nothing to take
            rtg.rtg_set_test_hooks(ctx.handle, 0, 0, 1)
            try:
                _same(ctx.all_pairs(pts, r, T, r), pairs)
            except rtg.RTGError as e:
                assert e.status == rtg.RTG_E_NOMEM
                break
        else:
            raise AssertionError("no allocation failed")
        rtg.rtg_set_test_hooks(ctx.handle, 0, 0, 0)
        _same(ctx.brute_force(pts, r), exact)
        ix.close()


def test_default_brute_force_without_room_for_tiles():
    # whichever allocation of a first call fails: refused, or decided on the CUDA cores
    n, d = 4500, 4
    pts = gen.points_uniform(23, n, d, np.float32)
    r = gen.radius_for_degree(n, d, 9.0)
    ex = oracle.brute(pts, r)
    refused, plain, tiles = 0, 0, 0
    for after in range(1, 24):
        with rtg.Context(0) as ctx:
            rtg.rtg_set_test_hooks(ctx.handle, 0, 0, after)
            try:
                if _same(ctx.brute_force(pts, r), ex) > 0:
                    tiles += 1
                else:
                    plain += 1
            except rtg.RTGError as e:
                assert e.status == rtg.RTG_E_NOMEM
                refused += 1
    assert plain == 3 and refused > 5 and tiles > 0, (refused, plain, tiles)


@pytest.mark.parametrize("scale", [2.0 ** 27, 2.0 ** 28, 2.0 ** 29, 2.0 ** 61, 2.0 ** -60])
@pytest.mark.parametrize("d", [3, 8])
def test_cells_on_either_side_of_the_limits_of_the_subnormal_term(d, scale):
    # the error bound leaves the subnormal roundings out below 2^28 (coordinates, cells) and 2^60
    # (shifts and rotated coordinates)
    pts = gen.points_uniform(70 + d, 600, d) * scale
    r = gen.radius_for_degree(600, d) * scale
    T = gen.transforms(70 + d, d, 3, r)
    ref = oracle.rtg(pts, r, T, r).csr
    with rtg.Context(0) as ctx:
        res = ctx.all_pairs(pts, r, T, r)
        rp, col = res.download()
        res.release()
    assert ref.nnz > 0
    assert np.array_equal(rp, ref.row_ptr)
    assert np.array_equal(col, ref.col)
