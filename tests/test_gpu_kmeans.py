"""GPU parity: k-means (array container keyed by cluster id).

Assignments must equal the FP64 oracle's exactly; centroids must be within
1e-5 relative (per centroid, ||c - c64|| / max(||c64||, 1)) of the oracle's.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _rel_err(c, ref):
    num = np.linalg.norm(c.astype(np.float64) - ref.astype(np.float64), axis=1)
    den = np.maximum(np.linalg.norm(ref.astype(np.float64), axis=1), 1.0)
    return float((num / den).max())


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _run(mr, x, init, iters, precision=0, on_device=True):
    if on_device:
        return mr.kmeans(_dev(x), _dev(init), iters, precision)
    return mr.kmeans(x, init, iters, precision)


def _assign_all(x, c):
    """The oracle's FP64 assignment of every point, computed serially on row
    slices by a pool of host threads (the oracle call releases the GIL)."""
    import concurrent.futures as cf
    import os
    nth = max(1, min(32, os.cpu_count() or 1))
    step = (x.shape[0] + nth - 1) // nth
    parts = [x[i: i + step] for i in range(0, x.shape[0], step)]
    with cf.ThreadPoolExecutor(nth) as ex:
        return np.concatenate(list(ex.map(lambda p: oracle.kmeans_assign(p, c), parts)))


def _run_ctx(mr, ctx, dx, cur, iters, precision):
    n, d = dx.shape
    j = ctx.add_job(mr.KMEANS_F32, dx, km_dims=d, km_k=cur.shape[0], km_iters=iters, km_init=_dev(cur),
                    km_precision=precision)
    ctx.run()
    out = mr.split_kmeans_result(ctx.fetch(j), n, d, cur.shape[0])
    ctx.release(j)
    return out


@pytest.mark.parametrize("n,d,k,iters", [
    (20_000, 64, 256, 3),   # the workload's shape, reduced N
    (5_001, 37, 50, 2),     # ragged dims / tiles
    (3_000, 100, 20, 2),    # D > 64: chunked dimensions
    (4_000, 16, 300, 2),    # K > 256: chunked centroids
    (6_000, 128, 260, 2),   # K*D sums too large for shared memory: the sorted update
    (9_001, 64, 300, 2),    # window-sorted update with K not a multiple of 32
    (5_000, 64, 1, 2),      # window-sorted update, one cluster
    (6_000, 8, 3_000, 2),   # K x D sums fit, but not beside the window buffers: the row-pipelined update
    (3_001, 67, 20, 2),     # D > 64 and not a multiple of 4: the plain local-array update
    (777, 3, 1, 2),         # K = 1: the global mean
    (64, 8, 64, 1),         # every point its own centroid
])
def test_kmeans_fp32_vs_oracle(mr, n, d, k, iters):
    x, _, _ = synth.kmeans_points(n, d, max(1, min(k, 256)), seed=n + d + k)
    init = synth.kmeans_init(x, k, seed=n)
    c_ref, a_ref = oracle.kmeans(x, init, iters)
    c, a, stats = _run(mr, x, init, iters)
    assert np.array_equal(a, a_ref)
    assert _rel_err(c, c_ref) <= TOL
    assert int(stats[2]) == iters


@pytest.mark.parametrize("precision", [0, 1])
def test_kmeans_points_not_16_byte_aligned(mr, precision):
    """Points 4 bytes into a buffer: no bulk copies and no 8-byte loads; the
    window-sorted update reads them with 4-byte loads."""
    import torch
    x, _, _ = synth.kmeans_points(5000, 64, 32, seed=51)
    init = synth.kmeans_init(x, 32, seed=52)
    buf = torch.zeros(x.size + 1, dtype=torch.float32, device="cuda")
    buf[1:] = torch.from_numpy(x.ravel()).cuda()
    c_ref, a_ref = oracle.kmeans(x, init, 3)
    c, a, stats = mr.kmeans(buf[1:].view(5000, 64), _dev(init), 3, precision)
    assert np.array_equal(a, a_ref)
    assert _rel_err(c, c_ref) <= TOL


def test_kmeans_host_inputs(mr):
    x, _, _ = synth.kmeans_points(4096, 32, 64, seed=5)
    init = synth.kmeans_init(x, 64, seed=6)
    c_ref, a_ref = oracle.kmeans(x, init, 2)
    c, a, _ = _run(mr, x, init, 2, on_device=False)
    assert np.array_equal(a, a_ref) and _rel_err(c, c_ref) <= TOL


def test_kmeans_exact_ties_take_lowest_index(mr):
    x, _, _ = synth.kmeans_points(6000, 8, 16, seed=21)
    init = synth.kmeans_init(x, 16, seed=22)
    init[9] = init[4]     # duplicate centroid: index 4 must win every tie
    init[15] = init[0]
    c_ref, a_ref = oracle.kmeans(x, init, 1)
    c, a, stats = _run(mr, x, init, 1)
    assert np.array_equal(a, a_ref)
    assert not np.any(a == 9) and not np.any(a == 15)
    assert int(stats[1]) > 0  # the tied points were re-checked in FP64
    assert _rel_err(c, c_ref) <= TOL


@pytest.mark.parametrize("precision,d", [(0, 64), (1, 64), (0, 8)])
def test_kmeans_all_centroids_tied(mr, precision, d):
    """Every centroid the same point: every distance ties, every point goes
    to the FP64 stage with all 256 centroids as candidates (in chunks of the
    stage's product scratch: 128 at D = 64, 256 at D = 8), and index 0 wins
    every tie, as in the definition."""
    x, _, _ = synth.kmeans_points(3000, d, 16, seed=81 + d)
    init = np.repeat(x[7:8], 256, axis=0)
    a_ref = oracle.kmeans_assign(x, init)
    c_ref, _ = oracle.kmeans_update(x, a_ref, init)
    c, a, st = _run(mr, x, init, 1, precision)
    assert np.array_equal(a, a_ref) and not np.any(a)
    assert int(st[1]) >= 2999  # (a point equal to the centroid may be decided earlier)
    assert _rel_err(c, c_ref) <= TOL


def test_kmeans_empty_cluster_keeps_centroid(mr):
    x, _, _ = synth.kmeans_points(3000, 4, 3, seed=31)
    init = np.concatenate([x[:3], np.full((1, 4), 1e4, dtype=np.float32)])
    c_ref, a_ref = oracle.kmeans(x, init, 3)
    c, a, _ = _run(mr, x, init, 3)
    assert np.array_equal(a, a_ref)
    assert np.array_equal(c[3], init[3])
    assert _rel_err(c, c_ref) <= TOL


def test_kmeans_teacher_forced_iterations(mr):
    """Each GPU iteration, started from the oracle's centroids, reproduces the
    oracle's assignment exactly and its update within tolerance."""
    x, _, _ = synth.kmeans_points(30_000, 64, 256, seed=41)
    cur = synth.kmeans_init(x, 256, seed=42)
    for _ in range(4):
        a_ref = oracle.kmeans_assign(x, cur)
        c_ref, _ = oracle.kmeans_update(x, a_ref, cur)
        c, a, _ = _run(mr, x, cur, 1)
        assert np.array_equal(a, a_ref)
        assert _rel_err(c, c_ref) <= TOL
        cur = c_ref


def test_kmeans_rejects_bad_args(mr):
    x = np.zeros((10, 4), dtype=np.float32)
    with pytest.raises(mr.MRError):
        mr.kmeans(x, np.zeros((2, 4), dtype=np.float32), 0)
    c = mr.Context()
    with pytest.raises(mr.MRError):
        c.add_job(mr.KMEANS_F32, x, km_dims=3, km_k=2, km_iters=1, km_init=np.zeros((2, 3), dtype=np.float32))
    c.close()


@pytest.mark.slow
def test_kmeans_full_size_fp32(mr):
    """4M x 64 points, K = 256, 10 iterations: determinism across a split run;
    the tenth iteration's assignment of EVERY point equals the FP64 oracle's
    on the GPU's ninth centroids, for the FP32 path and both tensor-core
    paths (whose persistent CTAs run ~216 tiles each here); and the final
    update equals the oracle's FP64 update within tolerance."""
    import torch
    x, _, _ = synth.kmeans_points(4 << 20, 64, 256)
    init = synth.kmeans_init(x, 256)
    dx = torch.from_numpy(x).cuda()
    c10, a10, _ = mr.kmeans(dx, _dev(init), 10)
    c9, _, _ = mr.kmeans(dx, _dev(init), 9)
    c10b, a10b, _ = mr.kmeans(dx, _dev(c9), 1)
    assert np.array_equal(c10, c10b) and np.array_equal(a10, a10b)
    a_ref = _assign_all(x, c9)
    assert np.array_equal(a10, a_ref)
    for precision in (1, 2):
        _, a_tc, st = mr.kmeans(dx, _dev(c9), 1, precision)
        assert np.array_equal(a_tc, a_ref), precision
        assert int(st[3]) == 0
    c_upd, _ = oracle.kmeans_update(x, a10, c9)
    assert _rel_err(c10, c_upd) <= TOL


@pytest.mark.parametrize("precision,d", [(0, 64), (1, 64), (2, 64), (1, 21)])
def test_kmeans_many_tiles_per_cta_teacher_forced(mr, precision, d):
    """The persistent kernels capped at 4 CTAs: each tensor-core CTA runs ~39
    tiles of 128 points (its copy ring, operand stages, TMEM accumulators and
    key hand-off all wrap many times; D = 21: the converters' own row loads),
    each FP32 CTA ~78 tiles of 64, and each update
    CTA its ~5,000 points in two windows.  Every assignment of every
    iteration, started from the oracle's centroids, equals the oracle's."""
    x, _, _ = synth.kmeans_points(20_000, d, 256, seed=45 + precision)
    cur = synth.kmeans_init(x, 256, seed=46)
    dx = _dev(x)
    ctx = mr.Context()
    ctx.set_option(mr.OPT_KM_GRID_CAP, 4)
    for _ in range(3):
        a_ref = oracle.kmeans_assign(x, cur)
        c_ref, _ = oracle.kmeans_update(x, a_ref, cur)
        c, a, st = _run_ctx(mr, ctx, dx, cur, 1, precision)
        assert np.array_equal(a, a_ref)
        assert _rel_err(c, c_ref) <= TOL
        assert int(st[3]) == 0
        cur = c_ref
    ctx.close()


@pytest.mark.parametrize("d,k", [(64, 256), (64, 17), (64, 380), (48, 256), (37, 17), (33, 100), (8, 64), (1, 5)])
def test_kmeans_window_update_many_windows(mr, d, k):
    """The update for D <= 64 sorts each window of 8,192 points (4,096 when
    the K x D sums leave too little shared memory: K = 380 at D = 64) by
    cluster and sums runs in registers (lanes past D idle).  Two CTAs of
    10,001 points each: a full window and a ragged one (4,096: two full and a
    ragged third), so the window loop, the per-window histogram and scatter
    and the run flushes across windows are all exercised, against the
    oracle's update from the same assignment."""
    import torch
    x, _, _ = synth.kmeans_points(20_002, d, min(k, 64), seed=71 + k + d)
    dx = torch.from_numpy(x).cuda()
    cur = synth.kmeans_init(x, k, seed=72)
    ctx = mr.Context()
    ctx.set_option(mr.OPT_KM_GRID_CAP, 2)
    for _ in range(2):
        a_ref = oracle.kmeans_assign(x, cur)
        c_ref, _ = oracle.kmeans_update(x, a_ref, cur)
        c, a, st = _run_ctx(mr, ctx, dx, cur, 1, 0)
        assert np.array_equal(a, a_ref)
        assert _rel_err(c, c_ref) <= TOL
        cur = c_ref
    ctx.close()


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_kmeans_eight_tiles_per_cta_natural_grid(mr, precision):
    """152 x 8 x 128 points at the default grid (one tensor-core CTA per SM):
    every CTA runs 8 tiles, past the two-deep rings' first reuse.  All points
    against the oracle, teacher-forced for two iterations."""
    import torch
    n = torch.cuda.get_device_properties(0).multi_processor_count * 8 * 128
    x, _, _ = synth.kmeans_points(n, 64, 256, seed=47)
    cur = synth.kmeans_init(x, 256, seed=48)
    dx = _dev(x)
    ctx = mr.Context()
    for _ in range(2):
        a_ref = _assign_all(x, cur)
        c_ref, _ = oracle.kmeans_update(x, a_ref, cur)
        c, a, st = _run_ctx(mr, ctx, dx, cur, 1, precision)
        assert np.array_equal(a, a_ref)
        assert _rel_err(c, c_ref) <= TOL
        cur = c_ref
    ctx.close()


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("n,d,k,iters", [
    (20_000, 64, 256, 3),   # the workload's shape, reduced N
    (5_001, 37, 50, 2),     # D < 64 (zero-padded), K not a multiple of 16
    (777, 3, 1, 2),         # K = 1
    (300, 64, 16, 1),       # fewer points than one CTA per SM
    (641, 1, 4, 2),         # D = 1, a last tile of one point
    (2_050, 48, 40, 2),     # D a multiple of 16 below 64
    (6_000, 64, 136, 2),    # 144 columns: the last epilogue quarter idle, the third partly masked
    (6_000, 20, 200, 2),    # 208 columns
])
def test_kmeans_bf16_tensor_core_vs_oracle(mr, precision, n, d, k, iters):
    x, _, _ = synth.kmeans_points(n, d, max(1, min(k, 256)), seed=n + d + k + 7)
    init = synth.kmeans_init(x, k, seed=n + 1)
    c_ref, a_ref = oracle.kmeans(x, init, iters)
    c, a, stats = _run(mr, x, init, iters, precision=precision)
    assert np.array_equal(a, a_ref)
    assert _rel_err(c, c_ref) <= TOL
    assert int(stats[3]) == 0


def test_kmeans_bf16_teacher_forced(mr):
    x, _, _ = synth.kmeans_points(30_000, 64, 256, seed=43)
    cur = synth.kmeans_init(x, 256, seed=44)
    for _ in range(3):
        a_ref = oracle.kmeans_assign(x, cur)
        c_ref, _ = oracle.kmeans_update(x, a_ref, cur)
        c, a, stats = _run(mr, x, cur, 1, precision=1)
        assert np.array_equal(a, a_ref)
        assert _rel_err(c, c_ref) <= TOL
        cur = c_ref


@pytest.mark.slow
def test_kmeans_full_size_bf16_matches_fp32_path(mr):
    """4M x 64, K = 256, 10 iterations: the tensor-core path gives the same
    assignments and centroids as the FP32 path (both equal the FP64 argmin
    each iteration, and the integer sums make the update deterministic)."""
    import torch
    x, _, _ = synth.kmeans_points(4 << 20, 64, 256)
    init = synth.kmeans_init(x, 256)
    dx = torch.from_numpy(x).cuda()
    c32, a32, _ = mr.kmeans(dx, _dev(init), 10, 0)
    c16, a16, st = mr.kmeans(dx, _dev(init), 10, 1)
    assert np.array_equal(a16, a32)
    assert np.array_equal(c16, c32)
    assert int(st[3]) == 0


@pytest.mark.parametrize("n,d,k", [(1_999, 64, 256), (2_001, 63, 255), (1_153, 1, 1), (1_281, 2, 9)])
@pytest.mark.parametrize("offset,scale", [(0.0, 1.0), (1000.0, 1.0), (-3e6, 1e4), (0.0, 1e-15), (1e15, 1e15)])
def test_kmeans_fp32_on_the_tensor_cores(mr, n, d, k, offset, scale):
    """FP32 jobs that take the tensor-core pass, at the edges of its shapes and
    with data far from the origin, tiny and huge: one round from the same
    centroids gives the oracle's assignments and centroids."""
    x, _, _ = synth.kmeans_points(n, d, max(1, min(k, 32)), seed=n + d)
    x = (x * np.float32(scale) + np.float32(offset)).astype(np.float32)
    init = synth.kmeans_init(x, k, seed=n)
    c_ref, a_ref = oracle.kmeans(x, init, 1)
    c, a, stats = _run(mr, x, init, 1, 0)
    assert np.array_equal(a, a_ref)
    assert _rel_err(c, c_ref) <= TOL
    assert int(stats[3]) == 0


@pytest.mark.parametrize("n,d,k", [
    (30_001, 64, 40),     # window-sorted update, 8-byte loads
    (30_001, 21, 9),      # window-sorted update, one dimension per lane
    (12_001, 96, 16),     # row-pipelined update
    (12_003, 67, 16),     # plain local-array update
    (12_001, 130, 260),   # sorted update
])
@pytest.mark.parametrize("precision", [0, 1])
def test_kmeans_update_by_changes(mr, n, d, k, precision):
    """Rounds in which few points change cluster update the sums by those
    points alone.  Ten rounds in one call equal ten calls of one round (each a
    full update), byte for byte: the sums are exact integers."""
    if precision and (d > 64 or k > 256):
        pytest.skip("shape outside the BF16 path")
    x, _, _ = synth.kmeans_points(n, d, 8, seed=n + d, sigma=4.0)
    dx = _dev(x)
    cur = synth.kmeans_init(x, k, seed=n)
    c10, a10, _ = mr.kmeans(dx, _dev(cur), 10, precision)
    moved, last = [], None
    for _ in range(10):
        cur, a, _ = mr.kmeans(dx, _dev(cur), 1, precision)
        moved.append(n if last is None else int((a != last).sum()))
        last = a
    assert np.array_equal(a10, last)
    assert np.array_equal(c10, cur)
    assert min(moved) <= n // 32 < max(moved)  # both kinds of update ran


@pytest.mark.parametrize("n,d", [(30_001, 64), (30_001, 21), (20_003, 33)])
def test_kmeans_changes_collected_or_direct(mr, n, d):
    """The window-sorted update collects the changes per CTA (up to n / 4 moved
    points) or adds them straight (up to n / 256): the rounds reach both, and
    equal single rounds (each a full update) byte for byte."""
    x, _, _ = synth.kmeans_points(n, d, 8, seed=n + d, sigma=2.0)
    cur = synth.kmeans_init(x, 8, seed=n)
    dx = _dev(x)
    c14, a14, _ = mr.kmeans(dx, _dev(cur), 14, 0)
    moved, last = [], None
    for _ in range(14):
        cur, a, _ = mr.kmeans(dx, _dev(cur), 1, 0)
        if last is not None:
            moved.append(int((a != last).sum()))
        last = a
    assert np.array_equal(a14, last)
    assert np.array_equal(c14, cur)
    assert any(0 < m <= n // 256 for m in moved)
    assert any(n // 256 < m <= n // 4 for m in moved)


@pytest.mark.parametrize("n,d,k,cap", [
    (1_999, 65, 3, 0),      # one value in the second dimension chunk
    (1_281, 128, 257, 0),   # one centroid in the second centroid chunk
    (20_001, 96, 300, 3),   # many tiles per CTA: two point buffers, two ring stages
    (12_003, 130, 520, 3),  # three dimension chunks (one point buffer), three centroid chunks, rows not 16-byte
    (5_003, 256, 256, 3),   # the widest rows
    (9_001, 5, 777, 3),     # few dimensions, many centroids: four ring stages
    (2_001, 3, 4_096, 0),   # the most centroids
    (130, 200, 100, 0),     # a last tile of two points
])
@pytest.mark.parametrize("offset", [0.0, 5e4])
def test_kmeans_wide_tensor_core_pass(mr, n, d, k, cap, offset):
    """FP32 jobs beyond 64 dimensions or 256 centroids: two rounds, each from
    the oracle's centroids, give the oracle's assignments and centroids."""
    x, _, _ = synth.kmeans_points(n, d, 16, seed=n + d)
    x = x + np.float32(offset)
    ctx = mr.Context()
    ctx.set_option(mr.OPT_KM_GRID_CAP, cap)
    dx, cur = _dev(x), synth.kmeans_init(x, min(k, n), seed=n)
    for _ in range(2):
        c_ref, a_ref = oracle.kmeans(x, cur, 1)
        c, a, st = _run_ctx(mr, ctx, dx, cur, 1, 0)
        assert np.array_equal(a, a_ref)
        assert _rel_err(c, c_ref) <= TOL
        assert int(st[3]) == 0
        cur = c_ref
    ctx.close()


@pytest.mark.parametrize("n,d,k,comps,sigma", [
    (600_011, 64, 256, 256, 1.0),    # listed rows copied by the bulk copy engine; most points skipped
    (600_011, 64, 256, 8, 4.0),      # overlapping clusters: few points skipped
    (2_000_003, 21, 67, 40, 2.0),    # listed rows loaded by the converters
    (1_100_001, 2, 130, 256, 1.0),   # many small clusters in the plane
])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_kmeans_skipped_points(mr, n, d, k, comps, sigma, precision):
    """Jobs large enough for the filter: nine rounds in one call equal nine
    calls of one round (which compute every distance), byte for byte."""
    x, _, _ = synth.kmeans_points(n, d, comps, seed=n + d, sigma=sigma)
    dx = _dev(x)
    cur = synth.kmeans_init(x, k, seed=n)
    c9, a9, _ = mr.kmeans(dx, _dev(cur), 9, precision)
    for _ in range(9):
        cur, a, _ = mr.kmeans(dx, _dev(cur), 1, precision)
    assert np.array_equal(a9, a)
    assert np.array_equal(c9, cur)


@pytest.mark.parametrize("n,d,k", [
    (3_000, 64, 256),  # four quarters of 64 columns
    (3_000, 64, 100),  # 32, 32, 32, 16 (12 of them padding)
    (2_000, 9, 144),   # 48 columns each
    (2_000, 5, 17),    # 16 columns, one centroid in the second quarter
    (2_000, 3, 2),
    (1_500, 80, 300),  # wide pass, 44 centroids in the last accumulator
    (1_500, 20, 700),
])
@pytest.mark.parametrize("spread", [0.0, 1e-6, 1e-4])
def test_kmeans_close_centroids_in_the_grid(mr, n, d, k, spread):
    """Groups of four centroids within `spread` of one another (equal at 0) that
    form rectangles in the 8 x 8 grid of an accumulator quarter: the smallest
    keys of rows and columns can hide two of them behind the other two."""
    rng = np.random.default_rng(n + d + k)
    group = np.array([8 * (c % 64 // 16) + (c % 8) // 2 + 64 * (c // 64) for c in range(k)])
    means = rng.normal(0, 3, (group.max() + 1, d)).astype(np.float32)
    init = (means[group] * (1 + spread * rng.standard_normal((k, d)))).astype(np.float32)
    x = (means[rng.integers(0, len(means), n)] + rng.normal(0, 0.5, (n, d))).astype(np.float32)
    c_ref, a_ref = oracle.kmeans(x, init, 1)
    for precision in (0, 1):
        if precision and (d > 64 or k > 256):
            continue
        c, a, _ = _run(mr, x, init, 1, precision)
        assert np.array_equal(a, a_ref)
        assert _rel_err(c, c_ref) <= TOL


@pytest.mark.parametrize("n,d,k,iters", [
    (20_000, 64, 64, 2),    # tensor-core pass, whole tiles in bulk copies
    (6_001, 37, 50, 2),     # values loaded by the converters
    (6_001, 100, 300, 2),   # wide tensor-core pass
    (400_009, 16, 250, 5),  # with the filter's bounds
    (3_000, 300, 20, 2),    # FP32 SIMT pass
])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 3e30])
@pytest.mark.parametrize("offset", [0.0, 1000.0])
def test_kmeans_centroids_not_finite(mr, n, d, k, iters, bad, offset):
    """Initial centroids with NaN or infinite coordinates, or whose norm
    overflows: the bound on the distances' error is then not finite, so it may
    decide no point.  Such a centroid wins no point and stays."""
    x, _, _ = synth.kmeans_points(n, d, 16, seed=n + d, sigma=4.0)
    x = x + np.float32(offset)
    init = synth.kmeans_init(x, k, seed=n)
    init[3] = bad
    init[k - 1, d // 2] = bad
    c_ref, a_ref = oracle.kmeans(x, init, iters)
    finite = np.isfinite(c_ref).all(axis=1)
    for precision in (0, 1, 2):
        if precision and (d > 64 or k > 256):
            continue
        c, a, _ = _run(mr, x, init, iters, precision)
        assert np.array_equal(a, a_ref), precision
        assert _rel_err(c[finite], c_ref[finite]) <= TOL
        assert np.array_equal(c[~finite], c_ref[~finite], equal_nan=True)


def _a256(v):
    return (v + 255) // 256 * 256


def _km_bytes(n, d, k, precision):
    """Device bytes within which a job has always run: the result, and scratch of
    the sizes the first form of the passes took."""
    scratch = (_a256(4 * k * d) + _a256(4 * n + 16) + _a256(8 * k * d) + 2 * _a256(8 * k) + 3 * 256 +
               2 * _a256(4 * n) + _a256(8 * n) + _a256(4 * k))
    if precision:
        scratch += _a256(4 * n) + _a256(4 * k * d)
    if 8 * k * d + 4 * k <= 200 * 1024:
        scratch += _a256(160 * 8 * k * d)
    return _a256((4 * k * d + 4 * n + 7) // 8 * 8 + 32) + scratch


@pytest.mark.parametrize("limit", ["budget", "allocator"])
@pytest.mark.parametrize("n,d,k,precision", [
    (3_000, 64, 256, 0), (3_000, 64, 256, 1), (500, 1, 1, 0), (40, 48, 17, 1), (7, 33, 250, 1),
    (2_000, 100, 300, 0), (900, 256, 1_000, 0),    # the wide pass's shapes, without room for its operands
    (600, 1_024, 64, 0), (50, 1_024, 4_096, 0), (700, 7, 4_096, 0), (2_100, 300, 200, 0),
])
def test_kmeans_runs_in_as_much_memory_as_ever(mr, n, d, k, precision, limit):
    """A budget, or an allocator's largest piece, of what a job needs at least."""
    import torch
    x, _, _ = synth.kmeans_points(n, d, 4, seed=n)
    init = x[np.random.default_rng(k).integers(0, n, k)].copy()
    room = _km_bytes(n, d, k, precision)
    if limit == "budget":
        ctx = mr.Context(hbm_budget=room)
    else:
        dev, stream = torch.cuda.current_device(), torch.cuda.current_stream().cuda_stream
        ctx = mr.Context(allocator=(
            lambda b: torch.cuda.caching_allocator_alloc(b, dev, stream) if b <= room else 0,
            torch.cuda.caching_allocator_delete))
    c2, a2, _ = _run_ctx(mr, ctx, _dev(x), init, 2, precision)
    ctx.close()
    # (the initial centroids hold equal ones, whose ties follow the last bit of
    # the first round's means: each round is compared from its own start)
    for _ in range(2):
        a_ref = oracle.kmeans_assign(x, init)
        c_ref, _ = oracle.kmeans_update(x, a_ref, init)
        init, a, _ = _run(mr, x, init, 1, precision)
        assert np.array_equal(a, a_ref)
        assert _rel_err(init, c_ref) <= TOL
    assert np.array_equal(a2, a) and np.array_equal(c2, init)


@pytest.mark.parametrize("n,d,k,comps,sigma,line", [
    (30_001, 64, 64, 8, 16.0, 4),     # window-sorted update, 8-byte loads
    (30_001, 21, 30, 4, 8.0, 4),      # one dimension per lane
    (30_001, 33, 64, 8, 16.0, 4),     # two dimensions per lane, 4-byte loads
    (12_001, 96, 16, 8, 4.0, 32),     # row-pipelined update
    (12_003, 67, 16, 8, 4.0, 32),     # plain local-array update
    (12_001, 130, 260, 8, 4.0, 8),    # sorted update
])
def test_kmeans_full_updates_and_updates_by_changes(mr, n, d, k, comps, sigma, line):
    """Rounds after the first on both sides of each update's line (n / line moved
    points): eight rounds in one call equal eight calls of one round, byte for
    byte."""
    x, _, _ = synth.kmeans_points(n, d, comps, seed=n + d, sigma=sigma)
    dx, cur = _dev(x), synth.kmeans_init(x, k, seed=n)
    c8, a8, _ = mr.kmeans(dx, _dev(cur), 8)
    moved, last = [], None
    for _ in range(8):
        cur, a, _ = mr.kmeans(dx, _dev(cur), 1)
        if last is not None:
            moved.append(int((a != last).sum()))
        last = a
    assert np.array_equal(a8, last) and np.array_equal(c8, cur)
    assert any(m > n // line for m in moved) and any(0 < m <= n // line for m in moved), moved


@pytest.mark.parametrize("n,d", [(500_009, 64), (450_001, 37)])
@pytest.mark.parametrize("precision", [0, 1])
def test_kmeans_skipped_points_not_16_byte_aligned(mr, n, d, precision):
    """The filter's list over points 4 bytes into a buffer, whose rows the
    converters load value by value: nine rounds in one call equal nine calls of
    one round, and the aligned points' result, byte for byte."""
    import torch
    x, _, _ = synth.kmeans_points(n, d, 100, seed=n + d)
    cur = synth.kmeans_init(x, 230, seed=n)
    buf = torch.zeros(x.size + 1, dtype=torch.float32, device="cuda")
    buf[1:] = torch.from_numpy(x.ravel()).cuda()
    off = buf[1:].view(n, d)
    torch.cuda.synchronize()
    c9, a9, _ = mr.kmeans(off, _dev(cur), 9, precision)
    ca, aa, _ = mr.kmeans(_dev(x), _dev(cur), 9, precision)
    for _ in range(9):
        cur, a, _ = mr.kmeans(off, _dev(cur), 1, precision)
    assert np.array_equal(a9, a) and np.array_equal(c9, cur)
    assert np.array_equal(aa, a) and np.array_equal(ca, cur)


@pytest.mark.parametrize("n,d,k,iters", [
    (400_003, 64, 256, 6),   # tensor-core pass, with the filter
    (100_003, 37, 100, 6),
    (60_001, 5, 17, 6),
    (30_001, 128, 512, 4),   # wide tensor-core pass
    (20_001, 256, 40, 4),
    (20_003, 9, 1_500, 4),
])
def test_kmeans_tensor_core_and_fp32_passes_agree(mr, n, d, k, iters):
    """The FP32 SIMT pass (which a context with a wait limit of its own keeps)
    against the tensor-core passes: the same bytes, since every assignment is the
    FP64 definition's and the sums are exact."""
    x, _, _ = synth.kmeans_points(n, d, 60, seed=n + d)
    init, dx = synth.kmeans_init(x, k, seed=n), _dev(x)
    with mr.Context() as ctx:
        ctx.set_option(mr.OPT_WAIT_POLLS, 1 << 20)
        before = ctx.kernel_launches
        c32, a32, _ = _run_ctx(mr, ctx, dx, init, iters, 0)
        simt = ctx.kernel_launches - before
    with mr.Context() as ctx:
        before = ctx.kernel_launches
        c, a, _ = _run_ctx(mr, ctx, dx, init, iters, 0)
        # (max |x| takes a kernel of its own only beside the SIMT pass)
        assert ctx.kernel_launches - before != simt
    assert np.array_equal(a, a32) and np.array_equal(c, c32)
    if d <= 64 and k <= 256:
        for precision in (1, 2):
            c, a, _ = mr.kmeans(dx, _dev(init), iters, precision)
            assert np.array_equal(a, a32) and np.array_equal(c, c32)


@pytest.mark.parametrize("n,d,k,limit", [
    (3_001, 257, 20, False),     # one dimension past the wide pass
    (2_003, 300, 300, False),    # SIMT pass with float selection, several threads' centroids in the settling
    (1_201, 1_024, 64, False),   # the most dimensions
    (1_024, 1_000, 257, False),
    (700, 513, 4_096, False),    # the most centroids
    (4_001, 16, 300, True),      # shapes of the wide pass, kept on the SIMT pass by a wait limit
    (4_001, 8, 3_000, True),
])
@pytest.mark.parametrize("offset", [0.0, 3e4])
def test_kmeans_fp32_simt_pass_and_settling(mr, n, d, k, limit, offset):
    """Shapes beyond the tensor-core passes: two rounds, each from the oracle's
    centroids.  The offset makes near ties of points that FP32 cannot tell."""
    x, _, _ = synth.kmeans_points(n, d, 16, seed=n + d)
    x = x + np.float32(offset)
    cur, dx = x[np.random.default_rng(k).integers(0, n, k)] + np.float32(0.125), _dev(x)
    with mr.Context() as ctx:
        if limit:
            ctx.set_option(mr.OPT_WAIT_POLLS, 1 << 20)
        for _ in range(2):
            a_ref = oracle.kmeans_assign(x, cur)
            c_ref, _ = oracle.kmeans_update(x, a_ref, cur)
            c, a, st = _run_ctx(mr, ctx, dx, cur, 1, 0)
            assert np.array_equal(a, a_ref)
            assert _rel_err(c, c_ref) <= TOL
            cur = c_ref


@pytest.mark.parametrize("n,d,k,rounds", [
    (400_003, 64, 200, 18),   # nearly every point listed for many rounds: the filter rests twice
    (400_009, 31, 60, 18),
    (393_216, 6, 250, 14),
])
@pytest.mark.parametrize("precision", [0, 2])
def test_kmeans_filter_at_rest(mr, n, d, k, rounds, precision):
    """Points without clusters: rounds with the filter, without it and its bounds,
    with the bounds alone, and with it again, in one call equal calls of one
    round, byte for byte."""
    x = np.random.default_rng(n + d).standard_normal((n, d), dtype=np.float32)
    dx, cur = _dev(x), synth.kmeans_init(x, k, seed=n)
    call, a_call, _ = mr.kmeans(dx, _dev(cur), rounds, precision)
    for _ in range(rounds):
        cur, a, _ = mr.kmeans(dx, _dev(cur), 1, precision)
    assert np.array_equal(a_call, a) and np.array_equal(call, cur)


@pytest.mark.parametrize("n,d,k", [(3_001, 16, 100), (2_000, 128, 300), (1_500, 300, 20), (1_203, 8, 2_000)])
def test_kmeans_points_that_are_many_centroids(mr, n, d, k):
    """Points that equal six and more of the centroids, others that tie among them,
    and some a least step away from one: the lowest index of a tie."""
    rng = np.random.default_rng(n)
    base = rng.normal(0, 1, (3, d)).astype(np.float32)
    init = base[rng.integers(0, 3, k)]
    init[k // 2] = rng.normal(0, 1, d)
    x = base[rng.integers(0, 3, n)].copy()
    x[::5] += rng.normal(0, 0.1, (len(x[::5]), d)).astype(np.float32)
    x[1::7, d - 1] = np.nextafter(x[1::7, d - 1], np.float32(9))
    x[2::7] *= np.float32(1e-22)
    init[-3:] = np.float32(0)
    init[-3:, 0] = np.float32(1e-22) * base[0, 0]
    a_ref = oracle.kmeans_assign(x, init)
    for precision in (0, 1):
        if precision and (d > 64 or k > 256):
            continue
        _, a, st = _run(mr, x, init, 1, precision)
        assert np.array_equal(a, a_ref)
        assert int(st[1]) > 0
