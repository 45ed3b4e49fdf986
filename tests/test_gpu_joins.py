"""Bucket joins (A4) on synthetic hashes against the bucket definition (the oracle): the one-hashmap
range join's segments and the joins' edges of tile, row and batch sizes."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2511_16576_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
T = 1 << 24


@pytest.fixture(scope="module")
def B():
    from paper_2511_16576_gb300 import binding
    binding.load()
    return binding


@pytest.fixture(scope="module")
def ctx(B):
    c = B.Context(0)
    yield c
    c.close()


def on_device(h, shift=0):
    """uint32 hashes on the device; shift = 1 puts the first row off a 16-byte boundary."""
    buf = torch.zeros(h.size + 4, dtype=torch.int32, device=DEV)
    out = buf[shift:shift + h.size].view(h.shape)
    out.copy_(torch.from_numpy(np.ascontiguousarray(h).view(np.int32)))
    return out


def hashes(rng, n, K, values):
    h = rng.integers(0, values, size=(n, K)).astype(np.uint32)
    h[rng.random(h.shape) < 0.05] = T
    return h


def check(B, ctx, orc, ph, qh, bands, shift=0):
    K = ph.shape[1]
    P = B.make_params(K, bands)
    index = B.lsh_build(ctx, on_device(ph), P)
    rp_ref, cand_ref = orc.candidates(qh, ph, bands, K // bands, T)
    q = on_device(qh, shift)
    for capacity in (None, int(rp_ref[-1])):  # counted and joined again; joined in one call
        row_ptr, cand = B.lsh_query(ctx, index, q, capacity=capacity)
        assert np.array_equal(row_ptr.cpu().numpy(), rp_ref)
        assert np.array_equal(cand.cpu().numpy(), cand_ref)
    index.close()
    return rp_ref


@pytest.mark.parametrize("K,values,n,Q", [
    (1, 3, 5000, 3),       # a third of the set per bucket, 512 segments a query
    (1, 1, 129, 2),        # every polygon in one bucket: 128 + 1 entries, one segment's tail
    (1, 1, 30_000, 100),   # more candidates than a call without a capacity makes room for
    (2, 4, 4097, 100),
    (3, 3, 20000, 37),
    (4, 2, 3000, 5000),    # 16-byte tuples, two segments per query
    (5, 2, 2000, 12000),   # one segment per query
    (8, 2, 1500, 64),
    (16, 1, 300, 7),       # tuples longer than the register form
])
@pytest.mark.parametrize("shift", [0, 1])
def test_one_hashmap(B, ctx, orc, K, values, n, Q, shift):
    rng = np.random.default_rng(K * 1000 + n)
    ph, qh = hashes(rng, n, K, values), hashes(rng, Q, K, values)
    qh[0] = T  # an invalid key: an empty row
    qh[-1, :] = 0
    rp = check(B, ctx, orc, ph, qh, 1, shift)
    assert rp[1] == 0 and rp[-1] > 0


def test_one_hashmap_in_the_query_graph(B, ctx):
    """The captured join (fixed buffers, a batch below the maximum) gives the plain call's rows."""
    w = synth.WORKLOADS["small"]
    db = synth.make_database(w)
    qs = synth.make_queries(w, db, 40)
    P = B.make_params(2, 1)
    up = lambda ps: (torch.from_numpy(ps.xy).to(DEV), torch.from_numpy(ps.offsets).to(DEV))
    h = B.minhash_sign(ctx, B.poly_upload(ctx, *up(db)), P)
    xy, off = up(qs)
    row_ptr, cand = B.lsh_query(ctx, (index := B.lsh_build(ctx, h, P)),
                                B.minhash_sign(ctx, B.poly_upload(ctx, xy, off), P))
    total = cand.numel()
    assert total > 0
    for cap in (total, total - 1):
        g = B.QueryGraph(ctx, index, 64, qs.xy.shape[0], cap, 8)
        g.run(xy, off)
        flags, got = g.status()
        assert got == total and flags == (0 if cap == total else 8)
        assert torch.equal(g.row_ptr[:qs.n + 1], row_ptr)
        assert cap < total or torch.equal(g.cand, cand)
        g.close()
    index.close()


@pytest.mark.parametrize("n,Q", [(1, 1), (63, 5), (64, 4), (129, 1), (4097, 9), (70_001, 3), (5000, 400)])
def test_bbox_join_segments(B, ctx, n, Q):
    """Box overlaps with positive area, ids ascending, for sets and batches around the edges of a
    segment (64 boxes), a query group (4) and a warp; empty boxes (beyond the domain) overlap nothing."""
    rng = np.random.default_rng(n + Q)

    def rects(k):
        c = rng.integers(-2000, 66_000, size=(k, 2))
        s = rng.integers(1, 6000, size=(k, 2))
        c[::50] += 100_000
        x0, y0, x1, y1 = c[:, 0], c[:, 1], c[:, 0] + s[:, 0], c[:, 1] + s[:, 1]
        xy = np.stack([x0, y0, x1, y0, x1, y1, x0, y1], 1).reshape(-1, 2).astype(np.int32)
        box = np.clip(np.stack([x0, y0, x1, y1], 1), 0, 65536)
        return B.poly_upload(ctx, torch.from_numpy(xy).to(DEV),
                             torch.arange(0, 4 * k + 1, 4, dtype=torch.int64, device=DEV)), box
    qp, qb = rects(Q)
    dbp, pb = rects(n)
    row_ptr, cand = B.bbox_join(ctx, qp, dbp)
    rp, cd = row_ptr.cpu().numpy(), cand.cpu().numpy()
    for q in range(Q):
        a = qb[q]
        exp = np.nonzero((a[0] < pb[:, 2]) & (pb[:, 0] < a[2]) & (a[1] < pb[:, 3]) & (pb[:, 1] < a[3]) &
                         (pb[:, 0] < pb[:, 2]) & (pb[:, 1] < pb[:, 3]))[0]
        assert np.array_equal(cd[rp[q]:rp[q + 1]], exp)


@pytest.mark.parametrize("K,bands,values,n,Q", [
    (4, 2, 2, 1, 1),            # one polygon: a single bit
    (4, 4, 3, 127, 9),          # around one 128-id vector, 16-byte rows
    (8, 2, 2, 128, 3),
    (6, 3, 2, 129, 700),        # more rows than resident blocks
    (8, 4, 1, 30_000, 100),     # more candidates than a call without a capacity makes room for
    (16, 2, 1, 300, 5),         # 8-hash tuples
    (36, 2, 1, 200, 4),         # tuples longer than the register form
    (32, 32, 40, 70_001, 20),   # one-hash bands: long rows with many duplicates
    (128, 64, 60, 5000, 33),
    (128, 128, 400, 30_000, 7), # every band slot in use
    (32, 8, 3, 403_000, 6),     # the last size of 256 threads, and the next two block sizes
    (32, 8, 3, 409_700, 6),
    (32, 8, 3, 852_100, 6),
    (16, 4, 5, 1 << 20, 5),     # the largest bitmap
    (16, 4, 5, (1 << 20) + 1, 5),    # the shared-memory set, few bands
    (16, 16, 90, (1 << 20) + 7, 5),  # its rows beyond 16,384 candidates (id-range passes)
])
@pytest.mark.parametrize("shift", [0, 1])
def test_banded_join(B, ctx, orc, K, bands, values, n, Q, shift):
    rng = np.random.default_rng(K * 1000 + n)
    ph, qh = hashes(rng, n, K, values), hashes(rng, Q, K, values)
    qh[0] = T
    qh[-1] = ph[n // 2]
    if Q > 2:
        ph[n // 3:n // 3 + min(n, 50)] = qh[1]
    rp = check(B, ctx, orc, ph, qh, bands, shift)
    assert rp[-1] > 0


@pytest.mark.parametrize("n,values", [(30_000, 3), (30_000, 9), (409_601, 3), (409_601, 9)])
def test_warp_join_and_what_it_leaves(B, ctx, orc, n, values):
    """Batches large enough for the warp join (1,024 queries, tuples of six): rows of no, a few, 128,
    129 and thousands of entries, the longer ones left to the bitmap or to the shared-memory set."""
    rng = np.random.default_rng(n + values)
    K, bands, Q = 96, 16, 1100
    ph, qh = hashes(rng, n, K, values), hashes(rng, Q, K, 1000)
    qh[:500:2] = ph[rng.integers(0, n, 250)]
    for q, copies in ((1, 8), (3, 9), (5, 300)):  # 128, 144 and 4,800 entries of one row
        qh[q] = 10_000 + q
        ph[rng.choice(n, copies, replace=False)] = qh[q]
    P = B.make_params(K, bands)
    index = B.lsh_build(ctx, on_device(ph), P)
    pick = np.concatenate([np.arange(8), rng.choice(Q, 24, replace=False)])
    rp_ref, cand_ref = orc.candidates(np.ascontiguousarray(qh[pick]), ph, bands, K // bands, T)
    full = None
    for capacity in (None, 1 << 22):
        row_ptr, cand = B.lsh_query(ctx, index, on_device(qh), capacity=capacity)
        rp, cd = row_ptr.cpu().numpy(), cand.cpu().numpy()
        for i, q in enumerate(pick):
            assert np.array_equal(cd[rp[q]:rp[q + 1]], cand_ref[rp_ref[i]:rp_ref[i + 1]]), q
        assert full is None or (np.array_equal(rp, full[0]) and np.array_equal(cd, full[1]))
        full = (rp, cd)
    # the fill alone, from the counted rows
    cand = torch.empty(len(full[1]), dtype=torch.int32, device=DEV)
    q = on_device(qh)
    B._check(B.load().pmh_lsh_query_fill(ctx.handle, index.handle, q.data_ptr(), Q, row_ptr.data_ptr(),
                                         cand.data_ptr(), cand.numel(), None))
    assert np.array_equal(cand.cpu().numpy(), full[1])
    index.close()


def taken(f):
    """Device bytes that a call took and kept."""
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    f()
    torch.cuda.synchronize()
    return free - torch.cuda.mem_get_info()[0]


def test_staging_memory(B, orc):
    """The staging pool holds no more than the capacity, and a join that stages nothing takes none, in a
    plain call and in a captured graph."""
    rng = np.random.default_rng(5)
    Q, slack = 16_384, 8 << 20
    for n, K, bands, pool in ((5000, 64, 8, 1 << 20), (409_601, 64, 8, 0)):
        ph, qh = hashes(rng, n, K, 500), hashes(rng, Q, K, 500)
        qh[:50] = ph[:50]
        c = B.Context(0)
        index = B.lsh_build(c, on_device(ph), B.make_params(K, bands))
        q = on_device(qh)
        row_ptr = torch.empty(Q + 1, dtype=torch.int64, device=DEV)
        cand = torch.empty(1 << 20, dtype=torch.int32, device=DEV)
        B.lsh_query(c, index, q[:8], capacity=8)  # (kernels loaded)
        out = []
        assert taken(lambda: out.append(B.lsh_query(c, index, q, capacity=1 << 20))) <= 5 * pool + slack
        rp_ref, cand_ref = orc.candidates(np.ascontiguousarray(qh[:100]), ph, bands, K // bands, T)
        assert np.array_equal(out[0][0].cpu().numpy()[:101], rp_ref)
        assert np.array_equal(out[0][1].cpu().numpy()[:rp_ref[-1]], cand_ref)
        if pool == 0:  # two result arrays of 6 bytes a candidate, no third of 4
            cap = 64 << 20
            g = []
            assert taken(lambda: g.append(B.QueryGraph(c, index, 64, 4096, cap, 8))) <= 6 * cap + 8 * slack
            g[0].close()
        index.close()
        c.close()


def rows_of(B, ctx, orc, ph, qh, bands, pick):
    """lsh_query of all queries, without and with a capacity; the picked rows against the oracle."""
    K = ph.shape[1]
    index = B.lsh_build(ctx, on_device(ph), B.make_params(K, bands))
    rp_ref, cand_ref = orc.candidates(np.ascontiguousarray(qh[pick]), ph, bands, K // bands, T)
    q, lengths = on_device(qh), None
    for capacity in (None, "total"):
        if capacity:
            capacity = int(rp[-1])
        row_ptr, cand = B.lsh_query(ctx, index, q, capacity=capacity)
        rp, cd = row_ptr.cpu().numpy(), cand.cpu().numpy()
        for i, p in enumerate(pick):
            assert np.array_equal(cd[rp[p]:rp[p + 1]], cand_ref[rp_ref[i]:rp_ref[i + 1]]), p
        assert lengths is None or np.array_equal(lengths, np.diff(rp))
        lengths = np.diff(rp)
    index.close()
    return lengths


@pytest.mark.parametrize("K,bands,n", [(8, 4, 409_601), (2, 2, 852_100), (4, 2, 1 << 20), (4, 2, (1 << 20) + 1),
                                       (32, 16, 1 << 20), (32, 16, (1 << 20) + 1), (16, 4, 409_600),
                                       (16, 4, 409_601)])
@pytest.mark.parametrize("Q", [5, 200, 800])
def test_largest_bitmaps(B, ctx, orc, K, bands, n, Q):
    """Tuples of one or two hashes up to 2^20 ids, longer ones up to 409,600, and the sets just above (merge
    and open-addressing set); batches that leave SMs a query, give them 512 threads, and reuse their
    bitmap for another row."""
    rng = np.random.default_rng(n + K)
    ph, qh = hashes(rng, n, K, 400 if K // bands <= 2 else 7), hashes(rng, Q, K, 400 if K // bands <= 2 else 7)
    qh[0] = T
    qh[1::3] = ph[rng.integers(0, n, len(qh[1::3]))]
    ph[[0, n - 1, n - 2, n // 2]] = qh[2]  # the first and last bits
    pick = np.unique(np.concatenate([np.arange(3), rng.integers(0, Q, 4), [Q - 1]]))
    lengths = rows_of(B, ctx, orc, ph, qh, bands, pick)
    assert lengths[0] == 0 and lengths[2] >= 4


@pytest.mark.parametrize("n", [409_600, 700_000])
def test_bitmaps_with_threads_by_fit(B, ctx, orc, n):
    """More queries than two per SM: the block's size follows from how many bitmaps fit an SM."""
    rng = np.random.default_rng(n)
    Q = 1200
    ph, qh = hashes(rng, n, 8, 300), hashes(rng, Q, 8, 300)
    assert rows_of(B, ctx, orc, ph, qh, 4, rng.choice(Q, 8, replace=False)).sum() > 0


def test_set_join_long_rows(B, ctx, orc):
    """Rows around the small set's 4,096 and the large set's 16,384 distinct ids, beyond them (id-range
    passes) and past the staging pool, on a set above the bitmap's limit."""
    rng = np.random.default_rng(9)
    n, K, bands = 420_000, 48, 16
    ph = rng.integers(1000, 1 << 20, (n, K)).astype(np.uint32)
    sizes = [1, 127, 128, 129, 4095, 4096, 4097, 16_383, 16_384, 16_385, 32_768, 40_000, 200_000]
    qh = rng.integers(1 << 21, 1 << 22, (len(sizes) + 1, K)).astype(np.uint32)
    for i, size in enumerate(sizes):  # each id in one or two of the query's bands
        ids = rng.choice(n, size, replace=False)
        for b in range(2):
            part = ids if b == 0 else ids[::3]
            j = (3 * i + b) % bands
            ph[part, 3 * j:3 * j + 3] = qh[i, 3 * j:3 * j + 3]
    lengths = rows_of(B, ctx, orc, ph, qh, bands, np.arange(len(qh)))
    assert lengths[-1] == 0 and lengths[4] <= 4096 < lengths[10] and lengths.max() > 100_000
    # past the pool: 4,096 ids per query of a batch of long rows
    many = np.repeat(qh[7:10], 3, axis=0)
    rows_of(B, ctx, orc, ph, many, bands, np.arange(len(many)))


@pytest.mark.parametrize("n", [30_000, 409_601])
def test_count_then_fill_without_a_capacity(B, ctx, orc, n):
    """The documented two calls: a count with capacity 0 (nothing staged; the warp join leaves rows to the
    next join), then the fill, or a second whole call."""
    rng = np.random.default_rng(n)
    K, bands, Q = 96, 16, 1100
    ph, qh = hashes(rng, n, K, 1000), hashes(rng, Q, K, 1000)
    qh[:400:2] = ph[rng.integers(0, n, 200)]
    for q, copies in ((1, 8), (3, 9), (5, 300)):  # 128, 144 and 4,800 entries of one row
        qh[q] = 10_000 + q
        ph[rng.choice(n, copies, replace=False)] = qh[q]
    pick = np.concatenate([np.arange(8), rng.choice(Q, 12, replace=False)])
    rp_ref, cand_ref = orc.candidates(np.ascontiguousarray(qh[pick]), ph, bands, K // bands, T)
    index = B.lsh_build(ctx, on_device(ph), B.make_params(K, bands))
    q = on_device(qh)
    lib = B.load()
    row_ptr = torch.empty(Q + 1, dtype=torch.int64, device=DEV)
    total = ctypes.c_int64()
    call = lambda cand, cap: lib.pmh_lsh_query(ctx.handle, index.handle, q.data_ptr(), Q, row_ptr.data_ptr(), cand, cap,
                                               ctypes.byref(total), torch.cuda.current_stream().cuda_stream)
    assert call(None, 0) == B.PMH_ERR_CAPACITY and total.value > 0
    rp = row_ptr.cpu().numpy()
    assert rp[-1] == total.value
    for again in (False, True):
        cand = torch.full((total.value,), -1, dtype=torch.int32, device=DEV)
        if again:
            assert call(cand.data_ptr(), total.value) == 0
        else:
            B._check(lib.pmh_lsh_query_fill(ctx.handle, index.handle, q.data_ptr(), Q, row_ptr.data_ptr(),
                                            cand.data_ptr(), total.value, torch.cuda.current_stream().cuda_stream))
        cd = cand.cpu().numpy()
        for i, p in enumerate(pick):
            assert np.array_equal(cd[rp[p]:rp[p + 1]], cand_ref[rp_ref[i]:rp_ref[i + 1]]), p
    index.close()


@pytest.mark.parametrize("K,bands,n", [(8, 4, 30_000), (12, 4, 200_000), (4, 2, 600_000)])
@pytest.mark.parametrize("Q", [255, 256, 5000])
def test_rows_of_few_bands(B, ctx, orc, K, bands, n, Q):
    """Batches around the warp join's, most rows of a candidate or none, some of 100 to 10,000 entries (left
    to the bitmap), and a block whose last rows are such."""
    rng = np.random.default_rng(n + Q)
    rows = K // bands
    ph, qh = hashes(rng, n, K, int(n ** (1 / rows)) * 3), hashes(rng, Q, K, int(n ** (1 / rows)) * 3)
    long = np.unique(np.concatenate([rng.choice(Q, 9, replace=False), [Q - 1, Q - 2]]))
    for i, q in enumerate(long):
        qh[q] = (1 << 22) + 7 * q
        ph[rng.choice(n, 60 + 1000 * i, replace=False), :rows] = qh[q, :rows]
    lengths = rows_of(B, ctx, orc, ph, qh, bands, np.concatenate([long, rng.choice(Q, 8, replace=False)]))
    assert lengths[long].max() > 5000 and np.median(lengths) < 10


def test_few_bands_in_the_query_graph(B, ctx):
    """The captured joins of a batch that takes the warp join, dense and sparse rows: the plain call's rows."""
    db = synth.star_polygons(3000, 3, n_range=(8, 40), f_range=(1e-4, 2e-1))
    qs = synth.perturbed_queries(db, 300, 5)
    P = B.make_params(8, 4, 1 << 22)
    up = lambda ps: (torch.from_numpy(ps.xy).to(DEV), torch.from_numpy(ps.offsets).to(DEV))
    h = B.minhash_sign(ctx, B.poly_upload(ctx, *up(db)), P)
    index = B.lsh_build(ctx, h, P)
    xy, off = up(qs)
    row_ptr, cand = B.lsh_query(ctx, index, B.minhash_sign(ctx, B.poly_upload(ctx, xy, off), P))
    total = cand.numel()
    assert total > 0
    for cap in (total, total - 1):
        g = B.QueryGraph(ctx, index, 400, xy.shape[0] + 9, cap, 8)
        g.run(xy, off)
        assert g.status() == (0 if cap == total else 8, total)
        assert torch.equal(g.row_ptr[:qs.n + 1], row_ptr) and int(g.row_ptr[400]) == total
        assert cap < total or torch.equal(g.cand, cand)
        g.close()
    index.close()
