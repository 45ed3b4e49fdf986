"""Bucket joins (A4) on synthetic hashes against the bucket definition (the oracle): the one-hashmap
range join's segments and the joins' edges of tile, row and batch sizes."""
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
