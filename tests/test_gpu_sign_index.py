"""Signing through the stream index (A1): the counter-free kernels that production calls run against
the counting build (which the other tests run) and the oracle, over the forms of the index."""
import numpy as np
import pytest
import torch

from paper_2511_16576_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
SEED = 0x5EED


@pytest.fixture(scope="module")
def B():
    from paper_2511_16576_gb300 import binding
    binding.load()
    return binding


# every cell crossed by the boundary (finest grid, two passes) / most cells inside / spiky rings
# with long slab lists / rings above 256 and above 4,096 vertices
SHAPES = {
    "smallest": dict(n=20_000, n_range=(4, 40), n_dist="loguniform", f_range=(1e-5, 5e-5)),
    "combined": dict(n=20_000, n_range=(8, 1024), n_dist="loguniform", f_range=(1e-5, 1e-2), fractal=True,
                     comonotone=True),
    "stars": dict(n=8000, n_range=(16, 256), n_dist="loguniform", f_range=(1e-4, 1e-2)),
    "large": dict(n=300, n_range=(200, 20_000), n_dist="loguniform", f_range=(1e-3, 1e-1), fractal=True,
                  comonotone=True),
}


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("K", [128, 3, 37, 300])
def test_production_hashes(B, orc, shape, K):
    kw = dict(SHAPES[shape])
    n = max(64, kw.pop("n") * 32 // max(K, 32))
    db = synth.star_polygons(n, 61 + K, **kw)
    ctx = B.Context(0)
    P = B.make_params(K, 1, 1 << 24, SEED, flags=B.FLAG_STREAM_INDEX)
    polys = B.poly_upload(ctx, torch.from_numpy(db.xy).to(DEV), torch.from_numpy(db.offsets).to(DEV))
    counted = B.minhash_sign(ctx, polys, P)
    B.sign_count_work(ctx, False)
    for _ in range(3):
        assert torch.equal(B.minhash_sign(ctx, polys, P), counted)
    rows = np.unique(np.concatenate([np.argsort(np.diff(db.offsets))[-2:],
                                     np.random.default_rng(K).choice(db.n, 24, replace=False)]))
    sub = db.subset(rows)
    ref = orc.sign(sub.xy, sub.offsets, SEED, K, 1 << 24, nthreads=16)
    assert np.array_equal(counted[torch.from_numpy(rows).to(DEV)].cpu().numpy().view(np.uint32), ref)
    ctx.close()


@pytest.mark.parametrize("K", [1, 2, 12, 13])
def test_few_hashes(B, orc, K):
    """Large polygons of few hashes: walked or indexed by their area, staged or not."""
    ctx = B.Context(0)
    B.sign_count_work(ctx, False)
    P = B.make_params(K, 1, 1 << 22, SEED, flags=B.FLAG_STREAM_INDEX)
    for n_range in ((3, 40), (250, 600)):
        db = synth.star_polygons(1500, 9 + K, n_range=n_range, n_dist="loguniform", f_range=(1e-4, 0.1))
        polys = B.poly_upload(ctx, torch.from_numpy(db.xy).to(DEV), torch.from_numpy(db.offsets).to(DEV))
        got = B.minhash_sign(ctx, polys, P).cpu().numpy().view(np.uint32)
        assert np.array_equal(got, orc.sign(db.xy, db.offsets, SEED, K, 1 << 22, nthreads=16))
    ctx.close()


def _strips(n, length, seed):
    """Thin slanted strips of 4 to 300 vertices and widths from nothing (no lattice point) to 60."""
    rng = np.random.default_rng(seed)
    rings = []
    for i in range(n):
        h = int(rng.choice([2, 4, 32, 40, 150]))
        a, w = rng.uniform(0.2, 1.3), rng.choice([0.3, 2.0, 8.0, 60.0])
        d, t = np.array([np.cos(a), np.sin(a)]), np.linspace(0, length, h)[:, None]
        o = rng.uniform(1000, 64000 - length, 2)
        side = np.array([-d[1], d[0]]) * w * (0.5 + np.sin(np.pi * t / length))
        rings.append(np.rint(np.concatenate([o + d * t + side / 2, (o + d * t - side / 2)[::-1]])))
    off = np.concatenate([[0], np.cumsum([len(r) for r in rings])]).astype(np.int64)
    return np.concatenate(rings).astype(np.int32), off


@pytest.mark.parametrize("n,K,T", [(300, 256, 6000), (5000, 33, 3000), (9000, 130, 1500), (40, 128, 9000)])
@pytest.mark.parametrize("count", [True, False])
def test_more_leftover_walks_than_the_queue_holds(orc, n, K, T, count):
    """Thin polygons under large boxes: 70,000 to a million hashes without a point of the level's (the
    last set: fewer than the queue holds), through the plain call and a captured graph."""
    from paper_2511_16576_gb300 import binding as B
    ctx = B.Context(0)
    B.sign_count_work(ctx, count)
    P = B.make_params(K, 1, T, 0x5EED, flags=B.FLAG_STREAM_INDEX)
    xy, off = _strips(n, 20_000, n)
    up = [torch.from_numpy(a).to(DEV) for a in (xy, off)]
    polys = B.poly_upload(ctx, *up)
    ref = orc.sign(xy, off, 0x5EED, K, T, nthreads=16)
    assert (ref == T).any() and (ref < T).any()
    h = B.minhash_sign(ctx, polys, P)
    assert np.array_equal(h.cpu().numpy().view(np.uint32), ref)
    index = B.lsh_build(ctx, h, P)
    g = B.QueryGraph(ctx, index, max_queries=n + 7, max_vertices=xy.shape[0], cand_capacity=1 << 20, m=4)
    g.run(*up)
    assert np.array_equal(g.hashes[:n].cpu().numpy().view(np.uint32).reshape(n, K), ref)
    g.close()
    ctx.close()


@pytest.mark.parametrize("K", [1, 2, 3, 8, 9, 31, 32, 33])
@pytest.mark.parametrize("count", [True, False])
def test_few_hashes(orc, K, count):
    """Polygons of every size and area around the forms of few hashes (walked briefly or through the index,
    staged or larger rings), and their queries through a captured graph."""
    from paper_2511_16576_gb300 import binding as B
    ctx = B.Context(0)
    B.sign_count_work(ctx, count)
    T = 1 << 20
    P = B.make_params(K, 1, T, SEED, flags=B.FLAG_STREAM_INDEX)
    parts = [synth.star_polygons(n, 40 + i, n_range=r, n_dist="loguniform", f_range=f)
             for i, (n, r, f) in enumerate([(300, (3, 60), (1e-2, 2e-1)), (300, (200, 300), (1e-4, 1e-1)),
                                            (200, (4, 256), (1e-5, 1e-3)), (30, (3000, 9000), (1e-3, 1e-1))])]
    far = np.array([[70_000, 70_000], [70_009, 70_000], [70_000, 70_009]], np.int32)  # no lattice point
    xy = np.concatenate([p.xy for p in parts] + [far])
    sizes = np.concatenate([np.diff(p.offsets) for p in parts] + [[3]])
    order = np.random.default_rng(K).permutation(len(sizes))
    first = np.concatenate([[0], np.cumsum(sizes)])
    xy = np.ascontiguousarray(np.concatenate([xy[first[i]:first[i] + sizes[i]] for i in order]))
    off = np.concatenate([[0], np.cumsum(sizes[order])]).astype(np.int64)
    ref = orc.sign(xy, off, SEED, K, T, nthreads=16)
    up = [torch.from_numpy(a).to(DEV) for a in (xy, off)]
    h = B.minhash_sign(ctx, B.poly_upload(ctx, *up), P)
    assert np.array_equal(h.cpu().numpy().view(np.uint32), ref)
    n = len(sizes)
    g = B.QueryGraph(ctx, B.lsh_build(ctx, h, P), n + 3, xy.shape[0], 1 << 21, 4)
    g.run(*up)
    assert np.array_equal(g.hashes[:n].cpu().numpy().view(np.uint32).reshape(n, K), ref)
    g.close()
    ctx.close()


@pytest.mark.parametrize("K,f,T", [(40, (2e-5, 2.1e-5), 1 << 20), (40, (1e-4, 1e-3), 1 << 20), (33, (1e-3, 2e-1), 1 << 20),
                                   (40, (1e-6, 3e-6), 1 << 17), (2050, (2e-4, 1e-3), 1 << 16)])
def test_index_with_coverage_masks(orc, K, f, T):
    """Rings above the staged size through the index and the masks: limits of every level that the form
    reads (and, at K = 2,050, without the finest)."""
    from paper_2511_16576_gb300 import binding as B
    ctx = B.Context(0)
    db = synth.star_polygons(60 if K < 2000 else 8, 21, n_range=(257, 1500), n_dist="loguniform", f_range=f)
    P = B.make_params(K, 1, T, SEED, flags=B.FLAG_STREAM_INDEX | B.FLAG_COVERAGE_MASK)
    polys = B.poly_upload(ctx, torch.from_numpy(db.xy).to(DEV), torch.from_numpy(db.offsets).to(DEV))
    h = B.minhash_sign(ctx, polys, P).cpu().numpy().view(np.uint32)
    assert np.array_equal(h, orc.sign(db.xy, db.offsets, SEED, K, T, nthreads=16))
    if K < 2000 and 1e-5 < f[0] < 1e-3:  # (the others walk: larger ones by cost, smaller ones past the index)
        assert B.sign_work(ctx)["walk_points"] < 0.2 * h.astype(np.int64).sum()
    ctx.close()
