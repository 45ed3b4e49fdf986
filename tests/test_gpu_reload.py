"""Upload and reload (A0): the fused copy, preparation and slab sizes, and slab lists that keep
their buffers, at the edges of a round of vertices, of the shared counters and of alignment."""
import numpy as np
import pytest
import torch

from paper_2511_16576_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
SEED, T, K = 0x5EED, 1 << 22, 8
SIZES = [3, 31, 32, 33, 127, 128, 129, 255, 256, 257, 300, 2047, 2048, 2052, 2056, 5000, 64, 9001]


def _sets():
    """Three sets of the same sizes: stars, rings whose edges cross most of their slabs (lists
    many times as long), and the stars again, shifted."""
    off = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
    rng = np.random.default_rng(3)
    star, tall = [], []
    for n in SIZES:
        a = np.sort(rng.uniform(0, 2 * np.pi, n))
        r = rng.uniform(3000, 9000, n)
        star.append(np.stack([20000 + r * np.cos(a), 30000 + r * np.sin(a)], 1))
        y = np.where(np.arange(n) % 2 == 0, rng.integers(9000, 12000, n), rng.integers(40000, 50000, n))
        tall.append(np.stack([10000 + np.arange(n) * 4, y], 1))
    star = np.rint(np.concatenate(star)).astype(np.int32)
    return off, star, np.concatenate(tall).astype(np.int32), star + 1500


@pytest.fixture(scope="module")
def B():
    from paper_2511_16576_gb300 import binding
    binding.load()
    return binding


def _dev(xy, odd):
    """[n, 2] on the device, 4 bytes off an 8-byte boundary if odd."""
    flat = torch.empty(xy.size + 2, dtype=torch.int32, device=DEV)
    v = flat[1:1 + xy.size] if odd else flat[:xy.size]
    v.copy_(torch.from_numpy(xy).reshape(-1))
    return v.view(-1, 2)


def _check(B, ctx, orc, polys, xy, off):
    bbox, area2 = polys.prep()
    bbox, area2 = bbox.cpu().numpy(), area2.cpu().numpy()
    for p, (b, e) in enumerate(zip(off[:-1], off[1:])):
        v = xy[b:e].astype(np.int64)
        w = np.roll(v, -1, 0)
        assert area2[p] == (v[:, 0] * w[:, 1] - w[:, 0] * v[:, 1]).sum()
        lo, hi = np.maximum(v.min(0), 0), np.minimum(v.max(0), 65536)
        assert list(bbox[p]) == [lo[0], lo[1], max(hi[0], lo[0]), max(hi[1], lo[1])]
    ref = orc.sign(xy, off, SEED, K, T, nthreads=16)
    for flags in (0, B.FLAG_STREAM_INDEX):
        P = B.make_params(K, 1, T, SEED, flags=flags)
        assert np.array_equal(B.minhash_sign(ctx, polys, P).cpu().numpy().view(np.uint32), ref)


@pytest.mark.parametrize("where", ["device", "odd", "host"])
def test_reload(B, orc, where):
    off, *sets = _sets()
    ctx = B.Context(0)

    def put(xy):
        if where == "host":
            return torch.from_numpy(xy).pin_memory(), torch.from_numpy(off).pin_memory()
        return _dev(xy, where == "odd"), torch.from_numpy(off).to(DEV)

    polys = (B.poly_upload_pinned if where == "host" else B.poly_upload)(ctx, *put(sets[0]))
    _check(B, ctx, orc, polys, sets[0], off)
    for xy in sets[1:]:
        B.poly_reload(polys, *put(xy))
        _check(B, ctx, orc, polys, xy, off)
    far = sets[0].copy()
    far[-1, 1] = (1 << 20) + 1
    with pytest.raises(Exception):
        B.poly_reload(polys, *put(far))
    B.poly_reload(polys, *put(sets[1]))
    _check(B, ctx, orc, polys, sets[1], off)
    ctx.close()


def test_class_order_of_many(B, orc):
    """Sets of one, two and a few thousand polygons over the three signing classes."""
    ctx = B.Context(0)
    for n, rng_ in ((1, (3, 9)), (2, (3000, 9000)), (3000, (4, 600))):
        db = synth.star_polygons(n, 5, n_range=rng_, n_dist="loguniform", f_range=(1e-4, 1e-2))
        polys = B.poly_upload(ctx, torch.from_numpy(db.xy).to(DEV), torch.from_numpy(db.offsets).to(DEV))
        P = B.make_params(K, 1, T, SEED, flags=B.FLAG_STREAM_INDEX)
        got = B.minhash_sign(ctx, polys, P).cpu().numpy().view(np.uint32)
        assert np.array_equal(got, orc.sign(db.xy, db.offsets, SEED, K, T, nthreads=16))
    ctx.close()


def _star(n, cx, cy, r, seed):
    rng = np.random.default_rng(seed)
    a = (np.arange(n) + rng.uniform(0.1, 0.9, n)) * (2 * np.pi / n)
    rad = r * rng.uniform(0.8, 1.2, n)
    return np.rint(np.stack([cx + rad * np.cos(a), cy + rad * np.sin(a)], 1)).astype(np.int32)


def test_graph_on_a_set_reloaded_with_large_rings(B):
    """A graph captured while every ring is small refines a reloaded set's large rings by the launches that
    a graph captured on them takes, to the plain call's values; and leaves them out again."""
    small = [600] * 8
    large = [3000] + [257] * 6 + [258]
    assert sum(small) == sum(large)
    rings = lambda sizes: np.concatenate([_star(n, 20000 + 1500 * i, 30000 - 900 * i, 9000, i)
                                          for i, n in enumerate(sizes)])
    off = lambda sizes: np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    ctx = B.Context(0)
    P = B.make_params(32, 16, 1 << 16, SEED)
    up = lambda xy, o: (torch.from_numpy(xy).to(DEV), torch.from_numpy(o).to(DEV))
    sets = [up(rings(s), off(s)) for s in (small, large)]
    polys = B.poly_upload(ctx, *sets[0])
    index = B.lsh_build(ctx, B.minhash_sign(ctx, polys, P), P)
    q = up(rings(small)[:600], off(small[:1]))
    qp = B.poly_upload(ctx, *q)

    def graph():
        return B.QueryGraph(ctx, index, 1, 900, 4096, 8, db=polys, k=8)

    def replay(g):
        before = B.launch_count()
        g.run(*q)
        launches = B.launch_count() - before
        assert g.status()[0] == 0
        n = int(g.top_n[0])
        assert n > 0
        ids = g.ref_ids[0, :n]
        j = B.pair_jaccard(ctx, qp, polys, torch.zeros(n, dtype=torch.int32, device=DEV), ids.contiguous())
        assert torch.equal(g.ref_j[0, :n], j)
        return launches

    g = graph()
    launches = []
    for s in (0, 1, 0, 1):
        if launches:
            B.poly_reload(polys, *sets[s])
        fresh = graph()
        launches.append((replay(g), replay(fresh)))
        fresh.close()
    assert all(a == b for a, b in launches), launches
    assert launches[0][0] == launches[2][0] == launches[1][0] - 1 == launches[3][0] - 1
    g.close()
    ctx.close()


def test_first_slab_index_by_a_reload(B, orc):
    """A set uploaded without a ring of the slab index's size, reloaded with some, and without again."""
    sizes = [[200, 250, 150, 200], [500, 100, 80, 120], [200, 250, 150, 200]]
    ctx = B.Context(0)
    polys = None
    for k, s in enumerate(sizes):
        xy = np.concatenate([_star(n, 9000 + 12000 * i, 30000, 8000, 10 * k + i) for i, n in enumerate(s)])
        off = np.concatenate([[0], np.cumsum(s)]).astype(np.int64)
        arrays = torch.from_numpy(xy).to(DEV), torch.from_numpy(off).to(DEV)
        if polys is None:
            polys = B.poly_upload(ctx, *arrays)
        else:
            B.poly_reload(polys, *arrays)
        _check(B, ctx, orc, polys, xy, off)
    ctx.close()
