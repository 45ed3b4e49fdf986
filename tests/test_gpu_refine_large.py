"""Exact Jaccard (A8) of pairs with a ring above 1,024 vertices (a block per pair, the sets' y-slab
index) against the oracle: degenerate contacts, rings with and without a slab index, batches of
mixed sizes, refined lists and the query graph."""
import numpy as np
import pytest
import torch

from paper_2511_16576_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


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


def upload(B, ctx, polys):
    xy = np.concatenate([np.asarray(p, np.int32).reshape(-1, 2) for p in polys])
    off = np.concatenate([[0], np.cumsum([len(p) for p in polys])]).astype(np.int64)
    return B.poly_upload(ctx, torch.from_numpy(xy).to(DEV), torch.from_numpy(off).to(DEV))


def comb(teeth, dx=0, dy=0, swap=False, reverse=False):
    """A comb of 4 * teeth + 2 vertices: horizontal edges on every tooth, long vertical ones."""
    pts = [[1000, 1000]]
    for i in range(teeth):
        x = 1000 + 20 * i
        pts += [[x, 3000], [x + 10, 3000], [x + 10, 1200], [x + 20, 1200]]
    pts += [[1000 + 20 * teeth, 1000]]
    p = np.array(pts) + [dx, dy]
    if swap:
        p = p[:, ::-1]
    return p[::-1] if reverse else p


def ngon(n, r, cx, cy):
    t = np.arange(n) * 2 * np.pi / n
    return np.stack([np.rint(cx + r * np.cos(t)), np.rint(cy + r * np.sin(t))], 1)


A_COMB = comb(300)
FRACTAL = synth.star_polygons(2, 29, (3000, 3000), "uniform", (1e-2, 2e-2), fractal=True)
PAIRS = {
    "same": (A_COMB, A_COMB),
    "same, other orientation": (A_COMB, comb(300, reverse=True)),
    "one tooth on": (A_COMB, comb(300, 20)),
    "teeth sharing edges": (A_COMB, comb(300, 10)),
    "rows on vertices": (A_COMB, comb(300, 5, 200)),
    "one row up": (A_COMB, comb(290, 0, 1)),
    "crossing combs": (A_COMB, comb(300, swap=True)),
    "square in the comb's gap": (A_COMB, [[1010, 1200], [1020, 1200], [1020, 2000], [1010, 2000]]),
    "square over teeth": ([[900, 2000], [2000, 2000], [2000, 3000], [900, 3000]], A_COMB),
    "tall triangle": ([[1500, 0], [1600, 60000], [1400, 60000]], A_COMB),
    "touching tops": (A_COMB, comb(300, 0, 2000)),
    "regular polygons": (ngon(1100, 9000, 30000, 30000), ngon(2500, 9000, 33000, 30001)),
    "small ring with lists that overflow": (comb(255), comb(300, 3, 3)),
    "fractals": (FRACTAL.poly(0), FRACTAL.poly(1) + (FRACTAL.centre[0] - FRACTAL.centre[1]).astype(np.int32)),
    "inside": (ngon(1200, 20000, 30000, 30000), FRACTAL.poly(0) // 8 + 25000),
}


def test_large_pairs_match_the_oracle(B, ctx, orc):
    names = list(PAIRS)
    qa, pb = upload(B, ctx, [PAIRS[n][0] for n in names]), upload(B, ctx, [PAIRS[n][1] for n in names])
    idx = torch.arange(len(names), dtype=torch.int32, device=DEV)
    j = B.pair_jaccard(ctx, qa, pb, idx, idx)
    swapped = B.pair_jaccard(ctx, pb, qa, idx, idx)
    assert torch.equal(j, B.pair_jaccard(ctx, qa, pb, idx, idx))  # sums do not depend on their order
    for e, n in enumerate(names):
        a, b = (np.ascontiguousarray(p, np.int32) for p in PAIRS[n])
        ref = orc.jaccard(a, b)
        assert abs(j[e].item() - ref) <= 1e-12 + 1e-9 * ref, (n, j[e].item(), ref)
        assert abs(swapped[e].item() - ref) <= 1e-12 + 1e-9 * ref, (n, swapped[e].item(), ref)


def test_reloaded_set_under_a_graph(B, ctx, orc):
    """A graph that refines large rings reads the slab lists of the set as reloaded since its
    capture, and gives what refine_topk gives."""
    def sets(seed):
        return synth.star_polygons(60, seed, (1200, 1200), "uniform", (1e-2, 2e-2), fractal=True)
    first, second = sets(51), sets(52)
    n = min(first.n_vertices, second.n_vertices)
    assert abs(first.n_vertices - second.n_vertices) < 0.2 * n

    def padded(ps, total):  # the same vertex count: repeat the last polygon's last vertices
        pad = np.repeat(ps.xy[-1:], total - ps.n_vertices, axis=0)
        off = ps.offsets.copy()
        off[-1] = total
        return torch.from_numpy(np.concatenate([ps.xy, pad])).to(DEV), torch.from_numpy(off).to(DEV)
    total = max(first.n_vertices, second.n_vertices)
    P = B.make_params(32, 1, flags=0)
    xy, off = padded(first, total)
    dbp = B.poly_upload(ctx, xy, off)
    index = B.lsh_build(ctx, B.minhash_sign(ctx, dbp, P), B.make_params(32, 32))
    qs = synth.perturbed_queries(second, 12, 53)
    qxy, qoff = torch.from_numpy(qs.xy).to(DEV), torch.from_numpy(qs.offsets).to(DEV)
    g = B.QueryGraph(ctx, index, qs.n, qs.xy.shape[0], 4096, 8, db=dbp, k=4)
    xy, off = padded(second, total)
    B.poly_reload(dbp, xy, off)
    B.lsh_rebuild(ctx, index, B.minhash_sign(ctx, dbp, P))
    g.run(qxy, qoff)
    assert g.status()[0] == 0
    ids, j = B.refine_topk(ctx, B.poly_upload(ctx, qxy, qoff), dbp, g.top_ids, g.top_n, 4)
    assert torch.equal(ids, g.ref_ids) and torch.equal(j, g.ref_j)
    for q in range(qs.n):
        p = int(ids[q, 0])
        assert p >= 0 and abs(j[q, 0].item() - orc.jaccard(qs.poly(q), second.poly(p))) <= 1e-9
    g.close()
    index.close()
