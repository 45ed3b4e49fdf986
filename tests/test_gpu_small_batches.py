"""Captured batches of a few queries (A9): staged polygons signed by their 32-hash chunks when the
batch leaves warps idle, whole when it does not, against the oracle."""
import numpy as np
import pytest
import torch

from paper_2511_16576_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
T, SEED = 1 << 24, 0x5EED


@pytest.mark.parametrize("K", [32, 33, 128, 200])
@pytest.mark.parametrize("maxq", [1, 5, 3000])
def test_hashes(orc, K, maxq):
    from paper_2511_16576_gb300 import binding as B
    ctx = B.Context(0)
    P = B.make_params(K, 1, T, SEED, flags=B.FLAG_STREAM_INDEX)
    db = synth.star_polygons(200, 3, n_range=(3, 300), f_range=(1e-4, 1e-2))
    up = [torch.from_numpy(a).to(DEV) for a in (db.xy, db.offsets)]
    polys = B.poly_upload(ctx, *up)
    index = B.lsh_build(ctx, B.minhash_sign(ctx, polys, P), P)
    g = B.QueryGraph(ctx, index, max_queries=maxq, max_vertices=300 * maxq, cand_capacity=1 << 22, m=4)
    try:
        for n, sizes in ((1, (3, 5)), (min(5, maxq), (250, 262)), (maxq, (3, 280))):
            qs = synth.star_polygons(n, 11 + n, n_range=sizes, f_range=(1e-4, 1e-2))
            g.run(torch.from_numpy(qs.xy).to(DEV), torch.from_numpy(qs.offsets).to(DEV))
            assert g.status()[0] == 0
            rows = np.unique(np.linspace(0, n - 1, 40).astype(int))
            sub = qs.subset(rows)
            ref = orc.sign(sub.xy, sub.offsets, SEED, K, T, nthreads=16)
            assert np.array_equal(g.hashes[:n].cpu().numpy().view(np.uint32).reshape(n, K)[rows], ref)
    finally:
        g.close()
        ctx.close()


def test_graph_refuses_a_rebuilt_stream_index():
    """The index rebuilt for another seed and the same K (buffers of the same sizes, whose addresses may
    come back): the graph captured on the first one is refused, also after a rebuild for its own seed."""
    from paper_2511_16576_gb300 import binding as B
    db = synth.star_polygons(300, 3, f_range=(1e-3, 1e-2))
    up = lambda ps: (torch.from_numpy(ps.xy).to(DEV), torch.from_numpy(ps.offsets).to(DEV))
    ctx = B.Context(0)
    P = [B.make_params(32, 8, 1 << 22, seed, 5, B.FLAG_STREAM_INDEX) for seed in (11, 12)]
    index = B.lsh_build(ctx, B.minhash_sign(ctx, B.poly_upload(ctx, *up(db)), P[0]), P[0])
    xy, off = up(db.subset(np.arange(4)))
    g = B.QueryGraph(ctx, index, 4, xy.shape[0], 4096, 4)
    g.run(xy, off)
    first = g.hashes[:4].clone()
    for p in (P[1], P[0]):
        B.stream_index_build(ctx, p)
        with pytest.raises(B.PmhError) as e:
            g.run(xy, off)
        assert e.value.code == -6  # PMH_ERR_STATE
    g.close()
    g = B.QueryGraph(ctx, index, 4, xy.shape[0], 4096, 4)
    g.run(xy, off)
    assert torch.equal(g.hashes[:4], first)
    g.close()
    ctx.close()
