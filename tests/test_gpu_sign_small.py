"""Signing of small sets (A1): items of fewer hashes, rings at the edge of the one that is tested
whole, hashes inside and beyond the first 128 stream points, against the oracle."""
import numpy as np
import pytest
import torch

from paper_2511_16576_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
SEED = 0x5EED


@pytest.mark.parametrize("n", [1, 40, 1500])
@pytest.mark.parametrize("K", [1, 5, 32, 37])
def test_small_sets(orc, n, K):
    from paper_2511_16576_gb300 import binding as B
    parts = [synth.star_polygons(n, 7 + K, n_range=r, f_range=f)
             for r, f in (((63, 66), (1e-2, 0.1)), ((3, 12), (1e-4, 1e-2)), ((250, 260), (1e-3, 1e-1)))]
    ctx = B.Context(0)
    for db in parts:
        ref = orc.sign(db.xy, db.offsets, SEED, K, 1 << 22, nthreads=16)
        for T in (1 << 22, 100, 200):  # a T that ends inside the first 128 points, one just after
            want = np.minimum(ref, T) if T < (1 << 22) else ref
            P = B.make_params(K, 1, T, SEED)
            polys = B.poly_upload(ctx, torch.from_numpy(db.xy).to(DEV), torch.from_numpy(db.offsets).to(DEV))
            for count in (True, False):
                B.sign_count_work(ctx, count)
                got = B.minhash_sign(ctx, polys, P).cpu().numpy().view(np.uint32)
                assert np.array_equal(got, want)
    ctx.close()
