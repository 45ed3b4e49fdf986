"""Agreement counts and band bits (A5) over the forms of a row: lengths, band widths, not-found
hashes, empty rows, and batches from one pair to many."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
T = 1000


@pytest.mark.parametrize("K,bands", [(128, 1), (128, 2), (128, 4), (128, 8), (128, 16), (128, 32), (128, 64),
                                     (128, 128), (96, 32), (96, 12), (4, 1), (4, 4), (32, 16), (36, 9), (60, 20),
                                     (30, 10), (132, 33), (256, 32)])
@pytest.mark.parametrize("Q,most", [(1, 1), (1, 33), (3, 9), (700, 60), (2000, 700)])
def test_counts_and_bands(K, bands, Q, most):
    from paper_2511_16576_gb300 import binding as B
    ctx = B.Context(0)
    rng = np.random.default_rng(K * 1000 + bands * 7 + Q)
    rows = K // bands
    db = rng.integers(0, 3, (500, K)).astype(np.int32)
    q = rng.integers(0, 3, (Q, K)).astype(np.int32)
    same = rng.random(Q) < 0.5  # half the queries agree with db row 0 almost everywhere
    q[same] = db[0]
    q[same, rng.integers(0, K)] = 7
    db[db == 2], q[q == 2] = T, T  # not found on both sides is no agreement
    n = rng.integers(0, most + 1, Q)
    n[rng.random(Q) < 0.2] = 0
    n[-1] = most
    rp = np.concatenate([[0], np.cumsum(n)]).astype(np.int64)
    cand = rng.integers(0, 500, rp[-1]).astype(np.int32)
    cand[rng.random(len(cand)) < 0.3] = 0
    P = B.make_params(K, bands, T, 3)
    dv = [torch.from_numpy(a).to(DEV) for a in (q, db, rp, cand)]
    for want_bands in (True, False):
        got = B.jaccard_estimate(ctx, *dv, P, want_bands)
        count, mask = got if want_bands else (got[0] if isinstance(got, tuple) else got, None)
        count = count.cpu().numpy().astype(np.int64)
        row = np.repeat(np.arange(Q), n)
        for x0 in range(0, len(cand), 1 << 15):
            r, c = row[x0:x0 + (1 << 15)], cand[x0:x0 + (1 << 15)]
            eq = (q[r] == db[c]) & (q[r] != T)
            assert np.array_equal(count[x0:x0 + len(r)], eq.sum(1))
            if mask is not None:
                full = eq.reshape(-1, bands, rows).all(2)[:, :32]
                bits = (full.astype(np.int64) << np.arange(full.shape[1])).sum(1)
                assert np.array_equal(mask[x0:x0 + len(r)].cpu().numpy().view(np.uint32), bits)
    ctx.close()
