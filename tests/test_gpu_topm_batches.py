"""Top-m lists (A6) of batches large enough for the warp-per-row kernel: rows of every length around
a warp, its 128-pair limit and the block kernel's, ties, duplicate pairs, special scores."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("Q", [511, 512, 777])
@pytest.mark.parametrize("m", [1, 10, 128, 200])
def test_topm_of_large_batches(Q, m):
    from paper_2511_16576_gb300 import binding as B
    ctx = B.Context(0)
    rng = np.random.default_rng(Q + m)
    lens = rng.choice([0, 1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 130, 400], Q)
    row_ptr = np.zeros(Q + 1, np.int64)
    row_ptr[1:] = np.cumsum(lens)
    E = int(row_ptr[-1])
    cand = rng.integers(0, 60, E).astype(np.int32)  # duplicates within a row
    count = rng.integers(0, 9, E).astype(np.uint16)
    count[rng.random(E) < 0.01] = 5000  # ranks as 4,096
    score = rng.choice(np.array([0.0, 0.25, 0.5, 1.0, np.inf], np.float32), E)
    t = lambda a: torch.from_numpy(a).to(DEV)
    ids, nn = B.topm(ctx, t(row_ptr), t(cand), t(count.view(np.int16)), m)
    ids_s, nn_s = B.topm(ctx, t(row_ptr), t(cand), None, m, score=t(score))
    ids, nn, ids_s, nn_s = (x.cpu().numpy() for x in (ids, nn, ids_s, nn_s))
    for q in range(Q):
        r = slice(row_ptr[q], row_ptr[q + 1])
        key = -np.minimum(count[r].astype(np.int64), 4096)
        for got, n, k in ((ids[q], nn[q], key), (ids_s[q], nn_s[q], -score[r].astype(np.float64))):
            exp = cand[r][np.lexsort((cand[r], k))][:m]
            assert n == len(exp) and np.array_equal(got[:n], exp) and (got[n:] == -1).all()
    ctx.close()
