"""The prefix sums behind row pointers at the edge between one block and three launches: candidate
rows of every count pass must add up to the exact join."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("Q", [1, 31, 255, 256, 257, 2048, 8191, 8192, 8193, 20_000])
def test_row_pointers(Q):
    from paper_2511_16576_gb300 import binding as B
    ctx = B.Context(0)
    rng = np.random.default_rng(Q)
    P = B.make_params(2, 1, 1 << 20, 7, lsh_seed=9)
    db = rng.integers(0, 40, (3000, 2)).astype(np.int32)
    q = rng.integers(0, 60, (Q, 2)).astype(np.int32)  # some rows empty
    X = B.lsh_build(ctx, torch.from_numpy(db).to(DEV), P)
    rp, cand = B.lsh_query(ctx, X, torch.from_numpy(q).to(DEV))[:2]
    key = db[:, 0] * 1000 + db[:, 1]
    count = dict(zip(*np.unique(key, return_counts=True)))
    want = np.array([count.get(k, 0) for k in q[:, 0] * 1000 + q[:, 1]])
    rp = rp.cpu().numpy()
    assert rp[0] == 0 and np.array_equal(np.diff(rp), want)
    i = int(np.argmax(want))
    got = cand[rp[i]:rp[i + 1]].cpu().numpy()
    assert np.array_equal(got, np.flatnonzero(key == q[i, 0] * 1000 + q[i, 1]))
    ctx.close()
