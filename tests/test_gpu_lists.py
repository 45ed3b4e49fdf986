"""Fixed-width lists to CSR, at the edge between one block and three launches."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("Q,m", [(1, 1), (1, 1024), (33, 32), (1024, 8), (1024, 9), (1025, 1), (8, 1024), (3000, 5)])
def test_lists_to_csr(Q, m):
    from paper_2511_16576_gb300 import binding as B
    ctx = B.Context(0)
    rng = np.random.default_rng(Q + m)
    n = rng.integers(0, m + 1, Q).astype(np.int32)
    n[0], n[-1] = 0 if Q > 1 else m, m
    ids = rng.integers(0, 1 << 30, (Q, m)).astype(np.int32)
    rp, cand = B.lists_to_csr(ctx, torch.from_numpy(ids).to(DEV), torch.from_numpy(n).to(DEV))
    rp = rp.cpu().numpy()
    assert np.array_equal(rp, np.concatenate([[0], np.cumsum(n)]))
    want = np.concatenate([ids[q, :n[q]] for q in range(Q)])
    assert np.array_equal(cand.cpu().numpy()[:rp[-1]], want)
    ctx.close()
