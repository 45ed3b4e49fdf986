"""Reranker gradients (A7): several chunks per block, and features that are only 4-byte aligned,
against the oracle network with the same bf16 rounding points."""
import numpy as np
import pytest
import torch

from test_gpu_rerank import oracle_run, random_features

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("n,shift", [(128, 2), (300, 2), (20_000, 0), (40_001, 6)])
def test_gradients_over_chunks_and_alignments(orc, n, shift):
    from paper_2511_16576_gb300 import binding as B
    ctx = B.Context(0)
    rng = np.random.default_rng(n)
    feat, label = random_features(rng, n), rng.random(n).astype(np.float32)
    flat = B.init_rerank_params(seed=n)
    r = B.Reranker(ctx, flat)
    buf = torch.zeros(feat.size + 8, dtype=torch.int16, device=DEV)
    f_d = buf[shift:shift + feat.size].view(n, 48)  # shift 2 and 6: off a 16-byte boundary
    f_d.copy_(torch.from_numpy(feat))
    grads, loss = r.gradients(f_d, torch.from_numpy(label).to(DEV))
    _, ref_loss, g_ref = oracle_run(orc, B, feat, label, flat)
    assert abs(float(loss.item()) - ref_loss) <= 1e-3 * ref_loss
    for got, ref in zip(B.unpack_params(grads.cpu().numpy().astype(np.float64)), g_ref):
        got, ref = got.reshape(-1), ref.reshape(-1)
        assert np.linalg.norm(got - ref) <= 2e-2 * np.linalg.norm(ref) + 1e-9
    r.close()
    ctx.close()
