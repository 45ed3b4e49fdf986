"""Several host threads, a context each, in kernels whose shared memory differs by call."""
import ctypes
import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def test_bitmap_joins_of_a_large_and_small_sets():
    """The bitmap of 1,000,000 ids (122 KB of shared memory) beside six threads with bitmaps of one
    vector: no call is refused, and every row is found."""
    from paper_2511_16576_gb300 import binding as B
    lib = B.load()
    rng = np.random.default_rng(1)
    P = B.make_params(4, 2)
    keep, bad = [], []

    def caller(n, calls):
        h = torch.from_numpy(rng.integers(0, 1000, (n, 4)).astype(np.int32)).to(DEV)
        ctx = B.Context(0)
        index = B.lsh_build(ctx, h, P)
        q, rows = h[:4].clone(), torch.empty(5, dtype=torch.int64, device=DEV)
        cand = torch.empty(1 << 16, dtype=torch.int32, device=DEV)
        want = B.lsh_query(ctx, index, q)[1].numel()
        stream, total = torch.cuda.Stream(), ctypes.c_int64()
        keep.append((h, ctx, index, q, rows, cand, stream))
        args = (ctx.handle, index.handle, q.data_ptr(), 4, rows.data_ptr(), cand.data_ptr(), cand.numel(),
                ctypes.byref(total), stream.cuda_stream)

        def go():
            for _ in range(calls):
                rc = lib.pmh_lsh_query(*args)
                if rc != 0 or total.value != want:
                    bad.append((n, rc, total.value, lib.pmh_last_error()))
        return go
    threads = [threading.Thread(target=f) for f in
               [caller(1_000_000, 6000)] + [caller(100 + i, 8000) for i in range(6)]]
    torch.cuda.synchronize()
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, (len(bad), bad[0])


def test_topm_beside_the_capture_of_graphs():
    """Top-m of counts up to 4,096 (49 KB of shared memory) beside a thread that captures query graphs at
    K = 8 (33 KB)."""
    from paper_2511_16576_gb300 import binding as B
    lib = B.load()
    bad = []
    n = 300
    rows = torch.arange(0, 601, n, dtype=torch.int64, device=DEV)
    cand = torch.arange(600, dtype=torch.int32, device=DEV)
    count = torch.arange(600, dtype=torch.int16, device=DEV)
    ids, nn = torch.empty((2, 64), dtype=torch.int32, device=DEV), torch.empty(2, dtype=torch.int32, device=DEV)
    P = B.make_params(8, 2)
    ctx1 = B.Context(0)
    index = B.lsh_build(ctx1, torch.zeros((64, 8), dtype=torch.int32, device=DEV), P)
    ctx0, stream = B.Context(0), torch.cuda.Stream()
    torch.cuda.synchronize()
    done = threading.Event()

    def capture():
        while not done.is_set():
            B.QueryGraph(ctx1, index, 4, 64, 256, 8).close()

    def topm():
        for _ in range(40_000):
            rc = lib.pmh_topm(ctx0.handle, rows.data_ptr(), cand.data_ptr(), count.data_ptr(), None, 2, 64,
                              ids.data_ptr(), nn.data_ptr(), stream.cuda_stream)
            if rc != 0:
                bad.append((rc, lib.pmh_last_error()))
        done.set()
    threads = [threading.Thread(target=f) for f in (capture, topm)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not bad, (len(bad), bad[0])
    assert torch.equal(ids[0].cpu(), torch.arange(299, 235, -1, dtype=torch.int32))
