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
