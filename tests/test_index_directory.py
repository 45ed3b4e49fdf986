"""The bucket index's directory: every slot is written, and no lookup leaves it, up to the end of the
last valid composite's bucket (index arithmetic on the CPU; the joins that look it up on the GPU)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
T = 1 << 24

HARNESS = r'''
#include <stdint.h>
#include "directory.cuh"
struct Checked {  // the directory, counting reads out of its range
    const int64_t* dir;
    int64_t len;
    int64_t* outside;
    int64_t operator[](int64_t s) const
    {
        if (s >= 0 && s < len) return dir[s];
        ++*outside;
        return 0;
    }
};
extern "C" void layout(uint32_t bands, int64_t entries, int64_t* out)
{
    const int bits = pmh_band_bits(bands);
    const int64_t cmax = pmh_dir_cmax(bands, bits);
    const int sh = pmh_dir_shift(entries, cmax);
    out[0] = bits, out[1] = cmax, out[2] = sh, out[3] = pmh_dir_len(cmax, sh);
}
extern "C" int64_t fill(const uint32_t* comp, int64_t m, int sh, int64_t cmax, int64_t* dir, int64_t len)
{
    int64_t outside = 0, from, to;
    for (int64_t e = 0; e <= m; ++e) {
        pmh_dir_slots(comp, m, e, sh, cmax, &from, &to);
        for (int64_t s = from; s <= to; ++s) {
            if (s < 0 || s >= len || dir[s] != -1) ++outside;  // each slot once
            else dir[s] = e;
        }
    }
    return outside;
}
extern "C" int64_t lookup(const uint32_t* comp, const int64_t* dir, int64_t len, int sh, const uint32_t* c,
                          int64_t n, int64_t* out)
{
    int64_t outside = 0;
    const Checked d{dir, len, &outside};
    for (int64_t i = 0; i < n; ++i) out[i] = pmh_comp_lower_bound(comp, d, sh, c[i]);
    return outside;
}
'''


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("directory")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2511_16576_gb300", "csrc"),
                    str(d / "h.cpp"), "-o", str(d / "h.so")], check=True)
    lib = ctypes.CDLL(str(d / "h.so"))
    lib.fill.restype = lib.lookup.restype = ctypes.c_int64
    return lib


def ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


@pytest.mark.parametrize("bands", [1, 2, 3, 7, 8, 15, 16, 31, 63, 64, 127, 128])
@pytest.mark.parametrize("n", [0, 1, 2, 40, 3000, 120_000])
def test_lookups_stay_inside(harness, bands, n):
    m = n * bands if n < 100_000 else n * min(bands, 8)
    lay = np.zeros(4, np.int64)
    harness.layout(ctypes.c_uint32(bands), ctypes.c_int64(m), ptr(lay))
    bits, cmax, sh, length = (int(v) for v in lay)
    rng = np.random.default_rng(bands * 1000 + n)
    for valid in (1.0, 0.7, 0.0):  # shares of valid entries; all ones: invalid
        comp = np.where(rng.random(m) < valid, rng.integers(0, cmax, m), 0xFFFFFFFF).astype(np.uint32)
        if m and valid:
            comp[rng.integers(0, m, 3)] = cmax - 1  # the last valid composite
        comp.sort()
        d = np.full(length, -1, np.int64)
        assert harness.fill(ptr(comp), ctypes.c_int64(m), sh, ctypes.c_int64(cmax), ptr(d),
                            ctypes.c_int64(length)) == 0
        assert (d >= 0).all() or m == 0
        if m == 0:
            d[:] = 0  # (an empty index is cleared)
        c = np.concatenate([np.arange(bands, dtype=np.int64) << (32 - bits),
                            (np.arange(1, bands + 1, dtype=np.int64) << (32 - bits)) - 1, [0, cmax - 1, cmax],
                            rng.integers(0, cmax, 500), comp[comp < cmax][:500]]).astype(np.uint32)
        c = np.unique(np.concatenate([c, np.minimum(c.astype(np.int64) + 1, cmax).astype(np.uint32)]))
        got = np.zeros(len(c), np.int64)
        assert harness.lookup(ptr(comp), ptr(d), ctypes.c_int64(length), sh, ptr(c),
                              ctypes.c_int64(len(c)), ptr(got)) == 0
        assert np.array_equal(got, np.searchsorted(comp, c))


def mix(z):
    z &= (1 << 64) - 1
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & ((1 << 64) - 1)
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & ((1 << 64) - 1)
    return z ^ (z >> 31)


# (bands, rows, lsh_seed, x): the tuple (1, .., rows - 1, x) of the last band has the largest composite
@pytest.mark.gpu
@pytest.mark.parametrize("bands,rows,lsh_seed,x,n,Q", [
    (1, 1, 48, 6_950_326, 300, 5),          # range join
    (31, 1, 20, 10_832_831, 500, 5),        # bitmap join
    (2, 5, 153, 1_877_182, 3000, 1100),     # warp join
    (16, 6, 7, 7_243_220, 3000, 1100),
    (31, 5, 21, 14_524_631, 409_601, 3),    # shared-memory set
    (15, 6, 1, 4_975_946, 409_601, 3),      # warp merge
])
def test_last_composite(orc, bands, rows, lsh_seed, x, n, Q):
    import torch
    from paper_2511_16576_gb300 import binding as B
    key = mix(lsh_seed + bands * 0x9E3779B97F4A7C15)
    for v in list(range(1, rows)) + [x]:
        key = mix(key ^ v)
    bits = bands.bit_length()
    assert key >> (32 + bits) == (1 << (32 - bits)) - 1
    K = bands * rows
    rng = np.random.default_rng(bands)
    ph = rng.integers(0, 4, (n, K)).astype(np.uint32) + 20
    qh = rng.integers(0, 1000, (Q, K)).astype(np.uint32) + 2000
    last = np.array(list(range(1, rows)) + [x], np.uint32)
    ph[::37, -rows:] = last
    ph[5, :] = T  # invalid entries sort behind the last bucket
    qh[::2, -rows:] = last
    qh[1] = ph[1]
    ctx = B.Context(0)
    P = B.make_params(K, bands, T, 3, lsh_seed)
    dev = lambda a: torch.from_numpy(a.view(np.int32)).cuda()
    index = B.lsh_build(ctx, dev(ph), P)
    rp_ref, cand_ref = orc.candidates(qh, ph, bands, rows, T)
    for capacity in (None, int(rp_ref[-1])):
        row_ptr, cand = B.lsh_query(ctx, index, dev(qh), capacity=capacity)
        assert np.array_equal(row_ptr.cpu().numpy(), rp_ref)
        assert np.array_equal(cand.cpu().numpy(), cand_ref)
    assert rp_ref[1] == len(ph[::37])
    index.close()
    ctx.close()
