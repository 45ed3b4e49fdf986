// estimate.cu -- steps A5 (agreement estimate) and A6 (top-m selection).
//
// A5 follows Theorem 1: Pr[h_k(q) = h_k(p)] = J(q, p), so the fraction of
// agreeing positions estimates J.  The candidate pairs of all rows are cut into
// chunks of consecutive pairs that warps take in turn (rows range from a few
// candidates to thousands, so a block per row would leave the grid waiting on
// the longest).  Rows of at most 128 hashes: a lane holds four of the query's hashes
// and reads the candidates' as 16-byte vectors (512 bytes per row at K = 128), the count
// is a warp reduction, and the band-match bits and the reranker's features (A7) come from
// the same equality bits; longer rows read both sides and gather the bits in shared memory.
//
// A6 orders each candidate row by a 64-bit key (ranks by a warp for short rows of a large
// batch, else a block's bitonic sort in shared memory), keeping the first m:
// key = (K - count) << 32 | id for the plain form, or (~orderable(score)) << 32 | id for a
// learned score.
#include <cuda_bf16.h>

#include <algorithm>

#include "pmh_internal.cuh"

namespace {

constexpr int kMaxK = 4096;
constexpr int kAgreeWarps = 4;
constexpr int kAgreeChunk = 64;  // consecutive pairs per warp turn, fewer in a small batch
constexpr int kAgreeGroup = 4;   // pairs compared at a time (their loads in flight together)

// pairs per warp turn: kAgreeChunk, or so many that every warp of the grid gets a turn (a
// multiple of the pairs compared at a time).  32 pairs with features: 51 us by one
// warp, 8.9 us by sixteen
__device__ __forceinline__ int64_t agree_chunk(int64_t total, int64_t nwarps, int group)
{
    const int64_t per = (total + nwarps - 1) / nwarps;
    return min((int64_t)kAgreeChunk, (per + group - 1) / group * group);
}

// the row holding pair x: the last q with row_ptr[q] <= x
__device__ __forceinline__ int64_t agree_row_of(const int64_t* __restrict__ row_ptr, int64_t Q, int64_t x)
{
    int64_t lo = 0, hi = Q;
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (row_ptr[mid] <= x) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Rows of at most 128 hashes (K % 4 == 0): a lane holds four hashes of the query, read once per
// row of candidates, and eight pairs' rows are in flight at a time.  The band bits come from
// the lanes' four equality bits with one shuffle or ballot (bands whose hashes do not straddle
// lanes unevenly: rows 1, 2, or a multiple of 4).  Bound by the issue rate and L2: with the
// query reloaded and the equality words built in shared memory for every pair it was 170
// issue slots a pair.  4,096 queries, 4.0M pairs of 300,000 rows, 64 x 2 bands: 606 -> 352 us
// (5.9 TB/s of rows, two thirds of them out of L2)
constexpr int kAgreeRowK = 128;
constexpr int kAgreeRowGroup = 8;

template <bool kFeat>  // (kFeat: K = 128)
__global__ void __launch_bounds__(kAgreeWarps * 32, kFeat ? 6 : 8)
agree_short_kernel(const uint32_t* __restrict__ qh, const uint32_t* __restrict__ ph,
                   const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ cand, int64_t Q,
                   int64_t cap, int K, int bands, int rows, uint32_t T, uint16_t* __restrict__ count,
                   uint32_t* __restrict__ bandmask, __nv_bfloat16* __restrict__ feat, FeatSrc qf,
                   FeatSrc pf, const int* __restrict__ d_flags)
{
    constexpr int G = kAgreeRowGroup;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (d_flags && *d_flags) return;  // failed validation or candidate overflow
    const int64_t total = min(row_ptr[Q], cap);
    const int64_t nwarps = (int64_t)gridDim.x * kAgreeWarps;
    // (a pair's feature inputs are fetched pair by pair: two pairs a warp while that fills no grid)
    const int64_t chunk = agree_chunk(total, nwarps, kFeat ? 2 : G);
    const bool in = lane < K / 4;
    // band `lane` in the equality bits: bits [bsh, bsh + rows) of lane bsrc, or (rows % 4 == 0) the
    // rows / 4 lanes from lane bsh on
    const bool whole = rows >= 4, band = lane < bands;
    const int bsrc = whole ? 0 : (lane * rows) >> 2, bsh = whole ? (rows / 4) * lane : (lane * rows) & 3;
    const uint32_t bneed = whole ? (rows >= 128 ? ~0u : (1u << (rows / 4)) - 1u) : (1u << rows) - 1u;
    uint4 u = make_uint4(0u, 0u, 0u, 0u);
    unsigned live = 0;  // this lane's hashes of the query that were found (not T)
    int64_t uq = -1;    // the query u holds
    for (int64_t ch = (int64_t)blockIdx.x * kAgreeWarps + wid; ch * chunk < total; ch += nwarps) {
        const int64_t x0 = ch * chunk, x1 = min(x0 + chunk, total);
        const int64_t q0 = agree_row_of(row_ptr, Q, x0);
        for (int64_t xb = x0; xb < x1; xb += 32) {
            const int nvalid = (int)min((int64_t)32, x1 - xb);
            int64_t ql = q0;
            int32_t pl = 0;
            if (lane < nvalid) {
                while (row_ptr[ql + 1] <= xb + lane) ++ql;
                pl = cand[xb + lane];
            }
            const int64_t qprev = __shfl_up_sync(0xffffffffu, ql, 1);
            const unsigned turns = __ballot_sync(0xffffffffu, lane < nvalid && ql != (lane ? qprev : uq));
            int my_count = 0;
            unsigned my_bands = 0;
            for (int t0 = 0; t0 < nvalid; t0 += G) {
                uint4 v[G];
#pragma unroll
                for (int t = 0; t < G; ++t) {
                    const int64_t pp = __shfl_sync(0xffffffffu, pl, t0 + t);
                    v[t] = make_uint4(0u, 0u, 0u, 0u);
                    if (in && t0 + t < nvalid) v[t] = __ldg(reinterpret_cast<const uint4*>(ph + pp * K) + lane);
                }
#pragma unroll
                for (int t = 0; t < G; ++t) {
                    if (t0 + t >= nvalid) continue;  // warp-uniform
                    if ((turns >> (t0 + t)) & 1u) {
                        uq = __shfl_sync(0xffffffffu, ql, t0 + t);
                        if (in) u = __ldg(reinterpret_cast<const uint4*>(qh + uq * K) + lane);
                        live = in ? (unsigned)(u.x != T) | ((unsigned)(u.y != T) << 1) |
                                        ((unsigned)(u.z != T) << 2) | ((unsigned)(u.w != T) << 3)
                                  : 0u;
                    }
                    const unsigned bits = ((unsigned)(u.x == v[t].x) | ((unsigned)(u.y == v[t].y) << 1) |
                                           ((unsigned)(u.z == v[t].z) << 2) | ((unsigned)(u.w == v[t].w) << 3)) &
                                          live;
                    int ct = __popc(bits), lt = 0, gt = 0;
                    if (kFeat) {  // the three counts in one sum (10 bits each)
                        lt = (u.x < v[t].x) + (u.y < v[t].y) + (u.z < v[t].z) + (u.w < v[t].w);
                        gt = (u.x > v[t].x) + (u.y > v[t].y) + (u.z > v[t].z) + (u.w > v[t].w);
                        const int sum = __reduce_add_sync(0xffffffffu, ct | (lt << 10) | (gt << 20));
                        ct = sum & 1023;
                        lt = (sum >> 10) & 1023;
                        gt = sum >> 20;
                    } else {
                        ct = __reduce_add_sync(0xffffffffu, ct);
                    }
                    if (lane == t0 + t) my_count = ct;
                    if (bandmask) {
                        const uint32_t from = whole ? __ballot_sync(0xffffffffu, bits == 0xFu)
                                                    : __shfl_sync(0xffffffffu, bits, bsrc);
                        const unsigned mb = __ballot_sync(0xffffffffu, band && ((from >> (bsh & 31)) & bneed) == bneed);
                        if (lane == t0 + t) my_bands = mb;
                    }
                    if (kFeat) {
                        const int64_t q = __shfl_sync(0xffffffffu, ql, t0 + t);
                        const int64_t pp = __shfl_sync(0xffffffffu, pl, t0 + t);
                        const float fhi = pmh_feature_col(lane, K, ct, lt, gt, pmh_feat_pair(qf, pf, q, pp));
                        __nv_bfloat16* f = feat + (xb + t0 + t) * 48;
                        f[lane] = __float2bfloat16_rn(bits == 0xFu ? 1.f : 0.f);
                        if (lane < 16) f[32 + lane] = __float2bfloat16_rn(fhi);
                    }
                }
            }
            if (lane < nvalid) {
                if (count) count[xb + lane] = (uint16_t)my_count;
                if (bandmask) bandmask[xb + lane] = my_bands;
            }
        }
    }
}

// Rows of any K.  Warps take chunks of consecutive pairs (the row of the first by
// binary search over row_ptr); 32 pairs at a time each lane reads one pair's
// candidate id and steps its row on from there, and the warp then compares the
// pairs four at a time (ids and rows by shuffle).  Per pair:
// equality bits of the K hashes (16-byte loads when K % 4 == 0), the count (warp
// sum), the full-match bits of the first 32 bands and, optionally, the reranker's
// feature row.
template <bool kFeat>  // feature rows written (a build without their work for the counts alone)
__global__ void __launch_bounds__(kAgreeWarps * 32, 6)
agree_rows_kernel(const uint32_t* __restrict__ qh, const uint32_t* __restrict__ ph,
                  const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ cand, int64_t Q,
                  int64_t cap, int K, int bands, int rows, uint32_t T, uint16_t* __restrict__ count,
                  uint32_t* __restrict__ bandmask, __nv_bfloat16* __restrict__ feat, FeatSrc qf,
                  FeatSrc pf, const int* __restrict__ d_flags)
{
    __shared__ uint32_t eqbits[kAgreeWarps][kAgreeGroup][kMaxK / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (d_flags && *d_flags) return;  // failed validation or candidate overflow
    const int64_t total = min(row_ptr[Q], cap);
    const int64_t nwarps = (int64_t)gridDim.x * kAgreeWarps;
    const int K4 = K / 4;
    // equality words in shared memory: for the band bits, and for the features' groups
    // unless K = 128 (then lane l holds group l's four hashes)
    const bool need_eq = bandmask || (kFeat && K != 128);
    const int64_t chunk = agree_chunk(total, nwarps, kAgreeGroup);
    for (int64_t ch = (int64_t)blockIdx.x * kAgreeWarps + wid; ch * chunk < total; ch += nwarps) {
        const int64_t x0 = ch * chunk, x1 = min(x0 + chunk, total);
        const int64_t q0 = agree_row_of(row_ptr, Q, x0);
        for (int64_t xb = x0; xb < x1; xb += 32) {
            const int nvalid = (int)min((int64_t)32, x1 - xb);
            const int64_t xl = xb + lane;
            int64_t ql = q0;
            int32_t pl = 0;
            if (lane < nvalid) {
                while (row_ptr[ql + 1] <= xl) ++ql;
                pl = cand[xl];
            }
            for (int t0 = 0; t0 < nvalid; t0 += kAgreeGroup) {
                const int64_t x = xb + t0;
                int64_t qq[kAgreeGroup], pp[kAgreeGroup];
                bool ok[kAgreeGroup];
    #pragma unroll
                for (int t = 0; t < kAgreeGroup; ++t) {
                    ok[t] = t0 + t < nvalid;
                    qq[t] = __shfl_sync(0xffffffffu, ql, (t0 + t) & 31);
                    pp[t] = __shfl_sync(0xffffffffu, pl, (t0 + t) & 31);
                }
                // lt / gt: hashes with h(q) < h(p) / h(q) > h(p); grp: K = 128, lane l's four
                // hashes (group l of the features' 32-group split) all equal
                int c[kAgreeGroup] = {0, 0, 0, 0}, lt[kAgreeGroup] = {0, 0, 0, 0}, gt[kAgreeGroup] = {0, 0, 0, 0};
                bool grp[kAgreeGroup] = {false, false, false, false};
                if ((K & 3) == 0) {
                    for (int base = 0; base < K4; base += 32) {
                        const int i = base + lane;
                        uint4 u[kAgreeGroup], v[kAgreeGroup];
    #pragma unroll
                        for (int t = 0; t < kAgreeGroup; ++t) {
                            u[t] = v[t] = make_uint4(0u, 0u, 0u, 0u);
                            if (ok[t] && i < K4) {
                                u[t] = __ldg(reinterpret_cast<const uint4*>(qh + qq[t] * K) + i);
                                v[t] = __ldg(reinterpret_cast<const uint4*>(ph + pp[t] * K) + i);
                            }
                        }
    #pragma unroll
                        for (int t = 0; t < kAgreeGroup; ++t) {
                            unsigned bits = 0;
                            if (i < K4) {
                                bits = (unsigned)((u[t].x == v[t].x) & (u[t].x != T)) |
                                       ((unsigned)((u[t].y == v[t].y) & (u[t].y != T)) << 1) |
                                       ((unsigned)((u[t].z == v[t].z) & (u[t].z != T)) << 2) |
                                       ((unsigned)((u[t].w == v[t].w) & (u[t].w != T)) << 3);
                                if (kFeat) {
                                    lt[t] += (u[t].x < v[t].x) + (u[t].y < v[t].y) + (u[t].z < v[t].z) +
                                             (u[t].w < v[t].w);
                                    gt[t] += (u[t].x > v[t].x) + (u[t].y > v[t].y) + (u[t].z > v[t].z) +
                                             (u[t].w > v[t].w);
                                }
                            }
                            c[t] += __popc(bits);
                            grp[t] = bits == 0xFu;
                            if (need_eq) {
                                // hash 4i+e is bit (4i+e) % 32 of word i / 8: OR eight lanes' nibbles
                                unsigned w0 = bits << ((lane & 7) * 4);
                                w0 |= __shfl_xor_sync(0xffffffffu, w0, 1);
                                w0 |= __shfl_xor_sync(0xffffffffu, w0, 2);
                                w0 |= __shfl_xor_sync(0xffffffffu, w0, 4);
                                if ((lane & 7) == 0 && i < K4) eqbits[wid][t][i >> 3] = w0;
                            }
                        }
                    }
                } else {
                    for (int base = 0; base < K; base += 32) {
                        const int i = base + lane;
    #pragma unroll
                        for (int t = 0; t < kAgreeGroup; ++t) {
                            const bool in = ok[t] && i < K;
                            const uint32_t a = in ? qh[qq[t] * K + i] : 0u, b = in ? ph[pp[t] * K + i] : 0u;
                            const bool eq = in && a == b && a != T;
                            const unsigned bal = __ballot_sync(0xffffffffu, eq);
                            c[t] += eq;
                            if (kFeat && in) {
                                lt[t] += a < b;
                                gt[t] += a > b;
                            }
                            if (lane == 0) eqbits[wid][t][base / 32] = bal;
                        }
                    }
                }
                __syncwarp();
    #pragma unroll
                for (int t = 0; t < kAgreeGroup; ++t) {
                    if (!ok[t]) continue;  // warp-uniform
                    const int64_t xt = x + t;
                    int ct, ltt = 0, gtt = 0;
                    if (kFeat && K < 1024) {  // the three counts in one sum (10 bits each)
                        const int sum = __reduce_add_sync(0xffffffffu, c[t] | (lt[t] << 10) | (gt[t] << 20));
                        ct = sum & 1023;
                        ltt = (sum >> 10) & 1023;
                        gtt = sum >> 20;
                    } else {
                        ct = __reduce_add_sync(0xffffffffu, c[t]);
                        if (kFeat) {
                            ltt = __reduce_add_sync(0xffffffffu, lt[t]);
                            gtt = __reduce_add_sync(0xffffffffu, gt[t]);
                        }
                    }
                    if (count && lane == 0) count[xt] = (uint16_t)ct;
                    if (bandmask) {
                        bool all = lane < bands;
                        for (int r = 0; r < rows && all; ++r) {
                            const int k = lane * rows + r;
                            all = (eqbits[wid][t][k >> 5] >> (k & 31)) & 1u;
                        }
                        const unsigned mb = __ballot_sync(0xffffffffu, all);
                        if (lane == 0) bandmask[xt] = mb;
                    }
                    if (kFeat) {
                        float flo, fhi;
                        if (K == 128) {
                            flo = grp[t] ? 1.f : 0.f;
                            fhi = pmh_feature_col(lane, K, ct, ltt, gtt, pmh_feat_pair(qf, pf, qq[t], pp[t]));
                        } else {
                            pmh_feature_values(eqbits[wid][t], K, ct, ltt, gtt, pmh_feat_pair(qf, pf, qq[t], pp[t]),
                                               lane, flo, fhi);
                        }
                        __nv_bfloat16* f = feat + xt * 48;
                        f[lane] = __float2bfloat16_rn(flo);
                        if (lane < 16) f[32 + lane] = __float2bfloat16_rn(fhi);
                    }
                }
                __syncwarp();
            }
        }
    }
}

// orderable float bits: larger float -> larger unsigned
__device__ __forceinline__ uint32_t f2ord(float f)
{
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

constexpr int kTopThreads = 256;
constexpr int kTopChunk = 2048;  // new items merged per round

__device__ void bitonic_sort_u64(uint64_t* s, int n /* power of two */)
{
    for (int k = 2; k <= n; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < n; i += blockDim.x) {
                int l = i ^ j;
                if (l > i) {
                    uint64_t a = s[i], b = s[l];
                    bool up = (i & k) == 0;
                    if ((a > b) == up) {
                        s[i] = b;
                        s[l] = a;
                    }
                }
            }
            __syncthreads();
        }
    }
}

// Short rows (at most kShortRow pairs), a warp each: every key's rank among the row's keys
// (from shared memory) is its place in the list, so nothing is sorted and nothing waits
// on a barrier.  4,096 rows of 64: 16 us with the block kernel's empty launch behind it, 30 us
// with a block and a bitonic sort each.
constexpr int kShortRow = 128;
constexpr int kShortWarps = 8;

__device__ __forceinline__ uint64_t topm_key(const int32_t* cand, const uint16_t* count, const float* score, int K,
                                             int64_t x)
{
    const uint32_t hi = score ? ~f2ord(score[x]) : (uint32_t)(K - min((int)count[x], K));
    return ((uint64_t)hi << 32) | (uint32_t)cand[x];
}

__global__ void __launch_bounds__(kShortWarps * 32)
topm_short_kernel(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ cand,
                  const uint16_t* __restrict__ count, const float* __restrict__ score, int64_t Q, int K, int m,
                  int32_t* __restrict__ out_ids, int32_t* __restrict__ out_n, const int* __restrict__ d_flags)
{
    __shared__ uint64_t keys[kShortWarps][kShortRow];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t q = (int64_t)blockIdx.x * kShortWarps + wid;
    if (q >= Q) return;
    const bool failed = d_flags && *d_flags;
    const int64_t b = failed ? 0 : row_ptr[q], e = failed ? 0 : row_ptr[q + 1];
    if (e - b > kShortRow) return;  // topm_kernel's
    const int n = (int)(e - b), kept = min(n, m);
    uint64_t mine[kShortRow / 32];
    int rank[kShortRow / 32];
#pragma unroll
    for (int u = 0; u < kShortRow / 32; ++u) {
        const int i = 32 * u + lane;
        mine[u] = i < n ? topm_key(cand, count, score, K, b + i) : ~0ull;
        rank[u] = 0;
        keys[wid][i] = mine[u];
    }
    __syncwarp();
    const int nu = (n + 31) >> 5;  // (short rows skip the empty registers)
    for (int j = 0; j < n; ++j) {
        const uint64_t k = keys[wid][j];
#pragma unroll
        for (int u = 0; u < kShortRow / 32; ++u)
            if (u < nu) rank[u] += k < mine[u];
    }
    // equal keys (the same pair twice) share a rank: their ranks' sum is short, and each is
    // moved behind the equal ones before it
    int sum = 0;
#pragma unroll
    for (int u = 0; u < kShortRow / 32; ++u) sum += 32 * u + lane < n ? rank[u] : 0;
    if (__reduce_add_sync(0xffffffffu, sum) != n * (n - 1) / 2)
        for (int j = 0; j < n; ++j)
#pragma unroll
            for (int u = 0; u < kShortRow / 32; ++u)
                rank[u] += j < 32 * u + lane && keys[wid][j] == mine[u];
#pragma unroll
    for (int u = 0; u < kShortRow / 32; ++u)
        if (32 * u + lane < n && rank[u] < m) out_ids[q * m + rank[u]] = (int32_t)(uint32_t)(mine[u] & 0xFFFFFFFFu);
    for (int i = kept + lane; i < m; i += 32) out_ids[q * m + i] = -1;
    if (lane == 0) out_n[q] = kept;
}

// one block per query.  Count form: a histogram of the row's counts (0..K) gives
// the largest threshold c* with at least m pairs of count >= c*; every key of
// those pairs is gathered and sorted, and the first m kept -- the m best keys
// (count desc, id asc) all have count >= c*, so the list is the full sort's.  A
// row whose gathered set would pass kSelMax (a long tie at c*), and the score
// form, take the merge form: the running top-m kept in s[0..m), each new chunk
// of the row appended and sorted with it.
constexpr int kSelMax = 2048;
constexpr int kTopMaxM = 1024;   // of the callers
constexpr int kTopCap = 4096;    // keys of the longest list: a power of two
static_assert(kTopCap >= kTopMaxM + kTopChunk && kTopCap >= kSelMax, "the longest list fits");
constexpr int kTopSmemMax = (int)(sizeof(uint64_t) * kTopCap + sizeof(int) * (kMaxK + 1));

__global__ void __launch_bounds__(kTopThreads)
topm_kernel(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ cand,
            const uint16_t* __restrict__ count, const float* __restrict__ score, int K, int m,
            int cap /* power of two >= max(m + kTopChunk, kSelMax) */, int min_row, int32_t* __restrict__ out_ids,
            int32_t* __restrict__ out_n, const int* __restrict__ d_flags)
{
    extern __shared__ uint64_t s[];  // cap keys, then (count form) K + 1 histogram bins
    __shared__ int sel_c, sel_total, sel_n;
    const int64_t q = blockIdx.x;
    const bool failed = d_flags && *d_flags;
    const int64_t b = failed ? 0 : row_ptr[q], e = failed ? 0 : row_ptr[q + 1];
    if (e - b < min_row) return;  // topm_short_kernel's
    int kept = 0;
    bool merged = true;
    if (!score && e - b > m) {
        int* hist = reinterpret_cast<int*>(s + cap);
        for (int i = threadIdx.x; i <= K; i += blockDim.x) hist[i] = 0;
        if (threadIdx.x == 0) {  // (the warp below always finds the threshold)
            sel_c = 0;
            sel_total = (int)min(e - b, (int64_t)INT32_MAX);
            sel_n = 0;
        }
        __syncthreads();
        for (int64_t x = b + threadIdx.x; x < e; x += blockDim.x) atomicAdd(&hist[min((int)count[x], K)], 1);
        __syncthreads();
        if (threadIdx.x < 32) {
            // lane l sums bins [l*seg, (l+1)*seg); suffix sums over the lanes find the
            // lane holding c*, which then walks its bins downwards
            const int lane = threadIdx.x, seg = (K + 32) / 32;
            const int lo = lane * seg, hi = min(lo + seg, K + 1);
            int mine = 0;
            for (int c = lo; c < hi; ++c) mine += hist[c];
            int suf = mine;  // bins >= lo
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_down_sync(0xffffffffu, suf, o);
                if (lane + o < 32) suf += y;
            }
            const int above = suf - mine;  // bins >= hi
            if (above < m && suf >= m) {
                int acc = above, c = hi - 1;
                for (; c >= lo; --c) {
                    acc += hist[c];
                    if (acc >= m) break;
                }
                sel_c = c;
                sel_total = acc;
            }
        }
        __syncthreads();
        const int cstar = sel_c, total = sel_total;
        if (total <= kSelMax) {
            merged = false;
            for (int64_t x = b + threadIdx.x; x < e; x += blockDim.x) {
                const int c = min((int)count[x], K);
                if (c >= cstar) {
                    const int pos = atomicAdd(&sel_n, 1);
                    if (pos < total) s[pos] = ((uint64_t)(uint32_t)(K - c) << 32) | (uint32_t)cand[x];
                }
            }
            int sz = 2;
            while (sz < total) sz <<= 1;
            for (int i = total + threadIdx.x; i < sz; i += blockDim.x) s[i] = ~0ull;
            __syncthreads();
            bitonic_sort_u64(s, sz);
            kept = m;
        }
    }
    for (int64_t base = b; merged && base < e; base += kTopChunk) {
        int take = (int)(e - base < kTopChunk ? e - base : kTopChunk);
        // sort only the occupied prefix, rounded up to a power of two (most lists are short)
        int sz = 2;
        while (sz < kept + take) sz <<= 1;
        for (int i = threadIdx.x; i < sz; i += blockDim.x) {
            uint64_t key = ~0ull;
            if (i >= kept && i < kept + take) {
                key = topm_key(cand, count, score, K, base + (i - kept));
            } else if (i < kept) {
                key = s[i];
            }
            s[i] = key;
        }
        __syncthreads();
        bitonic_sort_u64(s, sz);
        kept = min(m, kept + take);
    }
    for (int i = threadIdx.x; i < m; i += blockDim.x)
        out_ids[q * m + i] = i < kept ? (int32_t)(uint32_t)(s[i] & 0xFFFFFFFFu) : -1;
    if (threadIdx.x == 0) out_n[q] = kept;
}

// fixed-width lists (ids [Q][m], -1 padded, counts n[Q]) to compact CSR; rows at or
// past the device-side count d_n (optional) are empty
__global__ void list_counts_kernel(const int32_t* __restrict__ n, int64_t Q,
                                   const int64_t* __restrict__ d_n, int64_t* __restrict__ c)
{
    const int64_t live = d_n ? min(Q, *d_n) : Q;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < Q;
         q += (int64_t)gridDim.x * blockDim.x)
        c[q] = q < live ? n[q] : 0;
}

__global__ void list_copy_kernel(const int32_t* __restrict__ ids, const int32_t* __restrict__ n,
                                 int64_t Q, int m, const int64_t* __restrict__ d_n,
                                 const int64_t* __restrict__ row_ptr, int32_t* __restrict__ cand)
{
    if (d_n) Q = min(Q, *d_n);
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < Q * m;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t q = t / m;
        const int i = (int)(t - q * m);
        if (i < n[q]) cand[row_ptr[q] + i] = ids[t];
    }
}

// Both, with the prefix sum between them, for few lists: one block, bound by latency (one
// query's learned form: three launches of 2.5-3.5 us, one of 3.8)
constexpr int kListBlock = 1024;
constexpr int64_t kListsSmall = 8192;  // entries Q * m, with Q <= kListBlock
__global__ void __launch_bounds__(kListBlock)
lists_small_kernel(const int32_t* __restrict__ ids, const int32_t* __restrict__ n, int Q, int m,
                   const int64_t* __restrict__ d_n, int64_t* __restrict__ row_ptr, int32_t* __restrict__ cand)
{
    __shared__ int base[kListBlock], wsum[kListBlock / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int live = d_n ? (int)min((int64_t)Q, *d_n) : Q;
    const int mine = (int)threadIdx.x < live ? n[threadIdx.x] : 0;
    int x = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    const int pre = __reduce_add_sync(0xffffffffu, lane < wid ? wsum[lane] : 0);
    base[threadIdx.x] = pre + x - mine;
    if ((int)threadIdx.x < Q) {
        row_ptr[threadIdx.x] = pre + x - mine;
        if ((int)threadIdx.x == Q - 1) row_ptr[Q] = pre + x;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < live * m; t += kListBlock) {
        const int q = t / m, i = t - q * m;
        if (i < n[q]) cand[base[q] + i] = ids[t];
    }
}

}  // namespace

extern "C" int pmh_lists_to_csr(pmh_ctx ctx, const int32_t* d_ids, const int32_t* d_n, int64_t Q,
                                int32_t m, int64_t* d_row_ptr, int32_t* d_cand, void* stream)
{
    PMH_TRY(pmh_check_device(ctx));
    if (Q < 0 || m < 1 || !d_row_ptr || (Q > 0 && (!d_ids || !d_n || !d_cand)))
        return pmh_set_error(PMH_ERR_ARG, "bad arguments");
    cudaStream_t s = (cudaStream_t)stream;
    if (Q == 0) {
        PMH_CUDA_TRY(cudaMemsetAsync(d_row_ptr, 0, sizeof(int64_t), s));
        return PMH_OK;
    }
    int64_t* counts = nullptr;
    PMH_TRY(pmh_scratch(ctx, SCR_QUERY, sizeof(int64_t) * (size_t)Q, (void**)&counts));
    return pmh_launch_lists_to_csr(ctx, d_ids, d_n, Q, m, nullptr, counts, nullptr, d_row_ptr, d_cand, s);
}

int pmh_launch_lists_to_csr(pmh_ctx ctx, const int32_t* ids, const int32_t* n, int64_t Q, int32_t m,
                            const int64_t* d_q, int64_t* counts, int64_t* sums, int64_t* row_ptr,
                            int32_t* cand, cudaStream_t s)
{
    if (Q <= 0) return PMH_OK;
    if (Q <= kListBlock && Q * m <= kListsSmall) {
        lists_small_kernel<<<1, kListBlock, 0, s>>>(ids, n, (int)Q, m, d_q, row_ptr, cand);
        PMH_LAUNCHED("lists_small_kernel");
        return PMH_OK;
    }
    const int blocks = (int)std::min<int64_t>((Q * m + 255) / 256, (int64_t)ctx->sm_count * 32);
    list_counts_kernel<<<blocks, 256, 0, s>>>(n, Q, d_q, counts);
    PMH_LAUNCHED("list_counts_kernel");
    PMH_TRY(pmh_exclusive_scan_i64(ctx, counts, row_ptr, Q, s, sums));
    list_copy_kernel<<<blocks, 256, 0, s>>>(ids, n, Q, m, d_q, row_ptr, cand);
    PMH_LAUNCHED("list_copy_kernel");
    return PMH_OK;
}

int pmh_launch_agree(pmh_ctx ctx, const uint32_t* qh, const uint32_t* ph, const int64_t* row_ptr,
                     const int32_t* cand, int64_t Q, int64_t cap, const pmh_params* P,
                     uint16_t* count, uint32_t* bandmask, const int* d_flags, cudaStream_t s)
{
    return pmh_launch_agree_features(ctx, qh, ph, row_ptr, cand, Q, cap, P, count, bandmask, nullptr,
                                     FeatSrc{}, FeatSrc{}, d_flags, s);
}

int pmh_launch_agree_features(pmh_ctx ctx, const uint32_t* qh, const uint32_t* ph,
                              const int64_t* row_ptr, const int32_t* cand, int64_t Q, int64_t cap,
                              const pmh_params* P, uint16_t* count, uint32_t* bandmask,
                              uint16_t* feat, FeatSrc qf, FeatSrc pf, const int* d_flags,
                              cudaStream_t s)
{
    if (Q <= 0) return PMH_OK;
    const int blocks = ctx->sm_count * 16;  // persistent: pair chunks are handed out in turn
    // rows of at most 128 hashes that 16-byte loads can read, if the bands are whole lanes or lie
    // inside one; features only at K = 128 (a lane's hashes are then a feature's group)
    const bool bands_fit = !bandmask || P->rows <= 2 || P->rows % 4 == 0;
    const bool aligned = ((reinterpret_cast<uintptr_t>(qh) | reinterpret_cast<uintptr_t>(ph)) & 15) == 0;
    const bool short_rows = P->K % 4 == 0 && P->K <= kAgreeRowK && (!feat || P->K == 128) && bands_fit && aligned;
    auto fn = short_rows ? (feat ? agree_short_kernel<true> : agree_short_kernel<false>)
                         : (feat ? agree_rows_kernel<true> : agree_rows_kernel<false>);
    fn<<<blocks, kAgreeWarps * 32, 0, s>>>(qh, ph, row_ptr, cand, Q, cap, (int)P->K, (int)P->bands, (int)P->rows,
                                           P->T, count, bandmask, reinterpret_cast<__nv_bfloat16*>(feat), qf,
                                           pf, d_flags);
    PMH_LAUNCHED(short_rows ? "agree_short_kernel" : "agree_rows_kernel");
    return PMH_OK;
}

int pmh_launch_topm(const int64_t* row_ptr, const int32_t* cand, const uint16_t* count,
                    const float* score, int64_t Q, int32_t m, int K, int32_t* out_ids, int32_t* out_n,
                    const int* d_flags, cudaStream_t s)
{
    if (Q <= 0) return PMH_OK;
    int cap = 1;
    while (cap < m + kTopChunk || cap < kSelMax) cap <<= 1;
    const int kb = (K > 0 && K <= kMaxK) ? K : kMaxK;  // counts are <= K
    const size_t smem = sizeof(uint64_t) * cap + sizeof(int) * (size_t)(kb + 1);
    // (the largest list's and histogram's: the attribute is shared by all host threads, and a call
    // that set its own could lower it between another's set and its launch)
    PMH_CUDA_TRY(cudaFuncSetAttribute(topm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTopSmemMax));
    // large batches: the short rows a warp each, then a block per longer row (a batch of a few
    // hundred rows fills the device either way and saves the launch)
    const bool split = Q >= 512;
    if (split) {
        topm_short_kernel<<<(unsigned)((Q + kShortWarps - 1) / kShortWarps), kShortWarps * 32, 0, s>>>(
            row_ptr, cand, count, score, Q, kb, m, out_ids, out_n, d_flags);
        PMH_LAUNCHED("topm_short_kernel");
    }
    topm_kernel<<<(unsigned)Q, kTopThreads, smem, s>>>(row_ptr, cand, count, score, kb, m, cap,
                                                       split ? kShortRow + 1 : 0, out_ids, out_n, d_flags);
    PMH_LAUNCHED("topm_kernel");
    return PMH_OK;
}

extern "C" int pmh_jaccard_estimate(pmh_ctx ctx, const uint32_t* d_qhashes,
                                    const uint32_t* d_dbhashes, const int64_t* d_row_ptr,
                                    const int32_t* d_cand, int64_t Q, const pmh_params* params,
                                    uint16_t* d_count, uint32_t* d_bandmask, void* stream)
{
    PMH_TRY(pmh_check_device(ctx));
    PMH_TRY(pmh_check_params(params));
    if (Q < 0 || (Q > 0 && (!d_qhashes || !d_dbhashes || !d_row_ptr || !d_count)))
        return pmh_set_error(PMH_ERR_ARG, "bad arguments");
    return pmh_launch_agree(ctx, d_qhashes, d_dbhashes, d_row_ptr, d_cand, Q, INT64_MAX, params,
                            d_count, d_bandmask, nullptr, (cudaStream_t)stream);
}

extern "C" int pmh_topm(pmh_ctx ctx, const int64_t* d_row_ptr, const int32_t* d_cand,
                        const uint16_t* d_count, const float* d_score, int64_t Q, int32_t m,
                        int32_t* d_out_ids, int32_t* d_out_n, void* stream)
{
    PMH_TRY(pmh_check_device(ctx));
    if (Q < 0 || m < 1 || m > 1024 || (Q > 0 && (!d_row_ptr || !d_out_ids || !d_out_n)) ||
        (!d_count && !d_score))
        return pmh_set_error(PMH_ERR_ARG, "bad arguments (m in [1,1024])");
    if (Q > 0x7FFFFFFF) return pmh_set_error(PMH_ERR_ARG, "too many queries");
    return pmh_launch_topm(d_row_ptr, d_cand, d_count, d_score, Q, m, 0, d_out_ids, d_out_n, nullptr,
                           (cudaStream_t)stream);
}
