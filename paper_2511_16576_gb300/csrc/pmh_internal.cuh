// pmh_internal.cuh -- internal declarations of the PolyMinHash CUDA library.
//
// Shared by the library's translation units only (never by the CPU oracle).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <string>
#include <vector>

#include "../../include/polyminhash.h"

// ---------------------------------------------------------------------------
// Error reporting
// ---------------------------------------------------------------------------
int pmh_set_error(int code, const char* fmt, ...);
#define PMH_CUDA_TRY(call)                                                              \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess)                                                          \
            return pmh_set_error(PMH_ERR_CUDA, "%s failed: %s (%s:%d)", #call,         \
                                 cudaGetErrorString(e_), __FILE__, __LINE__);          \
    } while (0)
#define PMH_TRY(expr)              \
    do {                           \
        int rc_ = (expr);          \
        if (rc_ != PMH_OK) return rc_; \
    } while (0)

extern std::atomic<int64_t> g_pmh_launches;
// launch bookkeeping: count every kernel launch and check the launch status
#define PMH_LAUNCHED(name)                                                              \
    do {                                                                                \
        g_pmh_launches.fetch_add(1, std::memory_order_relaxed);                         \
        cudaError_t e_ = cudaGetLastError();                                            \
        if (e_ != cudaSuccess)                                                          \
            return pmh_set_error(PMH_ERR_CUDA, "launch of %s failed: %s", name,         \
                                 cudaGetErrorString(e_));                               \
    } while (0)

// ---------------------------------------------------------------------------
// Handles
// ---------------------------------------------------------------------------
enum ScratchSlot {
    SCR_SORT_A = 0,
    SCR_SORT_B,
    SCR_SORT_HIST,
    SCR_SCAN,
    SCR_QUERY,
    SCR_REFINE,
    SCR_MISC,
    SCR_JOIN,
    SCR_COUNT
};

// Stream index (stream_index.cu): per level l a 2^index_level_gbits(l)-square grid over
// the domain (8^2 to 512^2 cells) and the first index_level_points(l) points of every
// hash's stream bucketed by its cells: half a point per (cell, hash) on average, and
// four on the finest level, whose polygons have no finer grid to go to.
constexpr int kIndexLevels = 7;
constexpr int kIndexMaxPoints = 1 << 20;  // the finest level
__host__ __device__ constexpr int index_level_gbits(int l) { return 3 + l; }
__host__ __device__ constexpr int index_level_points(int l)
{
    return l == kIndexLevels - 1 ? kIndexMaxPoints : 1 << (2 * index_level_gbits(l) - 1);
}
// a level is built only if its entry offsets (K * points) fit in 31 bits
__host__ __device__ constexpr bool index_level_fits(int l, int K)
{
    return (long long)K * index_level_points(l) <= (1ll << 31);
}
constexpr int kWalkKernelLevel = 4;  // the coarsest level that sign_kernel's indexed form reads (128^2)
// polygons of at most this many vertices are staged in shared memory by the
// signing kernels; larger ones are read through their y-slab edge index
constexpr int kStagedMaxVerts = 256;
// polygons above this many vertices are signed in (polygon, 32-hash chunk) items, so that
// a few very large polygons spread over many warps; smaller ones are signed whole (the
// staging, slab lists and coverage mask are then built once per polygon)
constexpr int kChunkMinVerts = 4096;

// Cost model of sign_kernel's indexed form for one polygon (clipped box bb, twice its
// area), in warp instructions per hash: the walk examines about 2^32 / area
// points, 128 per round of ~130 instructions; the indexed form reads the cells
// under the bounding box, and sees about lim * bbox / 2^32 candidates, with lim = 8 * 2^32 /
// area or all of the level's points; a hash without one below lim (e^(-lim / walk) of them) walks
// on from there.  Returns lim (0: walk) and the cheapest level: a longer walk belongs to a
// smaller polygon, so a finer grid lays no more cells under its box, but the finest level's
// tables do not fit the L2 cache.  K = 128, one level of 8,192 points before: 20,000 rings of 300
// to 1,000 vertices and 2e-5 of the domain 115 ms, 3.6; 5,000 of 300 to 4,000 and 1e-4 to 1e-3 1.55,
// 1.21.  (Polygons above the staged size, with coverage masks.)
struct WalkIndexPlan {
    uint32_t lim;
    int level;
};
__host__ __device__ __forceinline__ WalkIndexPlan pmh_walk_index_plan(int4 bb, long long area2, int K)
{
    // single precision: the estimate only picks a form and a limit (any limit
    // gives the exact result), and double precision is slow on this GPU
    WalkIndexPlan plan{0u, kWalkKernelLevel};
    if (bb.z <= bb.x || bb.w <= bb.y) return plan;
    const float area = 0.5f * (float)(area2 < 0 ? -area2 : area2);
    const float walk = 4294967296.0f / fmaxf(area, 1.0f);
    const float walk_cost = ceilf(walk * (1.0f / 128.0f)) * 130.0f;
    const float box = (float)(bb.z - bb.x) * (float)(bb.w - bb.y) * (1.0f / 4294967296.0f);
    float best = walk_cost;
    for (int l = kWalkKernelLevel; l < kIndexLevels && index_level_fits(l, K); ++l) {
        const int shift = 16 - index_level_gbits(l);
        const float cells = (float)((((bb.z - 1) >> shift) - (bb.x >> shift) + 1) *
                                    (((bb.w - 1) >> shift) - (bb.y >> shift) + 1));
        const float lim = fminf((float)index_level_points(l), 8.0f * walk + 256.0f);
        if (lim * box > 24.0f) continue;  // (too many candidates)
        const float cost = 40.0f + cells * (l == kIndexLevels - 1 ? 8.0f : 2.0f) + expf(-lim / walk) * walk_cost;
        if (cost < best) {
            best = cost;
            plan.lim = (uint32_t)lim;
            plan.level = l;
        }
    }
    return plan;
}

// Level of the indexed form for a polygon's clipped box (sign_unified.cu): the finest
// grid that lays at most kPlanCells cells, and at most 32 a side, under the box.  Per
// (cell, hash) the form reads one word, 128 hashes at a time, and only the points of
// boundary cells below the hash's bound cost more, so finer cells are the cheaper ones
// until the words read outweigh the points saved.  -1: an empty box.
constexpr int kPlanCells = 128;
__host__ __device__ __forceinline__ int pmh_index_level(int4 bb, int K)
{
    if (bb.z <= bb.x || bb.w <= bb.y) return -1;
    int level = 0;
    for (int l = 1; l < kIndexLevels && index_level_fits(l, K); ++l) {
        const int shift = 16 - index_level_gbits(l);
        const int cx = ((bb.z - 1) >> shift) - (bb.x >> shift) + 1, cy = ((bb.w - 1) >> shift) - (bb.y >> shift) + 1;
        if (cx > 32 || cy > 32 || cx * cy > kPlanCells) break;
        level = l;
    }
    return level;
}

struct StreamIndex {
    uint64_t build = 0;  // the context's count of builds (0: none); buffers' addresses come back
    uint64_t seed = 0;
    int K = 0;
    // rows of index_pitch(K) hashes per cell:
    uint32_t* first[kIndexLevels] = {};  // [G * G][pitch]: 2 * the smallest index of the stream in the cell, + 1
                                         // if the cell holds more of the level's points; all ones if none
    uint32_t* beg[kIndexLevels] = {};    // [G * G + 1][pitch]: the first entry of (cell, hash)
    uint2* ent[kIndexLevels] = {};       // [K * M] (stream index, x | y << 16) by (hash, cell, index)
};
// hashes per row of the index's tables: a multiple of four (16-byte reads)
__host__ __device__ constexpr int index_pitch(int K) { return (K + 3) & ~3; }
struct IndexLevelView {
    const uint32_t* first;
    const uint32_t* beg;
    const uint2* ent;
    int M, gbits, shift;
};
struct StreamIndexView {
    int K, pitch;
    IndexLevelView lv[kIndexLevels];  // lv[0].first nullptr: no index
};

// Walks that the indexed form leaves over: a hash without a point below its level's
// limit, queued by the signing launches and walked by sign_walks_kernel.
struct WalkItem {
    int32_t p, k;    // polygon, hash
    uint32_t start;  // first stream index to examine
    uint32_t next;   // segments handed out
};
constexpr int kWalkItems = 32768;  // (beyond them a hash is marked in the output and found there)
// device counters of a signing call: [0] work-queue ticket, [1] queued walks, [2] walk ticket,
// [3] ticket of the marked hashes
constexpr int kSignTickets = 4;
struct WalkQueue {
    WalkItem* items;
    unsigned long long* tickets;  // [kSignTickets]
};

struct pmh_ctx_s {
    int device = 0;
    int sm_count = 0;
    int* d_status = nullptr;              // device status word (0 = ok)
    unsigned long long* d_tickets = nullptr;  // work-queue tickets [64]
    WalkItem* walks = nullptr;                // [kWalkItems]
    void* scratch[SCR_COUNT] = {};
    size_t scratch_bytes[SCR_COUNT] = {};
    int64_t* h_pinned = nullptr;          // small pinned host buffer [64]
    int sign_variant = -1;                // autotuned signing kernel (-1 = default)
    StreamIndex sindex;                   // cached stream index (PMH_FLAG_STREAM_INDEX)
    uint64_t sindex_builds = 0;
    int sign_timing = 0;                  // record per-kernel events in pmh_minhash_sign
    int sign_count = 1;                   // signing launches record their work counts
    std::vector<cudaEvent_t> sign_ev;     // three per recorded call
    size_t sign_ev_used = 0;
};

int pmh_stream_index_get(pmh_ctx ctx, const pmh_params* P, cudaStream_t s, StreamIndexView* out);

// per-polygon y-slab edge index (slabs.cu); S == 0 for polygons without one
struct SlabInfo {
    int64_t slab_base;  // first entry of the polygon's slab table in slab_ptr
    int64_t edge_base;  // first entry of its edge lists in slab_edges
    int32_t S;          // number of slabs
    int32_t slab_h;     // slab height (rows)
    int32_t ymin;       // lowest vertex y
};
constexpr int kSlabMinVerts = 256;  // polygons above this size get a slab index
// a set's slab index as kernels find it through a device-resident word: a reload rebuilds
// the arrays, and a captured graph that refines against the set reads the current ones
struct SlabPtrs {
    const SlabInfo* info;
    const int32_t* ptr;
    const int32_t* edges;
};
// floor(x / h) by a multiply: with m = floor(2^40 / h) + 1 (slab_div_magic), x * m / 2^40
// exceeds x / h by less than x / 2^40 < 2^-18 for x < 2^22, which is below the gap 1/h
// between x / h and the next integer for every h < 2^18 (slab heights here are at most
// 2^21 / 64 for polygons above 256 vertices, or 1), so the floor is exact
__host__ __device__ __forceinline__ uint64_t slab_div_magic(int h) { return (1ull << 40) / (uint64_t)h + 1ull; }
__host__ __device__ __forceinline__ int slab_div(int x, uint64_t m) { return (int)(((uint64_t)x * m) >> 40); }
// slabs of a polygon of n vertices and the given height
__host__ __device__ __forceinline__ int slab_count_for(int n, int height)
{
    int s = n / 4;
    s = s > 1 ? s : 1;
    const int hmax = height > 1 ? height : 1;
    s = s < hmax ? s : hmax;
    return s < (1 << 16) ? s : 1 << 16;
}
// where A0 writes the sizes of each polygon's slab table (S + 1) and edge lists (zero for
// polygons without an index)
struct SlabSizes {
    SlabInfo* info = nullptr;
    int64_t* ptr = nullptr;
    int64_t* edge = nullptr;
};
#ifdef __CUDACC__
// y of the two end points of the edges that end at vertices e0 + 32u + lane (u < 4) of the ring
// of n vertices at xy + b, four loads in flight per lane: an edge starts at the lane before's
// vertex (a rotation; lane 0 takes the round before's last one, first the ring's last vertex).
// Edge id of the edge that ends at vertex i: i - 1, or n - 1 for i = 0
__device__ __forceinline__ void ring_edge_ys(const int2* __restrict__ xy, int64_t b, int n, int e0, int lane,
                                             int& carry, int (&ay)[4], int (&by)[4])
{
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int i = e0 + 32 * u + lane;
        by[u] = i < n ? xy[b + i].y : 0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int r = __shfl_sync(0xffffffffu, by[u], (lane + 31) & 31);
        ay[u] = lane == 0 ? carry : r;
        carry = r;
    }
}
#endif

// Handles record their device so that they can be released after their context.
struct pmh_polys_s {
    pmh_ctx ctx = nullptr;
    int device = 0;
    int64_t n = 0, nv = 0;
    void* arrays = nullptr;    // one allocation: the arrays below, slab_info, d_slabs and the class order
    int2* xy = nullptr;
    int64_t* offsets = nullptr;
    int4* bbox = nullptr;      // x0, y0, x1, y1 half-open, clipped to the domain
    int64_t* area2 = nullptr;  // twice the signed area
    int32_t max_n = 0;         // largest vertex count
    float2* feat = nullptr;         // [n] log2(area) / 32, log2(n) / 16 (reranker inputs)
    SlabInfo* slab_info = nullptr;  // [n]
    int32_t* slab_ptr = nullptr;    // (with the edges in one allocation, kept by a reload while its lists fit)
    int32_t* slab_edges = nullptr;
    int64_t cap_slab_ptr = 0, cap_slab_edges = 0;
    SlabPtrs* d_slabs = nullptr;    // the three above, device-resident (rewritten by a reload)
    int32_t* order = nullptr;       // polygons by expected signing cost, largest first (built
                                    // on the first signing call without the stream index)
    int32_t* order_buf = nullptr;   // [n], the class order's
    int32_t* order_cls = nullptr;   // order_buf once built: the class order, polygons above kChunkMinVerts vertices, then
                                    // the others above kStagedMaxVerts, each by cost, then the
                                    // staged polygons (Morton order)
    int64_t n_indexed = 0;          // class 0: <= kStagedMaxVerts vertices
    int64_t n_whole_cost = 0;       // class 1: the rest up to kChunkMinVerts vertices
    uint32_t* mask = nullptr;       // [n][16] coverage masks
};

// the slab lists of P from the exclusive scans of its SlabSizes, whose totals the host knows
int pmh_build_slabs(pmh_polys P, const int64_t* ptr_base, const int64_t* edge_base, int64_t n_ptr,
                    int64_t n_edges, cudaStream_t s);
int pmh_launch_slabs_fixed(pmh_ctx ctx, const int2* xy, const int64_t* off, int64_t max_polys,
                           const int64_t* d_n, SlabInfo* info, int64_t* sizes, int64_t* sums,
                           int32_t* slab_ptr, int64_t cap_ptr, int32_t* slab_edges, int64_t cap_edges,
                           cudaStream_t s);
int pmh_build_masks(pmh_polys P, cudaStream_t s);

// coverage masks (masks.cu): 16 x 16 cells of 2^cwl x 2^chl lattice units over the
// clipped bounding box; 2 bits per cell (0 outside, 1 inside, 2 boundary)
constexpr int kMaskMaxVerts = 256;
__host__ __device__ __forceinline__ int mask_cell_log2(int w)
{
    int a = (w + 15) >> 4, l = 0;
    while ((1 << l) < a) ++l;
    return l;
}
int pmh_build_cost_order(pmh_polys P, cudaStream_t s);   // P->order (walk form without the index)
int pmh_build_class_order(pmh_polys P, cudaStream_t s);  // P->order_cls and the class counts

struct pmh_index_s {
    pmh_ctx ctx = nullptr;
    int device = 0;
    int64_t n = 0;
    pmh_params params{};
    int band_bits = 0;
    uint32_t* hashes = nullptr;     // [n][K]
    uint32_t* sorted_comp = nullptr;  // [n * bands] composite (band, key) sort keys
    int32_t* sorted_id = nullptr;     // [n * bands]
    int64_t* dir = nullptr;  // directory of the sorted composites (directory.cuh)
    int dir_shift = 32;
};

// grow-only scratch buffer of the context
int pmh_scratch(pmh_ctx ctx, int slot, size_t bytes, void** out);
int pmh_check_params(const pmh_params* p);
int pmh_check_device(pmh_ctx ctx);

// ---------------------------------------------------------------------------
// Stream points (SplitMix64, Steele/Lea/Flood 2014)
// ---------------------------------------------------------------------------
#define PMH_GAMMA 0x9E3779B97F4A7C15ull
#define PMH_M1 0xBF58476D1CE4E5B9ull
#define PMH_M2 0x94D049BB133111EBull

__host__ __device__ __forceinline__ uint64_t pmh_mix64(uint64_t z)
{
    z = (z ^ (z >> 30)) * PMH_M1;
    z = (z ^ (z >> 27)) * PMH_M2;
    return z ^ (z >> 31);
}

// low 32 bits of the mix: all a lattice point needs (x = bits 0..15, y = 16..31)
__device__ __forceinline__ uint32_t pmh_mix64_lo(uint64_t z)
{
    z = (z ^ (z >> 30)) * PMH_M1;
    z = (z ^ (z >> 27)) * PMH_M2;
    return (uint32_t)(z ^ (z >> 31));
}

// ---------------------------------------------------------------------------
// Scans (scan.cu)
// ---------------------------------------------------------------------------
// exclusive prefix sum of n int64 values in place-able form: out[i] = sum in[0..i-1],
// out[n] = total (out has n + 1 entries).  in may alias out.
// sums_buffer (optional, pmh_scan_sums_size(n) entries) replaces the context scratch,
// so that a captured graph owns every buffer it touches.  arrays > 1: as many scans, the
// arrays n + 1 entries apart.
int pmh_exclusive_scan_i64(pmh_ctx ctx, const int64_t* in, int64_t* out, int64_t n,
                           cudaStream_t s, int64_t* sums_buffer = nullptr, int arrays = 1);
int64_t pmh_scan_sums_size(int64_t n);

// ---------------------------------------------------------------------------
// Internal launchers shared by the public calls and the captured query graph.
// d_n (optional): device-side count that caps the launch-time size n, so a graph
// captured for a maximum batch serves any smaller batch.  d_flags (optional):
// device status word; bits 0-2 = invalid polygons (set by prep: 1 offsets,
// 2 fewer than 3 vertices, 4 coordinate range), bit 3 = candidate overflow (set
// by the join).  Kernels after a failed stage do nothing.
// ---------------------------------------------------------------------------
int pmh_launch_prep(int sm_count, const int2* src, int2* dst, const int64_t* off, int64_t n_polys,
                    const int64_t* d_n, int64_t n_vertices, int4* bbox, int64_t* area2, SlabSizes sz,
                    int* status, cudaStream_t s);
int pmh_launch_sign(pmh_ctx ctx, const int2* xy, const int64_t* off, const int4* bbox,
                    const SlabInfo* slabs, const int32_t* slab_ptr, const int32_t* slab_edges,
                    const int32_t* order, const pmh_params* P, int64_t n_polys,
                    const int64_t* d_n, const int* d_flags, unsigned long long* ticket,
                    uint32_t* out, cudaStream_t s, const int64_t* area2 = nullptr,
                    const StreamIndexView* sidx = nullptr, const uint32_t* masks = nullptr,
                    const int32_t* order_cls = nullptr, int64_t n_indexed = 0,
                    int64_t n_whole_cost = 0);
// every polygon, in persistent launches (sign_unified.cu): slots list[0 ..
// n_slots) (list nullptr: slot = polygon id), the first n_chunked as (polygon,
// 32-hash chunk) items, the rest whole; d_n (optional) caps n_slots on the
// device, d_flags (optional) skips a batch that failed validation; U = points
// per lane per round of the walk form (2, 4 or 8); work (optional) the six
// work counters.  The last n_indexed_tail slots of a class list (staged polygons
// of the indexed form, the class order's last class) get a launch of their own
// through a build of the kernel without the other paths.  wq: the call's counters and
// the queue of leftover walks, which a last launch takes (with a stream index).
int pmh_launch_sign_unified(pmh_ctx ctx, int U, const int2* xy, const int64_t* off,
                            const int4* bbox, const int64_t* area2, const SlabInfo* slabs,
                            const int32_t* slab_ptr, const int32_t* slab_edges, const int32_t* list,
                            int64_t n_slots, int64_t n_chunked, int64_t n_indexed_tail,
                            const int64_t* d_n, const int* d_flags, const pmh_params* P,
                            const StreamIndexView& S, const WalkQueue& wq, uint32_t* out,
                            unsigned long long* work, cudaStream_t s);
// bucket join (lsh.cu): the count pass (write false: counts) or the fill pass (write
// true: the CSR rows).  `stage` (nullable, pmh_join_stage_bytes(Q, pool_ints) bytes,
// the same buffer for both passes, 16-byte aligned) lets the count pass keep the rows
// it sorted, up to pool_ints ids in all, so that the fill pass copies them; the fill
// pass of a call whose count pass had no stage gets none either.  With one band the
// stage holds the count pass's segment counts instead and both passes need it; a join
// that stages nothing asks for 0 bytes and takes nullptr
size_t pmh_join_stage_bytes(pmh_index X, int64_t Q, int64_t pool_ints);
int pmh_launch_query(pmh_index X, const uint32_t* qh, int64_t Q, const int64_t* d_n,
                     int64_t* counts, const int64_t* row_ptr, int32_t* cand, int64_t cap,
                     void* stage, int64_t pool_ints, int* d_flags, bool write, cudaStream_t s);
int pmh_launch_agree(pmh_ctx ctx, const uint32_t* qh, const uint32_t* ph, const int64_t* row_ptr,
                     const int32_t* cand, int64_t Q, int64_t cap, const pmh_params* P,
                     uint16_t* count, uint32_t* bandmask, const int* d_flags, cudaStream_t s);
// per-set inputs of the reranker's features: log features, boxes and twice the areas
struct FeatSrc {
    const float2* feat;
    const int4* bbox;
    const int64_t* area2;
};

// a pair's per-polygon inputs of its feature row
struct FeatPair {
    float2 qf, pf;       // (log2 area / 32, log2 vertex count / 16)
    int4 qb, pb;         // bounding boxes
    long long qa2, pa2;  // twice the signed areas
};
__device__ __forceinline__ FeatPair pmh_feat_pair(const FeatSrc& qf, const FeatSrc& pf, int64_t q, int64_t p)
{
    return FeatPair{qf.feat[q], pf.feat[p], qf.bbox[q], pf.bbox[p], qf.area2[q], pf.area2[p]};
}

// Column 32 + col (col < 16) of the reranker's feature row of a pair (A7) from its
// comparison counts over the K hashes -- c equal (and not the sentinel), lt / gt
// lower / higher than the candidate's -- and the two polygons' inputs; 40..47 are
// zero.  Every kernel that writes feature rows takes these values from here, so all
// feed the network the same bf16 values.
__device__ __forceinline__ float pmh_feature_col(int col, int K, int c, int lt, int gt, const FeatPair& in)
{
    switch (col) {
    case 0: return (float)c / (float)K;
    case 1: return in.qf.x;
    case 2: return in.pf.x;
    case 3: return in.qf.y;
    case 4: return in.pf.y;
    case 5: return (float)lt / (float)K;
    case 6: return (float)gt / (float)K;
    case 7: {
        // upper bound of J: the intersection is at most min(|q|, |p|, overlap of the
        // two bounding boxes)
        const int4 qb = in.qb, pb = in.pb;
        const float ow = (float)max(0, min(qb.z, pb.z) - max(qb.x, pb.x));
        const float oh = (float)max(0, min(qb.w, pb.w) - max(qb.y, pb.y));
        const long long qa = in.qa2, pa = in.pa2;
        const float a = 0.5f * (float)(qa < 0 ? -qa : qa);
        const float bq = 0.5f * (float)(pa < 0 ? -pa : pa);
        const float mn = fminf(fminf(a, bq), ow * oh);
        const float den = a + bq - mn;
        return den > 0.f ? mn / den : 0.f;
    }
    default: return 0.f;
    }
}

// The feature row of a pair, one warp per pair: eq = K / 32 equality words (bit
// k % 32 of word k / 32 set iff h_k(q) = h_k(p) != T).  Lane l returns column l
// (all K / 32 hashes of group l equal) in lo and, for l < 16, column 32 + l in hi.
__device__ __forceinline__ void pmh_feature_values(const uint32_t* eq, int K, int c, int lt, int gt,
                                                   const FeatPair& in, int lane, float& lo, float& hi)
{
    const int g = K / 32;
    bool all = true;
    for (int t = 0; t < g && all; ++t) {
        const int k = lane * g + t;
        all = (eq[k >> 5] >> (k & 31)) & 1u;
    }
    lo = all ? 1.f : 0.f;
    hi = pmh_feature_col(lane, K, c, lt, gt, in);
}
int pmh_launch_agree_features(pmh_ctx ctx, const uint32_t* qh, const uint32_t* ph,
                              const int64_t* row_ptr, const int32_t* cand, int64_t Q, int64_t cap,
                              const pmh_params* P, uint16_t* count, uint32_t* bandmask,
                              uint16_t* feat, FeatSrc qf, FeatSrc pf, const int* d_flags,
                              cudaStream_t s);
// exact refinement of fixed-width top-m lists (ids [Q][m], nlist [Q]) to the top-k by
// (J desc, id asc) (refine.cu); jv: Q * m doubles of scratch; tickets: the grids' three
// counters; d_n (optional) caps Q on the device.  big (pmh_refine_queue_bytes(Q * m);
// nullable) is the queue of the pairs with a ring above kRefineBigVerts vertices, which
// then go to a cluster each; without it every pair takes the two-warp form.
struct RefineQueries {
    const int2* xy;
    const int64_t* off;
    const int64_t* area2;
    const int4* box;
    const SlabPtrs* slabs;  // nullptr: no slab lists
};
constexpr int kRefineBigVerts = 1024;
size_t pmh_refine_queue_bytes(int64_t n_pairs);
const void* pmh_refine_big_func();  // the kernel that takes the queue (a no-op when it is empty)
int pmh_launch_refine_topk(pmh_ctx ctx, const RefineQueries& qs, pmh_polys db, const int32_t* ids,
                           const int32_t* nlist, int64_t Q, const int64_t* d_n, int32_t m, int32_t k,
                           double* jv, unsigned long long* tickets, int32_t* big, int32_t* top_ids,
                           double* top_j, cudaStream_t s);
// fixed-width lists ids [Q][m] with counts n [Q] to compact CSR (row_ptr [Q + 1], cand);
// rows at or past *d_q (optional) are empty; counts: Q entries of scratch; sums: the
// scan's partial sums (pmh_scan_sums_size(Q) entries; nullptr: context scratch)
int pmh_launch_lists_to_csr(pmh_ctx ctx, const int32_t* ids, const int32_t* n, int64_t Q, int32_t m,
                            const int64_t* d_q, int64_t* counts, int64_t* sums, int64_t* row_ptr,
                            int32_t* cand, cudaStream_t s);
// per-polygon reranker inputs (log2 area / 32, log2 vertex count / 16) of polygons
// [0, n) (capped by *d_n when given)
int pmh_launch_poly_feat(int sm_count, const int64_t* area2, const int64_t* off, int64_t n,
                         const int64_t* d_n, float2* out, cudaStream_t s);
// reranker scores of n feature rows (rerank.cu)
int pmh_launch_rerank_forward(pmh_rerank r, const uint16_t* feat, int64_t n_rows, float* score,
                              int* d_flags, cudaStream_t s);
// the learned form's features, scores and top-m in one launch (rerank.cu): shortlist
// ids [Q][S] / counts n[Q] (top-S by count) to ids [Q][m] (-1 padded) and counts
// [Q] by (predicted Jaccard desc, id asc); S must divide 128 (S >= 4), K % 32 == 0
bool pmh_rerank_select_fits(int S, int K);
int pmh_launch_rerank_select(pmh_rerank r, const uint32_t* qh, const uint32_t* ph, const int32_t* sl_ids,
                             const int32_t* sl_n, int64_t Q, const int64_t* d_n, int S, int m,
                             const pmh_params* P, FeatSrc qf, FeatSrc pf, int32_t* out_ids, int32_t* out_n,
                             int* d_flags, cudaStream_t s);
// top-m per row (estimate.cu); K bounds the counts (0: up to 4,096)
int pmh_launch_topm(const int64_t* row_ptr, const int32_t* cand, const uint16_t* count,
                    const float* score, int64_t Q, int32_t m, int K, int32_t* out_ids, int32_t* out_n,
                    const int* d_flags, cudaStream_t s);

// signing kernel variants (points per lane per round x warps per block)
int pmh_sign_variant_count();
void pmh_sign_variant_shape(int v, int* points_per_lane, int* warps);

// stable LSD radix sort of (uint32 key, int32 value) pairs; result in keys/vals.
int pmh_radix_sort_u32(pmh_ctx ctx, uint32_t* keys, int32_t* vals, int64_t n, int key_bits,
                       cudaStream_t s);

// warp helpers
__device__ __forceinline__ unsigned pmh_lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}
