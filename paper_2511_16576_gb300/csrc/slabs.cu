// slabs.cu -- per-polygon y-slab edge index and cost order (part of step A0,
// used by the batching path of A1).
//
// The exact membership test of a point at height py only involves edges that
// straddle the horizontal line through it.  For a polygon with many vertices
// (coastline-like boundaries with up to 65,536 vertices) the y-range of its
// bounding box is cut into S equal slabs and every slab lists the edges whose
// row range [min(ay,by), max(ay,by)) meets it.  A test then reads one slab's
// list instead of all n edges; the parity of the crossings is order-independent,
// so the order inside a list does not matter.
//
// Layout (only polygons with n > kSlabMinVerts get slabs):
//   slab_info[p] = {slab_base, edge_base, S, slab_h | ymin}: see SlabInfo
//   slab_ptr[slab_base .. slab_base + S]  int32 offsets into the edge list
//   slab_edges[edge_base + ...]           int32 local edge ids (edge e = v_e -> v_e+1)
//
// The cost order sorts polygons by the expected number of stream points per
// hash, 2^32 / area (Theorem 2, E[h] = 1/S_p), largest first, so that the
// persistent signing grid starts the longest items first.
#include <algorithm>

#include "pmh_internal.cuh"

namespace {

// Per polygon (one warp, from the sizes that A0 left) count, prefix-sum and fill the slab
// lists: twice over the edges.  The counters of a polygon of at most kFillSmemSlabs slabs
// live in the warp's shared slice; those of a larger one in its slab table itself, whose
// entries the fill advances to the next slab's start and which is then moved up by one.
// Bound by the shared atomics and the scattered 4-byte stores (one per list entry).  400,000
// polygons of 8 to 1,024 vertices: 465 us (587 with counters reached through generic addresses)
constexpr int kFillThreads = 256;
constexpr int kFillSmemSlabs = 512;

// f(slab, edge) for every slab of every edge of the ring
template <class F>
__device__ __forceinline__ void for_slab_entries(const int2* __restrict__ xy, int64_t b, int n, int y0,
                                                 uint64_t hm, int lane, const F& f)
{
    int carry = xy[b + n - 1].y;
    for (int e0 = 0; e0 < n; e0 += 128) {
        int ay[4], by[4];
        ring_edge_ys(xy, b, n, e0, lane, carry, ay, by);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = e0 + 32 * u + lane;
            if (i >= n || ay[u] == by[u]) continue;
            const int lo = slab_div(min(ay[u], by[u]) - y0, hm);
            const int hi = slab_div(max(ay[u], by[u]) - 1 - y0, hm);
            for (int s = lo; s <= hi; ++s) f(s, i == 0 ? n - 1 : i - 1);
        }
    }
    __syncwarp();
}

__global__ void __launch_bounds__(kFillThreads, 8) slab_fill_kernel(const int2* __restrict__ xy, const int64_t* __restrict__ off,
                                 int64_t n_polys, const int64_t* __restrict__ d_n, SlabInfo* __restrict__ info,
                                 const int64_t* __restrict__ ptr_base, const int64_t* __restrict__ edge_base,
                                 int32_t* slab_ptr, int64_t cap_ptr, int32_t* __restrict__ slab_edges,
                                 int64_t cap_edges)
{
    __shared__ int scur[kFillThreads / 32][kFillSmemSlabs + 1];
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    if (d_n) n_polys = min(n_polys, *d_n);
    for (int64_t p = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); p < n_polys;
         p += nwarps) {
        const SlabInfo si = info[p];
        const int S = si.S, y0 = si.ymin;
        if (S <= 0) continue;
        const int64_t b = off[p];
        const int n = (int)(off[p + 1] - b);
        const uint64_t hm = slab_div_magic(si.slab_h);
        const int64_t pb = ptr_base[p], eb = edge_base[p];
        if (ptr_base[p + 1] > cap_ptr || edge_base[p + 1] > cap_edges) {
            // the lists do not fit the fixed buffers: this polygon is tested over all its edges
            if (lane == 0) info[p].S = 0;
            continue;
        }
        if (lane == 0) {
            info[p].slab_base = pb;
            info[p].edge_base = eb;
        }
        int32_t* sp = slab_ptr + pb;
        int32_t* le = slab_edges + eb;
        const bool small = S <= kFillSmemSlabs;
        int* cur = scur[threadIdx.x >> 5];
        for (int s = lane; s <= S; s += 32) (small ? cur : sp)[s] = 0;
        __syncwarp();
        if (small) for_slab_entries(xy, b, n, y0, hm, lane, [&](int s, int) { atomicAdd(&cur[s], 1); });
        else for_slab_entries(xy, b, n, y0, hm, lane, [&](int s, int) { atomicAdd(&sp[s], 1); });
        // exclusive prefix over S + 1 entries, 32 at a time
        int carry = 0;
        for (int base = 0; base <= S; base += 32) {
            const int s = base + lane;
            const int v = s < S ? (small ? cur[s] : __ldcg(sp + s)) : 0;
            int x = v;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (s <= S) {
                sp[s] = carry + x - v;
                if (small) cur[s] = carry + x - v;
            }
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
        __syncwarp();
        if (small) {
            for_slab_entries(xy, b, n, y0, hm, lane, [&](int s, int e) { le[atomicAdd(&cur[s], 1)] = e; });
        } else {
            for_slab_entries(xy, b, n, y0, hm, lane, [&](int s, int e) { le[atomicAdd(&sp[s], 1)] = e; });
            // sp[s] is now the end of slab s: move it up to s + 1, from the top
            for (int base = (S - 1) & ~31; base >= 0; base -= 32) {
                const int s = base + lane;
                const int v = s < S ? __ldcg(sp + s) : 0;
                __syncwarp();
                if (s < S) sp[s + 1] = v;
                __syncwarp();
            }
            if (lane == 0) sp[0] = 0;
            __syncwarp();
        }
    }
}

// cost key: expected stream points per hash ~ 2^33 / |area2|, as orderable float bits,
// complemented so that an ascending sort puts the most expensive polygon first
__global__ void cost_key_kernel(const int64_t* __restrict__ area2, int64_t n,
                                uint32_t* __restrict__ keys, int32_t* __restrict__ ids)
{
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        long long a = area2[p];
        const float aa = (float)(a < 0 ? -a : a);
        const float cost = 8589934592.0f / fmaxf(aa, 1.0f);
        keys[p] = ~__float_as_uint(cost);  // positive floats order like their bits
        ids[p] = (int32_t)p;
    }
}

// Morton code of a point of the 2^16 lattice (x bits at even positions)
__device__ __forceinline__ uint32_t morton16(uint32_t x, uint32_t y)
{
    auto spread = [](uint32_t v) {
        v &= 0xFFFFu;
        v = (v | (v << 8)) & 0x00FF00FFu;
        v = (v | (v << 4)) & 0x0F0F0F0Fu;
        v = (v | (v << 2)) & 0x33333333u;
        v = (v | (v << 1)) & 0x55555555u;
        return v;
    };
    return spread(x) | (spread(y) << 1);
}

// class key: polygons of more than kChunkMinVerts vertices (class 2) first, by
// decreasing expected cost -- the signing launch splits them into 32-hash items
// and starts the longest first -- then the others above kStagedMaxVerts (class 1),
// by decreasing expected cost, then the staged polygons (class 0) in Morton order
// of their box centres -- warps running at the same time then read nearby cells of
// the stream index, which keeps them in L2; counts classes 0 and 1 into n_cls[0],
// n_cls[1] (one atomic per block: one per thread serialised on two words took 260 us of
// 400,000 polygons).  16 bits -- the class and a 128 x 128 grid, or the cost to 1.6% -- order
// the work as well as 32 and take half the sort's passes
__global__ void class_key_kernel(const int4* __restrict__ bbox, const int64_t* __restrict__ area2,
                                 const int64_t* __restrict__ off, int64_t n,
                                 uint32_t* __restrict__ keys, int32_t* __restrict__ ids,
                                 unsigned long long* __restrict__ n_cls)
{
    __shared__ int sc[2];
    if (threadIdx.x < 2) sc[threadIdx.x] = 0;
    __syncthreads();
    int c0 = 0, c1 = 0;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        const long long a = area2[p];
        const float aa = (float)(a < 0 ? -a : a);
        const float cost = 8589934592.0f / fmaxf(aa, 1.0f);
        const int4 bb = bbox[p];
        const int64_t nv = off[p + 1] - off[p];
        const int cls = nv > kChunkMinVerts ? 2 : nv > kStagedMaxVerts ? 1 : 0;
        uint32_t key;
        if (cls == 0) {
            const uint32_t cx = (uint32_t)min((bb.x + bb.z) >> 1, 65535);
            const uint32_t cy = (uint32_t)min((bb.y + bb.w) >> 1, 65535);
            key = (2u << 14) | (morton16(cx, cy) >> 18);
        } else {
            key = ((uint32_t)(2 - cls) << 14) | ((~__float_as_uint(cost) << 1) >> 18);
        }
        keys[p] = key;
        ids[p] = (int32_t)p;
        c0 += cls == 0;
        c1 += cls == 1;
    }
    if (c0) atomicAdd(&sc[0], c0);
    if (c1) atomicAdd(&sc[1], c1);
    __syncthreads();
    if (threadIdx.x < 2 && sc[threadIdx.x]) atomicAdd(&n_cls[threadIdx.x], (unsigned long long)sc[threadIdx.x]);
}

}  // namespace

// room for a set's slab tables and edge lists, in one allocation: exactly as much at first, an
// eighth more when a reload has to grow them
static int grow_lists(pmh_polys P, int64_t n_ptr, int64_t n_edges)
{
    n_edges = std::max<int64_t>(n_edges, 1);
    if (P->slab_ptr && P->cap_slab_ptr >= n_ptr && P->cap_slab_edges >= n_edges) return PMH_OK;
    if (P->slab_ptr) {
        n_ptr = std::max(n_ptr + n_ptr / 8, P->cap_slab_ptr);
        n_edges = std::max(n_edges + n_edges / 8, P->cap_slab_edges);
        cudaFree(P->slab_ptr);
    }
    P->slab_ptr = P->slab_edges = nullptr;
    P->cap_slab_ptr = P->cap_slab_edges = 0;
    if (cudaMalloc(&P->slab_ptr, sizeof(int32_t) * (size_t)(n_ptr + n_edges)) != cudaSuccess) {
        cudaGetLastError();
        P->slab_ptr = nullptr;
        return pmh_set_error(PMH_ERR_NOMEM, "slab index allocation failed (%lld entries)",
                             (long long)(n_ptr + n_edges));
    }
    P->slab_edges = P->slab_ptr + n_ptr;
    P->cap_slab_ptr = n_ptr;
    P->cap_slab_edges = n_edges;
    return PMH_OK;
}

int pmh_build_slabs(pmh_polys P, const int64_t* ptr_base, const int64_t* edge_base, int64_t n_ptr,
                    int64_t n_edges, cudaStream_t s)
{
    if (P->n == 0) return PMH_OK;
    if (n_ptr > 0) {
        PMH_TRY(grow_lists(P, n_ptr, n_edges));
        const int blocks = (int)std::min<int64_t>((P->n + 7) / 8, (int64_t)P->ctx->sm_count * 32);
        slab_fill_kernel<<<blocks, kFillThreads, 0, s>>>(P->xy, P->offsets, P->n, nullptr, P->slab_info,
                                                         ptr_base, edge_base, P->slab_ptr, P->cap_slab_ptr,
                                                         P->slab_edges, P->cap_slab_edges);
        PMH_LAUNCHED("slab_fill_kernel");
    }
    // (from pinned memory, which the upload's last synchronisation frees)
    SlabPtrs* v = reinterpret_cast<SlabPtrs*>(P->ctx->h_pinned + 8);
    *v = SlabPtrs{P->slab_info, P->slab_ptr, P->slab_edges};
    PMH_CUDA_TRY(cudaMemcpyAsync(P->d_slabs, v, sizeof(*v), cudaMemcpyHostToDevice, s));
    return PMH_OK;
}

int pmh_build_cost_order(pmh_polys P, cudaStream_t s)
{
    pmh_ctx ctx = P->ctx;
    const int64_t n = P->n;
    if (n == 0) return PMH_OK;
    uint32_t* keys = nullptr;
    if (cudaMalloc(&P->order, sizeof(int32_t) * n) != cudaSuccess ||
        cudaMalloc(&keys, sizeof(uint32_t) * n) != cudaSuccess) {
        cudaGetLastError();
        if (keys) cudaFree(keys);
        return pmh_set_error(PMH_ERR_NOMEM, "cost order allocation failed");
    }
    int blocks = (int)std::min<int64_t>((n + 255) / 256, (int64_t)ctx->sm_count * 32);
    cost_key_kernel<<<blocks, 256, 0, s>>>(P->area2, n, keys, P->order);
    cudaError_t e = cudaGetLastError();
    g_pmh_launches.fetch_add(1);
    int rc = e == cudaSuccess ? pmh_radix_sort_u32(ctx, keys, P->order, n, 32, s)
                              : pmh_set_error(PMH_ERR_CUDA, "cost key: %s", cudaGetErrorString(e));
    const cudaError_t e2 = cudaStreamSynchronize(s);
    if (rc == PMH_OK && e2 != cudaSuccess)
        rc = pmh_set_error(PMH_ERR_CUDA, "cost order: %s", cudaGetErrorString(e2));
    cudaFree(keys);
    if (rc != PMH_OK) {
        cudaFree(P->order);
        P->order = nullptr;
    }
    return rc;
}

int pmh_build_class_order(pmh_polys P, cudaStream_t s)
{
    pmh_ctx ctx = P->ctx;
    const int64_t n = P->n;
    if (n == 0) return PMH_OK;
    // the class counts and the keys; the order's buffer stays the set's own
    unsigned long long* n_cls = nullptr;
    PMH_TRY(pmh_scratch(ctx, SCR_MISC, 2 * sizeof(unsigned long long) + sizeof(uint32_t) * (size_t)n,
                        (void**)&n_cls));
    uint32_t* keys = reinterpret_cast<uint32_t*>(n_cls + 2);
    P->order_cls = P->order_buf;
    PMH_CUDA_TRY(cudaMemsetAsync(n_cls, 0, 2 * sizeof(unsigned long long), s));
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, (int64_t)ctx->sm_count * 4);
    class_key_kernel<<<blocks, 256, 0, s>>>(P->bbox, P->area2, P->offsets, n, keys, P->order_cls, n_cls);
    PMH_LAUNCHED("class_key_kernel");
    PMH_TRY(pmh_radix_sort_u32(ctx, keys, P->order_cls, n, 16, s));
    PMH_CUDA_TRY(cudaMemcpyAsync(ctx->h_pinned, n_cls, 2 * sizeof(unsigned long long),
                                 cudaMemcpyDeviceToHost, s));
    PMH_CUDA_TRY(cudaStreamSynchronize(s));
    P->n_indexed = ctx->h_pinned[0];
    P->n_whole_cost = ctx->h_pinned[1];
    return PMH_OK;
}

// y-slab lists of a batch on fixed, caller-owned buffers, with no host
// synchronisation (for a captured pipeline): two exclusive scans of the sizes that A0
// wrote (zero past *d_n), and the lists of every polygon whose lists fit the
// buffers (slab_ptr: cap_ptr entries; slab_edges: cap_edges entries); a polygon
// whose lists do not fit gets S = 0 and is tested over all its edges.
// sizes: 2 * (max_polys + 1) entries; sums: pmh_scan_sums_size(max_polys).
int pmh_launch_slabs_fixed(pmh_ctx ctx, const int2* xy, const int64_t* off, int64_t max_polys,
                           const int64_t* d_n, SlabInfo* info, int64_t* sizes, int64_t* sums,
                           int32_t* slab_ptr, int64_t cap_ptr, int32_t* slab_edges, int64_t cap_edges,
                           cudaStream_t s)
{
    if (max_polys <= 0) return PMH_OK;
    int64_t* ptr_sizes = sizes;
    int64_t* edge_sizes = sizes + (max_polys + 1);
    PMH_TRY(pmh_exclusive_scan_i64(ctx, sizes, sizes, max_polys, s, sums, 2));
    const int blocks = (int)std::min<int64_t>((max_polys + 7) / 8, (int64_t)ctx->sm_count * 16);
    slab_fill_kernel<<<blocks, kFillThreads, 0, s>>>(xy, off, max_polys, d_n, info, ptr_sizes, edge_sizes,
                                                     slab_ptr, cap_ptr, slab_edges, cap_edges);
    PMH_LAUNCHED("slab_fill_kernel");
    return PMH_OK;
}
