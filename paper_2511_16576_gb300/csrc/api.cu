// api.cu -- contexts, errors, scratch memory and polygon upload (step A0).
//
// A0 follows Sec. 3.1 of the paper (per-polygon local MBR) with the fixed
// 65536^2 lattice as the global MBR; it also computes twice the signed area
// (exact int64 shoelace) for the refinement and the reranker features.
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <climits>

#include "pmh_internal.cuh"
#include "upload.cuh"

std::atomic<int64_t> g_pmh_launches{0};

static thread_local char g_err[512] = "";

int pmh_set_error(int code, const char* fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return code;
}

extern "C" const char* pmh_last_error(void) { return g_err; }
extern "C" int pmh_version(void) { return 10000; }
extern "C" int64_t pmh_launch_count(void) { return g_pmh_launches.load(); }

int pmh_check_device(pmh_ctx ctx)
{
    if (!ctx) return pmh_set_error(PMH_ERR_ARG, "null context");
    cudaGetLastError();  // a stale error of an earlier, unrelated call must not fail this one
    PMH_CUDA_TRY(cudaSetDevice(ctx->device));
    return PMH_OK;
}

int pmh_check_params(const pmh_params* p)
{
    if (!p) return pmh_set_error(PMH_ERR_ARG, "null params");
    if (p->K < 1 || p->K > 4096) return pmh_set_error(PMH_ERR_ARG, "K=%u not in [1,4096]", p->K);
    if (p->T < 1 || p->T > (1u << 31)) return pmh_set_error(PMH_ERR_ARG, "T=%u not in [1,2^31]", p->T);
    if (p->bands < 1 || p->bands > 128 || p->K % p->bands != 0 || p->rows != p->K / p->bands)
        return pmh_set_error(PMH_ERR_ARG, "bands=%u rows=%u do not split K=%u (bands <= 128)",
                             p->bands, p->rows, p->K);
    return PMH_OK;
}

int pmh_scratch(pmh_ctx ctx, int slot, size_t bytes, void** out)
{
    if (bytes == 0) bytes = 256;
    if (ctx->scratch_bytes[slot] < bytes) {
        if (ctx->scratch[slot]) {
            PMH_CUDA_TRY(cudaDeviceSynchronize());
            cudaFree(ctx->scratch[slot]);
            ctx->scratch[slot] = nullptr;
            ctx->scratch_bytes[slot] = 0;
        }
        size_t want = bytes + bytes / 4;
        if (cudaMalloc(&ctx->scratch[slot], want) != cudaSuccess) {
            cudaGetLastError();
            return pmh_set_error(PMH_ERR_NOMEM, "scratch allocation of %zu bytes failed", want);
        }
        ctx->scratch_bytes[slot] = want;
    }
    *out = ctx->scratch[slot];
    return PMH_OK;
}

extern "C" int pmh_create(pmh_ctx* out, int device)
{
    if (!out) return pmh_set_error(PMH_ERR_ARG, "null out");
    *out = nullptr;
    int count = 0;
    PMH_CUDA_TRY(cudaGetDeviceCount(&count));
    if (device < 0 || device >= count)
        return pmh_set_error(PMH_ERR_ARG, "device %d not in [0,%d)", device, count);
    cudaDeviceProp prop;
    PMH_CUDA_TRY(cudaGetDeviceProperties(&prop, device));
    if (prop.major != 10 || prop.minor != 3)
        return pmh_set_error(PMH_ERR_CUDA, "device %d is sm_%d%d; this library is built for sm_103a",
                             device, prop.major, prop.minor);
    PMH_CUDA_TRY(cudaSetDevice(device));
    pmh_ctx c = new pmh_ctx_s();
    c->device = device;
    c->sm_count = prop.multiProcessorCount;
    if (cudaMalloc(&c->d_status, 64 * sizeof(int)) != cudaSuccess ||
        cudaMalloc(&c->d_tickets, 64 * sizeof(unsigned long long)) != cudaSuccess ||
        cudaMalloc(&c->walks, sizeof(WalkItem) * kWalkItems) != cudaSuccess ||
        cudaMallocHost(&c->h_pinned, 64 * sizeof(int64_t)) != cudaSuccess) {
        cudaGetLastError();
        pmh_destroy(c);
        return pmh_set_error(PMH_ERR_NOMEM, "context allocation failed");
    }
    cudaMemset(c->d_status, 0, 64 * sizeof(int));
    cudaMemset(c->d_tickets, 0, 64 * sizeof(unsigned long long));
    PMH_CUDA_TRY(cudaDeviceSynchronize());
    *out = c;
    return PMH_OK;
}

extern "C" int pmh_destroy(pmh_ctx ctx)
{
    if (!ctx) return PMH_OK;
    cudaSetDevice(ctx->device);
    cudaDeviceSynchronize();
    for (int i = 0; i < SCR_COUNT; ++i)
        if (ctx->scratch[i]) cudaFree(ctx->scratch[i]);
    if (ctx->d_status) cudaFree(ctx->d_status);
    if (ctx->d_tickets) cudaFree(ctx->d_tickets);
    if (ctx->walks) cudaFree(ctx->walks);
    if (ctx->h_pinned) cudaFreeHost(ctx->h_pinned);
    for (cudaEvent_t e : ctx->sign_ev) cudaEventDestroy(e);
    for (int l = 0; l < kIndexLevels; ++l) {
        if (ctx->sindex.first[l]) cudaFree(ctx->sindex.first[l]);
        if (ctx->sindex.beg[l]) cudaFree(ctx->sindex.beg[l]);
        if (ctx->sindex.ent[l]) cudaFree(ctx->sindex.ent[l]);
    }
    delete ctx;
    return PMH_OK;
}

// ---------------------------------------------------------------------------
// A0: per-polygon preparation.  One warp per polygon: validation, bbox
// (clipped to the lattice domain, half-open), twice the signed area.
// status[0] |= 1 bad offsets, 2 < 3 vertices, 4 coordinate out of range;
// status[1] = max vertex count.
//
// kCopy: the vertices are copied from src to dst on the way (a device-to-device upload).
// sz.info: the sizes of every polygon's slab index too, from a second look at vertices that
// the caches still hold.
// Bound by memory at large sets (each vertex is read once, written once under kCopy): a
// lane keeps four vertices in flight, and an edge's start vertex is the lane before's (a
// rotation), so that no vertex is loaded twice.  400,000 polygons of 8 to 1,024 vertices (0.7 GB):
// 352 us; before, 297 us of preparation and 202 us of sizes followed a copy of the vertices
// ---------------------------------------------------------------------------
template <bool kCopy>
__global__ void __launch_bounds__(256, 6)
prep_kernel(const int2* __restrict__ src, int2* __restrict__ dst, const int64_t* __restrict__ off,
            int64_t n_polys, const int64_t* __restrict__ d_n, int64_t n_vertices,
            int4* __restrict__ bbox, int64_t* __restrict__ area2, SlabSizes sz, int* __restrict__ status)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    // (slots at or past the device-side count get empty sizes)
    const int64_t n_live = d_n ? min(n_polys, *d_n) : n_polys;
    const int LIM = 1 << 20;
    int nmax = 0;  // largest vertex count of the warp's polygons (one atomic at the end)
    for (int64_t p = warp; p < n_polys; p += nwarps) {
        SlabInfo si{0, 0, 0, 1, 0};
        long long entries = 0;
        if (p < n_live) {
            const int64_t b = off[p], e = off[p + 1];
            int flags = 0;
            if (b < 0 || e > n_vertices || e < b) flags |= 1;
            const int64_t n = e - b;
            if (n < 3) flags |= 2;
            if (flags) {
                if (lane == 0) {
                    atomicOr(&status[0], flags);
                    bbox[p] = make_int4(0, 0, 0, 0);
                    area2[p] = 0;
                }
            } else {
                int x0 = INT_MAX, y0 = INT_MAX, x1 = INT_MIN, y1 = INT_MIN;
                long long a2 = 0;
                int2 carry = src[e - 1];
                for (int64_t i0 = 0; i0 < n; i0 += 128) {
                    int2 v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int64_t i = i0 + 32 * u + lane;
                        v[u] = i < n ? src[b + i] : make_int2(0, 0);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int64_t i = i0 + 32 * u + lane;
                        const int rx = __shfl_sync(0xffffffffu, v[u].x, (lane + 31) & 31);
                        const int ry = __shfl_sync(0xffffffffu, v[u].y, (lane + 31) & 31);
                        const int wx = lane == 0 ? carry.x : rx, wy = lane == 0 ? carry.y : ry;
                        carry = make_int2(rx, ry);
                        if (i < n) {
                            if (kCopy) dst[b + i] = v[u];
                            x0 = min(x0, v[u].x);
                            x1 = max(x1, v[u].x);
                            y0 = min(y0, v[u].y);
                            y1 = max(y1, v[u].y);
                            a2 += (long long)wx * v[u].y - (long long)v[u].x * wy;
                        }
                    }
                }
                x0 = __reduce_min_sync(0xffffffffu, x0);
                y0 = __reduce_min_sync(0xffffffffu, y0);
                x1 = __reduce_max_sync(0xffffffffu, x1);
                y1 = __reduce_max_sync(0xffffffffu, y1);
                for (int o = 16; o > 0; o >>= 1) a2 += __shfl_xor_sync(0xffffffffu, a2, o);
                const bool bad = x0 < -LIM || x1 > LIM || y0 < -LIM || y1 > LIM;
                if (lane == 0) {
                    if (bad) atomicOr(&status[0], 4);
                    // clip to the lattice domain [0, 65536)
                    int cx0 = max(x0, 0), cy0 = max(y0, 0), cx1 = min(x1, 65536), cy1 = min(y1, 65536);
                    if (cx1 < cx0) cx1 = cx0;
                    if (cy1 < cy0) cy1 = cy0;
                    bbox[p] = make_int4(cx0, cy0, cx1, cy1);
                    area2[p] = a2;
                    nmax = max(nmax, (int)(n < INT_MAX ? n : INT_MAX));
                }
                if (sz.info && n > kSlabMinVerts && n <= INT_MAX && !bad) {
                    const int nv = (int)n, S = slab_count_for(nv, y1 - y0);
                    const int h = max((y1 - y0 + S - 1) / S, 1);
                    const uint64_t hm = slab_div_magic(h);
                    int cy = src[e - 1].y;
                    for (int e0 = 0; e0 < nv; e0 += 128) {
                        int ay[4], by[4];
                        ring_edge_ys(src, b, nv, e0, lane, cy, ay, by);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            if (e0 + 32 * u + lane >= nv || ay[u] == by[u]) continue;
                            const int lo = min(ay[u], by[u]) - y0, hi = max(ay[u], by[u]) - 1 - y0;
                            entries += slab_div(hi, hm) - slab_div(lo, hm) + 1;
                        }
                    }
                    for (int o = 16; o > 0; o >>= 1) entries += __shfl_xor_sync(0xffffffffu, entries, o);
                    si = SlabInfo{0, 0, S, h, y0};
                }
            }
        }
        if (sz.info && lane == 0) {
            sz.info[p] = si;
            sz.ptr[p] = si.S > 0 ? si.S + 1 : 0;
            sz.edge[p] = entries;
        }
    }
    if (lane == 0 && nmax > 0) atomicMax(&status[1], nmax);
}

int pmh_launch_prep(int sm_count, const int2* src, int2* dst, const int64_t* off, int64_t n_polys,
                    const int64_t* d_n, int64_t n_vertices, int4* bbox, int64_t* area2, SlabSizes sz,
                    int* status, cudaStream_t s)
{
    if (n_polys <= 0) return PMH_OK;
    const int blocks = (int)std::min<int64_t>((n_polys + 7) / 8, (int64_t)sm_count * 32);
    auto fn = dst ? prep_kernel<true> : prep_kernel<false>;
    fn<<<blocks, 256, 0, s>>>(src, dst, off, n_polys, d_n, n_vertices, bbox, area2, sz, status);
    PMH_LAUNCHED("prep_kernel");
    return PMH_OK;
}

// per-polygon reranker inputs: log2(area) / 32 and log2(vertex count) / 16 (polygons
// below the device-side count d_n, when given)
__global__ void poly_feat_kernel(const int64_t* __restrict__ area2, const int64_t* __restrict__ off,
                                 int64_t n, const int64_t* __restrict__ d_n, float2* __restrict__ out)
{
    if (d_n) n = min(n, *d_n);
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        const long long a2 = area2[p];
        const double a = 0.5 * (double)(a2 < 0 ? -a2 : a2);
        out[p] = make_float2(log2f((float)(a > 1.0 ? a : 1.0)) / 32.f,
                             log2f((float)(off[p + 1] - off[p])) / 16.f);
    }
}

static_assert(kPointerOnDevice == cudaMemoryTypeDevice, "upload.cuh's memory type");

// copy the arrays in, validate them and compute every per-polygon product (bbox,
// 2 x area, reranker inputs, slab lists, class order) into P's buffers
static int upload_fill(pmh_polys P, const int32_t* xy, const int64_t* offsets, bool host,
                       cudaStream_t s)
{
    pmh_ctx ctx = P->ctx;
    const int64_t n_polys = P->n, n_vertices = P->nv;
    cudaMemcpyKind kind = host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
    // vertices that lie on this device are copied by the kernel that reads them (upload.cuh)
    bool fused = false;
    if (!host && n_polys > 0) {
        cudaPointerAttributes at{};
        if (cudaPointerGetAttributes(&at, xy) == cudaSuccess)
            fused = pmh_reads_in_place((int)at.type, at.device, ctx->device, reinterpret_cast<uintptr_t>(xy));
        else
            cudaGetLastError();
    }
    cudaError_t e = cudaSuccess;
    if (n_vertices > 0 && !fused) e = cudaMemcpyAsync(P->xy, xy, sizeof(int2) * n_vertices, kind, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(P->offsets, offsets, sizeof(int64_t) * (n_polys + 1), kind, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(ctx->d_status, 0, 2 * sizeof(int), s);
    if (e != cudaSuccess) return pmh_set_error(PMH_ERR_CUDA, "upload copy failed: %s", cudaGetErrorString(e));
    // offsets[0] and offsets[n] are checked by the kernel through b/e bounds
    int64_t* sizes = nullptr;
    if (n_polys > 0) {
        PMH_TRY(pmh_scratch(ctx, SCR_MISC, sizeof(int64_t) * (size_t)(2 * (n_polys + 1)), (void**)&sizes));
        int64_t* edge = sizes + n_polys + 1;
        PMH_TRY(pmh_launch_prep(ctx->sm_count, fused ? reinterpret_cast<const int2*>(xy) : P->xy,
                                fused ? P->xy : nullptr, P->offsets, n_polys, nullptr, n_vertices, P->bbox,
                                P->area2, SlabSizes{P->slab_info, sizes, edge}, ctx->d_status, s));
        PMH_TRY(pmh_exclusive_scan_i64(ctx, sizes, sizes, n_polys, s, nullptr, 2));  // sizes, edge
        e = cudaMemcpyAsync(ctx->h_pinned + 1, sizes + n_polys, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(ctx->h_pinned + 2, edge + n_polys, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
        if (e != cudaSuccess) return pmh_set_error(PMH_ERR_CUDA, "upload failed: %s", cudaGetErrorString(e));
    }
    int st[2] = {0, 0};
    e = cudaMemcpyAsync(ctx->h_pinned, ctx->d_status, 2 * sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return pmh_set_error(PMH_ERR_CUDA, "upload failed: %s", cudaGetErrorString(e));
    memcpy(st, ctx->h_pinned, sizeof(st));
    if (st[0] & 1) return pmh_set_error(PMH_ERR_RANGE, "offsets are not increasing / in range");
    if (st[0] & 2) return pmh_set_error(PMH_ERR_RANGE, "a polygon has fewer than 3 vertices");
    if (st[0] & 4) return pmh_set_error(PMH_ERR_RANGE, "a coordinate exceeds |2^20|");
    P->max_n = st[1];
    const int64_t n_ptr = n_polys > 0 ? ctx->h_pinned[1] : 0, n_edges = n_polys > 0 ? ctx->h_pinned[2] : 0;
    if (n_polys > 0) {
        int blocks = (int)std::min<int64_t>((n_polys + 255) / 256, (int64_t)ctx->sm_count * 32);
        poly_feat_kernel<<<blocks, 256, 0, s>>>(P->area2, P->offsets, n_polys, nullptr, P->feat);
        g_pmh_launches.fetch_add(1);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return pmh_set_error(PMH_ERR_CUDA, "feature kernel: %s", cudaGetErrorString(e));
    }
    PMH_TRY(pmh_build_slabs(P, sizes, sizes + n_polys + 1, n_ptr, n_edges, s));
    return pmh_build_class_order(P, s);
}

int pmh_launch_poly_feat(int sm_count, const int64_t* area2, const int64_t* off, int64_t n,
                         const int64_t* d_n, float2* out, cudaStream_t s)
{
    if (n <= 0) return PMH_OK;
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, (int64_t)sm_count * 32);
    poly_feat_kernel<<<blocks, 256, 0, s>>>(area2, off, n, d_n, out);
    PMH_LAUNCHED("poly_feat_kernel");
    return PMH_OK;
}

static int upload_common(pmh_ctx ctx, const int32_t* xy, const int64_t* offsets, int64_t n_polys,
                         int64_t n_vertices, bool host, pmh_polys* out, void* stream)
{
    if (!out) return pmh_set_error(PMH_ERR_ARG, "null out");
    *out = nullptr;
    PMH_TRY(pmh_check_device(ctx));
    if (n_polys < 0 || n_polys >= (1ll << 31) || n_vertices < 0 || (!xy && n_vertices > 0) ||
        !offsets)
        return pmh_set_error(PMH_ERR_ARG, "bad polygon arguments (n_polys=%lld n_vertices=%lld)",
                             (long long)n_polys, (long long)n_vertices);
    pmh_polys P = new pmh_polys_s();
    P->ctx = ctx;
    P->device = ctx->device;
    P->n = n_polys;
    P->nv = n_vertices;
    // every array of a size known now in one allocation (256-byte steps): an upload of a batch of
    // queries is mostly its allocations, which cost 80 us each where they take a new block of
    // the driver's (100,000 polygons of 8 to 64 vertices: 679 us with nine allocations, 376;
    // 100 of 8 to 1,024: 163, 144)
    const size_t np = (size_t)(n_polys > 0 ? n_polys : 1);
    size_t bytes = 0;
    auto place = [&](size_t size) {
        const size_t at = bytes;
        bytes += (size + 255) & ~(size_t)255;
        return at;
    };
    const size_t at_xy = place(sizeof(int2) * (size_t)(n_vertices > 0 ? n_vertices : 1));
    const size_t at_off = place(sizeof(int64_t) * (size_t)(n_polys + 1)), at_bbox = place(sizeof(int4) * np);
    const size_t at_area = place(sizeof(int64_t) * np), at_feat = place(sizeof(float2) * np);
    const size_t at_info = place(sizeof(SlabInfo) * np), at_slabs = place(sizeof(SlabPtrs));
    const size_t at_order = place(sizeof(int32_t) * np);
    if (cudaMalloc(&P->arrays, bytes) != cudaSuccess) {
        cudaGetLastError();
        P->arrays = nullptr;
        pmh_polys_destroy(P);
        return pmh_set_error(PMH_ERR_NOMEM, "polygon allocation failed (%lld vertices)",
                             (long long)n_vertices);
    }
    char* base = static_cast<char*>(P->arrays);
    P->xy = reinterpret_cast<int2*>(base + at_xy);
    P->offsets = reinterpret_cast<int64_t*>(base + at_off);
    P->bbox = reinterpret_cast<int4*>(base + at_bbox);
    P->area2 = reinterpret_cast<int64_t*>(base + at_area);
    P->feat = reinterpret_cast<float2*>(base + at_feat);
    P->slab_info = reinterpret_cast<SlabInfo*>(base + at_info);
    P->d_slabs = reinterpret_cast<SlabPtrs*>(base + at_slabs);
    P->order_buf = reinterpret_cast<int32_t*>(base + at_order);
    const int rc = upload_fill(P, xy, offsets, host, (cudaStream_t)stream);
    if (rc != PMH_OK) {
        pmh_polys_destroy(P);
        return rc;
    }
    *out = P;
    return PMH_OK;
}

// release the per-polygon products that are built later than the upload (a reload drops them),
// and with `all` those of the upload itself
static void free_derived(pmh_polys p, bool all)
{
    void* late[] = {p->order, p->mask};
    for (void* b : late)
        if (b) cudaFree(b);
    p->order = nullptr;
    p->mask = nullptr;
    p->n_indexed = p->n_whole_cost = 0;
    p->order_cls = nullptr;
    if (!all) return;
    if (p->slab_ptr) cudaFree(p->slab_ptr);
    p->slab_ptr = p->slab_edges = nullptr;
    p->cap_slab_ptr = p->cap_slab_edges = 0;
}

extern "C" int pmh_poly_reload(pmh_polys polys, const int32_t* xy, const int64_t* offsets,
                               int64_t n_polys, int64_t n_vertices, int host_memory, void* stream)
{
    if (!polys) return pmh_set_error(PMH_ERR_ARG, "null polygons");
    PMH_TRY(pmh_check_device(polys->ctx));
    if (n_polys != polys->n || n_vertices != polys->nv || (!xy && n_vertices > 0) || !offsets)
        return pmh_set_error(PMH_ERR_ARG, "reload needs the set's own sizes (%lld polygons, %lld "
                             "vertices; got %lld, %lld)", (long long)polys->n, (long long)polys->nv,
                             (long long)n_polys, (long long)n_vertices);
    cudaStream_t s = (cudaStream_t)stream;
    // no kernel of any stream may still read the old data.  The slab lists and the class order
    // keep their buffers while the new lists fit (releasing and taking half a gigabyte was a
    // third of a reload of 400,000 polygons)
    PMH_CUDA_TRY(cudaDeviceSynchronize());
    PMH_CUDA_TRY(cudaMemsetAsync(polys->d_slabs, 0, sizeof(SlabPtrs), s));
    free_derived(polys, false);
    const int rc = upload_fill(polys, xy, offsets, host_memory != 0, s);
    if (rc != PMH_OK) {  // a reload that fails leaves no slab index behind
        cudaMemsetAsync(polys->d_slabs, 0, sizeof(SlabPtrs), s);
        cudaMemsetAsync(polys->slab_info, 0, sizeof(SlabInfo) * polys->n, s);
        cudaDeviceSynchronize();
        free_derived(polys, true);
        polys->max_n = INT32_MAX;  // (unknown)
    }
    return rc;
}

extern "C" int pmh_poly_upload(pmh_ctx ctx, const int32_t* d_xy, const int64_t* d_offsets,
                               int64_t n_polys, int64_t n_vertices, pmh_polys* out, void* stream)
{
    return upload_common(ctx, d_xy, d_offsets, n_polys, n_vertices, false, out, stream);
}

extern "C" int pmh_poly_upload_host(pmh_ctx ctx, const int32_t* h_xy, const int64_t* h_offsets,
                                    int64_t n_polys, int64_t n_vertices, pmh_polys* out,
                                    void* stream)
{
    return upload_common(ctx, h_xy, h_offsets, n_polys, n_vertices, true, out, stream);
}

extern "C" int pmh_polys_info(pmh_polys p, int64_t* n_polys, int64_t* n_vertices)
{
    if (!p) return pmh_set_error(PMH_ERR_ARG, "null polygons");
    if (n_polys) *n_polys = p->n;
    if (n_vertices) *n_vertices = p->nv;
    return PMH_OK;
}

extern "C" int pmh_polys_prep(pmh_polys p, int32_t* d_bbox, int64_t* d_area2, void* stream)
{
    if (!p) return pmh_set_error(PMH_ERR_ARG, "null polygons");
    PMH_TRY(pmh_check_device(p->ctx));
    cudaStream_t s = (cudaStream_t)stream;
    if (d_bbox && p->n)
        PMH_CUDA_TRY(cudaMemcpyAsync(d_bbox, p->bbox, sizeof(int4) * p->n, cudaMemcpyDeviceToDevice, s));
    if (d_area2 && p->n)
        PMH_CUDA_TRY(cudaMemcpyAsync(d_area2, p->area2, sizeof(int64_t) * p->n,
                                     cudaMemcpyDeviceToDevice, s));
    return PMH_OK;
}

extern "C" int pmh_polys_destroy(pmh_polys p)
{
    if (!p) return PMH_OK;
    cudaSetDevice(p->device);
    if (p->arrays) cudaDeviceSynchronize();
    void* bufs[] = {p->arrays, p->slab_ptr, p->order, p->mask};
    for (void* b : bufs)
        if (b) cudaFree(b);
    delete p;
    return PMH_OK;
}
