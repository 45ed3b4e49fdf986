// stream_index.cu -- the first M points of every hash's stream, bucketed by
// lattice cell (used by the indexed signing path of A1).
//
// Every polygon draws from the same K point streams (Sec. 3.2: fixed seeds per
// hash function), so the points themselves can be indexed once: for each hash
// k the points i < M are sorted (stably) by their cell in a G x G grid over the
// domain.  In a cell that lies inside a polygon only the cell's first point can
// be the hash, and in a cell that the boundary crosses only its points below the
// smallest one known to be inside; the smallest index found that way is h_k
// exactly if it is below M, because every point of the stream with index < M is
// in one of the cells.  If there is none, the ordinary walk continues from M.
//
// Layout: rows of P = K rounded up to four per cell; first[c * P + k] = 2 * smallest
// index of the list of (k, c), + 1 if the list goes on (all ones if it is empty): a warp
// reads one cell's words for 128 consecutive hashes as 512 bytes.  The entries are
// sorted by (hash k, cell c, stream index); entry e = (stream index, x | y << 16), one
// 8-byte load.  The list of (k, c) is [beg[c*P + k], beg[(c+1)*P + k]).
#include <algorithm>

#include "pmh_internal.cuh"

namespace {

__global__ void stream_points_kernel(uint64_t seed, int K, int M, int shift, int gbits,
                                     uint32_t* __restrict__ keys, int32_t* __restrict__ vals)
{
    const int64_t total = (int64_t)K * M;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int k = (int)(t / M);
        const int i = (int)(t - (int64_t)k * M);
        const uint64_t sk = pmh_mix64(seed + (uint64_t)(k + 1) * PMH_GAMMA);
        const uint32_t r = pmh_mix64_lo(sk + (uint64_t)(i + 1) * PMH_GAMMA);
        const uint32_t x = r & 0xFFFFu, y = r >> 16;
        const uint32_t cell = ((y >> shift) << gbits) | (x >> shift);
        keys[t] = ((uint32_t)k << (2 * gbits)) | cell;
        vals[t] = i;
    }
}

__global__ void cell_count_kernel(const uint32_t* __restrict__ keys, int64_t n,
                                  int64_t* __restrict__ counts)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(reinterpret_cast<unsigned long long*>(&counts[keys[e]]), 1ull);
}

__global__ void finish_index_kernel(const uint32_t* __restrict__ keys, const int32_t* __restrict__ vals,
                                    int64_t n, uint64_t seed, int gbits, uint2* __restrict__ ent)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int k = (int)(keys[e] >> (2 * gbits));
        const int i = vals[e];
        const uint64_t sk = pmh_mix64(seed + (uint64_t)(k + 1) * PMH_GAMMA);
        ent[e] = make_uint2((uint32_t)i, pmh_mix64_lo(sk + (uint64_t)(i + 1) * PMH_GAMMA));
    }
}

// list starts and first indexes (cell-major) from the k-major list starts; row G*G of beg
// holds each hash's end
__global__ void cell_record_kernel(const int64_t* __restrict__ starts, int K, int gbits,
                                   const uint2* __restrict__ ent, uint32_t* __restrict__ beg,
                                   uint32_t* __restrict__ first)
{
    const int64_t GG = (int64_t)1 << (2 * gbits);
    const int P = index_pitch(K);
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < GG * P;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t cl = t / P, k = t - cl * P;
        uint32_t b = 0, e = 0, f = 0xFFFFFFFFu;
        if (k < K) {  // (the row's padding holds empty lists)
            const int64_t c = (k << (2 * gbits)) + cl;
            b = (uint32_t)starts[c];
            e = (uint32_t)starts[c + 1];
            if (b < e) f = 2u * ent[b].x + (e - b > 1u);
        }
        beg[t] = b;
        first[t] = f;
        if (cl == GG - 1) beg[GG * P + k] = e;
    }
}

}  // namespace

// what the building of a level works on, sized for the largest: the levels share it, and the build
// synchronises once at its end
struct LevelScratch {
    uint32_t* keys = nullptr;
    int32_t* vals = nullptr;
    int64_t* counts = nullptr;
    int alloc(int64_t points, int64_t cells)
    {
        if (cudaMalloc(&keys, sizeof(uint32_t) * points) == cudaSuccess &&
            cudaMalloc(&vals, sizeof(int32_t) * points) == cudaSuccess &&
            cudaMalloc(&counts, sizeof(int64_t) * (cells + 1)) == cudaSuccess)
            return PMH_OK;
        cudaGetLastError();
        return pmh_set_error(PMH_ERR_NOMEM, "stream index scratch allocation failed");
    }
    void release()
    {
        cudaFree(keys);
        cudaFree(vals);
        cudaFree(counts);
    }
};

// One level: the first M points of every hash's stream on a 2^gbits-square grid.
// Allocates the level's tables (which the caller frees, also after a failure).
static int build_level(pmh_ctx ctx, const pmh_params* P, cudaStream_t s, int M, int gbits,
                       const LevelScratch& w, uint32_t** first, uint32_t** beg, uint2** ent)
{
    const int shift = 16 - gbits;
    const int64_t n = (int64_t)P->K * M;
    const int64_t n_cells = (int64_t)P->K << (2 * gbits);
    const int64_t rows = 1ll << (2 * gbits), pitch = index_pitch((int)P->K);
    if (cudaMalloc(first, sizeof(uint32_t) * rows * pitch) != cudaSuccess ||
        cudaMalloc(beg, sizeof(uint32_t) * (rows + 1) * pitch) != cudaSuccess ||
        cudaMalloc(ent, sizeof(uint2) * n) != cudaSuccess) {
        cudaGetLastError();
        return pmh_set_error(PMH_ERR_NOMEM, "stream index allocation failed");
    }
    const int blocks = ctx->sm_count * 16;
    stream_points_kernel<<<blocks, 256, 0, s>>>(P->seed, (int)P->K, M, shift, gbits, w.keys, w.vals);
    PMH_LAUNCHED("stream_points_kernel");
    int key_bits = 2 * gbits;
    while ((1ll << key_bits) < n_cells) ++key_bits;
    PMH_TRY(pmh_radix_sort_u32(ctx, w.keys, w.vals, n, key_bits, s));
    PMH_CUDA_TRY(cudaMemsetAsync(w.counts, 0, sizeof(int64_t) * (n_cells + 1), s));
    cell_count_kernel<<<blocks, 256, 0, s>>>(w.keys, n, w.counts);
    PMH_LAUNCHED("cell_count_kernel");
    PMH_TRY(pmh_exclusive_scan_i64(ctx, w.counts, w.counts, n_cells, s));
    finish_index_kernel<<<blocks, 256, 0, s>>>(w.keys, w.vals, n, P->seed, gbits, *ent);
    PMH_LAUNCHED("finish_index_kernel");
    cell_record_kernel<<<blocks, 256, 0, s>>>(w.counts, (int)P->K, gbits, *ent, *beg, *first);
    PMH_LAUNCHED("cell_record_kernel");
    return PMH_OK;
}

static StreamIndexView view_of(const StreamIndex& si)
{
    StreamIndexView v{};
    for (int l = 0; l < kIndexLevels; ++l)
        v.lv[l] = IndexLevelView{si.first[l], si.beg[l], si.ent[l], index_level_points(l), index_level_gbits(l),
                                 16 - index_level_gbits(l)};
    v.K = si.K;
    v.pitch = index_pitch(si.K);
    return v;
}

static void free_index(StreamIndex& si)
{
    for (int l = 0; l < kIndexLevels; ++l) {
        cudaFree(si.first[l]);
        cudaFree(si.beg[l]);
        cudaFree(si.ent[l]);
    }
    si = StreamIndex();
}

int pmh_stream_index_get(pmh_ctx ctx, const pmh_params* P, cudaStream_t s, StreamIndexView* out)
{
    StreamIndex& si = ctx->sindex;
    if (si.first[0] && si.seed == P->seed && si.K == (int)P->K) {
        *out = view_of(si);
        return PMH_OK;
    }
    if (si.first[0]) {
        cudaDeviceSynchronize();
        free_index(si);
    }
    StreamIndex fresh;
    LevelScratch scratch;
    const int K = (int)P->K;
    int64_t points = 0, cells = 0;  // (the finest level that fits; all but the finest always do: K <= 4096)
    for (int l = 0; l < kIndexLevels; ++l)
        if (index_level_fits(l, K)) {
            points = std::max(points, (int64_t)K * index_level_points(l));
            cells = std::max(cells, (int64_t)K << (2 * index_level_gbits(l)));
        }
    int rc = scratch.alloc(points, cells);
    for (int l = 0; l < kIndexLevels && rc == PMH_OK; ++l)
        if (index_level_fits(l, K))
            rc = build_level(ctx, P, s, index_level_points(l), index_level_gbits(l), scratch, &fresh.first[l],
                             &fresh.beg[l], &fresh.ent[l]);
    const cudaError_t e = cudaStreamSynchronize(s);
    if (rc == PMH_OK && e != cudaSuccess)
        rc = pmh_set_error(PMH_ERR_CUDA, "stream index build: %s", cudaGetErrorString(e));
    scratch.release();
    if (rc != PMH_OK) {
        free_index(fresh);
        return rc;
    }
    fresh.seed = P->seed;
    fresh.K = (int)P->K;
    fresh.build = ++ctx->sindex_builds;
    si = fresh;
    *out = view_of(si);
    return PMH_OK;
}

extern "C" int pmh_stream_index_build(pmh_ctx ctx, const pmh_params* params, void* stream)
{
    PMH_TRY(pmh_check_device(ctx));
    PMH_TRY(pmh_check_params(params));
    StreamIndexView v;
    return pmh_stream_index_get(ctx, params, (cudaStream_t)stream, &v);
}
