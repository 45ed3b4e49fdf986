// sign_unified.cu -- step A1 (Definition 2, Algorithm 1): persistent signing launches for
// polygons of every size, through the stream index: one for the rings above the staged size and
// one for the staged ones (a captured batch: one for both), one before them for few hashes of
// polygons of large area, and one behind them for the walks past the index.
//
// h_k(P) = min{ i : point i of stream k lies in P } is found, per polygon, in
// the indexed form or in the walk form:
//   * indexed form: the cells of one grid of the stream index (stream_index.cu)
//     under P's bounding box are classified as inside P, outside, or crossed by its
//     boundary.  Of an inside cell only the first point of the stream in it can be
//     the hash, and the index holds that index, so 128 hashes at a time (four a lane)
//     the inside cells cost one 16-byte read and four minima per cell.  Of a
//     boundary cell the first point is a candidate only if it is below the hash's
//     bound so far -- few are, the inside cells having set a bound already.  The
//     candidates of all lanes are queued and looked up 32 at a time (the point is
//     recomputed from its index) in a 32 x 32 coverage mask, which decides most;
//     the others are queued again and tested exactly 32 at a time, so that the long
//     part runs with every lane.  An inside point lowers its hash's bound, an outside
//     one is replaced by the next point of its cell below the bound.  A hash without
//     a point below the level's limit is queued, and a last launch walks on from there;
//   * walk form (no index, a very large polygon whose expected walk is short, or, in a launch of its
//     own, a few hashes of a polygon of large area):
//     Algorithm 1 in warp rounds of 32 * U consecutive stream points; box
//     candidates in index order (ballot + ffs), each decided by the mask or by the
//     warp-cooperative exact test.
// Edge sources: a polygon of at most 256 vertices is staged in the warp's
// shared-memory slice with its edges binned into 32 y-slabs; a larger one is
// read from global memory through the y-slab edge lists built at upload
// (slabs.cu), or through all its edges where it has none.  Either way an
// exact test reads only the edges of one slab.
//
// Work items come from one atomic ticket over a list of polygon slots: the
// first n_chunked slots are split into (polygon, 32-hash chunk) items -- the
// very large polygons (above 4,096 vertices), whose walks and tests cost the
// most, first and by decreasing cost -- and the remaining slots are whole
// polygons (all K hashes, so that the staging and the mask are paid once per
// polygon).  A
// staged polygon met in a chunked slot is signed whole by its chunk 0 (its
// other chunks return at once) unless the batch leaves warps idle, so the captured query
// pipeline can hand in every polygon as a chunked slot.  Every step is exact, so the result equals
// the definition bit for bit.
#include <algorithm>
#include <type_traits>

#include "sign_common.cuh"

namespace {

constexpr int kUniWarps = 4;       // warps per block
constexpr int kUniMinBlocks = 8;   // resident blocks per SM the registers are sized for
constexpr int kMaskN = 32;         // coverage mask cells per side
constexpr int kGroup = 128;        // hashes signed together, four a lane
constexpr int kQueue = 192;        // candidates: at most 31, + 128 of a cell, + 32 that follow exact tests
constexpr uint32_t kNoPoint = 0xFFFFFFFFu;
// A few hashes of a polygon of large area are walked in a launch of their own (sign_brief_kernel):
// K walks of 2^32 / area points cost less than the mask and the cells under the box.  100,000 stars
// of 16 to 256 vertices and 1e-4 to 1e-2 of the domain: K = 3 946 us through the index, 754; 8 994,
// 970; 10 1,024, 1,050; 5,000 fractal rings of 300 to 4,000 vertices: K = 3 168, 139; 8 176, 170;
// 16 180, 218.  Points per polygon from 1,500 to 4,500 measure within 5% of each other
constexpr int kBriefMaxK = 8;
constexpr float kBriefWalk = 3000.0f;
constexpr int kIdxU = 4;           // points per lane per round of a leftover walk
constexpr int kMaskMaxEdges = 4096;  // larger polygons skip the mask (every cell is a boundary cell)

// a warp's shared slice, and a staged ring's part of it
struct __align__(16) UniSlice {
    uint32_t best[kGroup];   // per hash of the group: 2 * smallest inside index found (+ 1); 16-byte accesses
    uint32_t bnd[kMaskN];    // bit i of row j: an edge touches cell (i, j)
    uint32_t inb[kMaskN];    // bit i of row j: untouched cell (i, j) lies inside
    uint32_t cell[kPlanCells];  // table rows of the inside cells (from the front) and of the boundary cells (from the back)
    uint2 queue[kQueue];     // (depth in the cell's list << 16 | boundary cell << 7 | hash, 2 * stream index + more)
    uint2 exact[64];         // the same, of candidates to test exactly
    uint32_t exact_xy[64];   // x | y << 16
};
struct UniWarp : UniSlice {
    int2 v[kSmemVerts + 1];  // staged vertices, v[n] = v[0]
    uint8_t ids[kSlabCap];   // staged edges by slab
    uint16_t beg[kSlabs + 1];
    int cnt[kSlabs];
};
// which polygons a build of the kernel takes: staged ones of the indexed form, larger ones, or all.
// The class order puts them apart; a captured batch is mixed.
enum class UniForm { kStaged, kLarge, kMixed };

// ---------------------------------------------------------------------------
// Edge sources.  vert(e) for e in [0, n] (vert(n) = vert(0)); row(py) gives the
// list positions [lo, hi) of the edges that can straddle the line y = py, and
// edge(t) the edge at list position t.
// ---------------------------------------------------------------------------
struct StagedSrc {
    const int2* v;
    const uint8_t* ids;
    const uint16_t* beg;
    int y0, sh;
    __device__ __forceinline__ int2 vert(int e) const { return v[e]; }
    __device__ __forceinline__ void row(int py, int& lo, int& hi) const
    {
        const int s = (py - y0) >> sh;
        lo = beg[s];
        hi = beg[s + 1];
    }
    __device__ __forceinline__ int edge(int t) const { return ids[t]; }
};

struct GlobalSrc {
    const int2* v;       // the polygon's first vertex
    int n;
    const int32_t* sp;   // slab table (nullptr: one list of every edge)
    const int32_t* se;   // edge lists
    int ymin;
    uint64_t magic;      // of the slab height
    __device__ __forceinline__ int2 vert(int e) const { return v[e == n ? 0 : e]; }
    __device__ __forceinline__ void row(int py, int& lo, int& hi) const
    {
        if (sp) {
            const int s = slab_div(py - ymin, magic);
            lo = sp[s];
            hi = sp[s + 1];
        } else {
            lo = 0;
            hi = n;
        }
    }
    __device__ __forceinline__ int edge(int t) const { return sp ? se[t] : t; }
};

// exact half-open membership, one point per lane
template <class Src, class W>
__device__ __forceinline__ bool lane_inside(const Src& s, int px, int py, W& w)
{
    int lo, hi;
    s.row(py, lo, hi);
    w.lane_edges += hi - lo;
    unsigned par = 0;
    for (int t = lo; t < hi; ++t) {
        const int e = s.edge(t);
        par ^= edge_parity(s.vert(e), s.vert(e + 1), px, py);
    }
    return par;
}

// exact half-open membership, warp-cooperative (lanes split the row's edges)
template <class Src, class W>
__device__ __forceinline__ bool warp_inside_src(const Src& s, int px, int py, int lane, W& w)
{
    int lo, hi;
    s.row(py, lo, hi);
    w.edges += hi - lo;
    unsigned par = 0;
    for (int t = lo + lane; t < hi; t += 32) {
        const int e = s.edge(t);
        par ^= edge_parity(s.vert(e), s.vert(e + 1), px, py);
    }
    return __popc(__ballot_sync(0xffffffffu, par)) & 1;
}

// stream points examined per hash, on average
__device__ __forceinline__ float expected_walk(long long area2)
{
    return 4294967296.0f / fmaxf(0.5f * (float)(area2 < 0 ? -area2 : area2), 1.0f);
}
// walks shorter than this are signed briefly
static float brief_limit(int K) { return K <= kBriefMaxK ? kBriefWalk / (float)K : 0.0f; }

// coverage mask frame of a clipped box: cells of 2^cwl x 2^chl lattice units aligned to
// the lattice (so that the cells of any grid of the stream index with at most 32 cells a
// side under the box are unions of mask cells), cell (0, 0) holding the box's corner
struct MaskFrame {
    int x0, y0, cwl, chl;
};
__device__ __forceinline__ MaskFrame mask_frame(int4 bb)
{
    MaskFrame f{0, 0, 0, 0};
    while (((bb.z - 1) >> f.cwl) - (bb.x >> f.cwl) >= kMaskN) ++f.cwl;
    while (((bb.w - 1) >> f.chl) - (bb.y >> f.chl) >= kMaskN) ++f.chl;
    f.x0 = (bb.x >> f.cwl) << f.cwl;
    f.y0 = (bb.y >> f.chl) << f.chl;
    return f;
}

// one slab holding every staged edge: the exact test then reads all n edges
__device__ __forceinline__ int single_slab(UniWarp& m, int n, int lane)
{
    for (int e = lane; e < n; e += 32) m.ids[e] = (uint8_t)e;
    if (lane == 0) m.beg[0] = 0;
    if (lane < kSlabs) m.beg[lane + 1] = (uint16_t)n;
    __syncwarp();
    return 16;
}

// 32 x 32 coverage mask of frame f over the clipped box bb (cell (i, j): lattice points
// f.x0 + [i*cw, (i+1)*cw) by f.y0 + [j*ch, (j+1)*ch)).  bnd marks every cell
// whose closed rectangle, grown by one unit on its low sides, meets an edge
// (and possibly a few neighbours: the marking is conservative).  Every lattice
// point of an unmarked cell (under the half-open reading, the point shifted up
// and right by an infinitesimal) then shares the membership of the whole
// rectangle.  Row j's unmarked cells are classified together from the edges
// crossing the line y = f.y0 + j*ch: a cell is inside iff an odd number of
// crossings lies left of it (none does on a line below the box, which no edge
// crosses).  A crossing lies in a marked cell of the row, at
// least one unit left of or strictly right of every unmarked cell, so its
// cell index -- computed in single precision, off by less than one unit --
// never moves it across an unmarked cell, and the classification is exact.
// Without a mask (use_mask false) every cell is a boundary cell.
template <class M, class Src, class W>
__device__ __forceinline__ void build_mask(M& m /* its bnd and inb */, const Src& src, int n, int4 bb, const MaskFrame& f,
                                           bool use_mask, int lane, W& work)
{
    const int cwl = f.cwl, chl = f.chl;
    if (!use_mask) {
        m.bnd[lane] = 0xFFFFFFFFu;
        m.inb[lane] = 0u;
        __syncwarp();
        return;
    }
    m.bnd[lane] = 0;
    __syncwarp();
    const float inv_cw = 1.0f / (float)(1 << cwl);
    const int ch = 1 << chl;
    for (int e = lane; e < n; e += 32) {
        const int2 a = src.vert(e), c = src.vert(e + 1);
        // rows whose grown band [j*ch - 1, (j+1)*ch] (relative) meets the edge's y-range
        const int ylo = min(a.y, c.y) - f.y0, yhi = max(a.y, c.y) - f.y0;
        const int j0 = max(0, ((ylo + ch - 1) >> chl) - 1);
        const int j1 = min(kMaskN - 1, (yhi + 1) >> chl);
        const float ax = (float)(a.x - f.x0), ay = (float)(a.y - f.y0);
        const float dx = (float)(c.x - a.x);
        const float inv_dy = c.y != a.y ? 1.0f / (float)(c.y - a.y) : 0.0f;
        for (int j = j0; j <= j1; ++j) {
            // the edge's x-range over the band (single precision, error < 1 unit)
            float t0 = 0.0f, t1 = 1.0f;
            if (c.y != a.y) {
                t0 = fminf(fmaxf(((float)((j << chl) - 1) - ay) * inv_dy, 0.0f), 1.0f);
                t1 = fminf(fmaxf(((float)((j + 1) << chl) - ay) * inv_dy, 0.0f), 1.0f);
            }
            const float xa = ax + dx * t0, xb = ax + dx * t1;
            // cells whose grown x-range [i*cw - 1, (i+1)*cw] meets it, one unit of margin
            const int i0 = max(0, (int)ceilf((fminf(xa, xb) - 1.0f) * inv_cw) - 1);
            const int i1 = min(kMaskN - 1, (int)floorf((fmaxf(xa, xb) + 2.0f) * inv_cw));
            if (i0 <= i1) {
                const uint32_t hi_bits = i1 == 31 ? 0xFFFFFFFFu : ((2u << i1) - 1u);
                atomicOr(&m.bnd[j], hi_bits & ~((1u << i0) - 1u));
            }
        }
    }
    __syncwarp();
    // lane j: parity of the crossings of the line y = f.y0 + j*ch left of each cell
    // (lines inside the box only: the slab lists cover [bb.y, bb.w))
    uint32_t word = 0;
    const int py = f.y0 + (lane << chl);
    if (py >= bb.y && py < bb.w) {
        int lo, hi;
        src.row(py, lo, hi);
        uint32_t par = 0;
        for (int t = lo; t < hi; ++t) {
            const int e = src.edge(t);
            const int2 a = src.vert(e), b = src.vert(e + 1);
            if ((a.y > py) != (b.y > py)) {
                const float x = (float)(a.x - f.x0) +
                                (float)(b.x - a.x) * ((float)(py - a.y) / (float)(b.y - a.y));
                const int ci = (int)floorf(x * inv_cw);
                par ^= ci < 0 ? 0xFFFFFFFFu : (ci >= kMaskN - 1 ? 0u : (0xFFFFFFFFu << (ci + 1)));
            }
        }
        work.lane_edges += hi - lo;
        word = par & ~m.bnd[lane];
    }
    m.inb[lane] = word;
    __syncwarp();
}

// Membership through the mask (warp-cooperative, for the walk form):
// untouched cells by their code, boundary cells by the exact test.
template <class Src>
struct MaskedWalker {
    const UniSlice* m;
    Src src;
    int x0, y0, cwl, chl;
    template <class W>
    __device__ __forceinline__ bool operator()(int px, int py, int lane, W& w) const
    {
        const int i = (px - x0) >> cwl, j = (py - y0) >> chl;
        if (!((m->bnd[j] >> i) & 1u)) {
            w.masked += 1;
            return (m->inb[j] >> i) & 1u;
        }
        return warp_inside_src(src, px, py, lane, w);
    }
};

// per-lane counts of the gather (widened at the end), and the same compiled away
struct GatherCounts {
    unsigned cells = 0, read = 0, cand = 0, masked = 0;
};
struct NoGather {
    Sink cells, read, cand, masked;
};

// The cells of level L under the box: inside cells to the front of m.cell, boundary
// cells to its back (as cell * pitch).  A grid cell is a block of mask cells; it is inside
// iff all of them are (a part outside the mask's frame is outside the box).
__device__ __forceinline__ void classify_cells(UniSlice& m, const IndexLevelView& L, int pitch, int4 bb,
                                               const MaskFrame& f, int& n_in, int& n_bnd, int lane)
{
    const unsigned full = 0xffffffffu;
    const int cx0 = bb.x >> L.shift, cy0 = bb.y >> L.shift;
    const int ncx = ((bb.z - 1) >> L.shift) - cx0 + 1, C = ncx * (((bb.w - 1) >> L.shift) - cy0 + 1);
    const int cw = 1 << (L.shift - f.cwl), ch = 1 << (L.shift - f.chl);  // mask cells a side
    n_in = n_bnd = 0;
    for (int c0 = 0; c0 < C; c0 += 32) {
        const int c = c0 + lane;
        bool in = false, bnd = false;
        uint32_t off = 0;
        if (c < C) {
            const int gy = c / ncx, gx = c - gy * ncx;
            off = (uint32_t)(((cy0 + gy) << L.gbits) | (cx0 + gx)) * (uint32_t)pitch;
            const int i0 = (((cx0 + gx) << L.shift) - f.x0) >> f.cwl, j0 = (((cy0 + gy) << L.shift) - f.y0) >> f.chl;
            const int ia = max(i0, 0), ib = min(i0 + cw, kMaskN);
            const uint32_t cols = (ib == 32 ? 0xFFFFFFFFu : (1u << ib) - 1u) & ~((1u << ia) - 1u);
            uint32_t any = 0, all = cols;
            for (int j = max(j0, 0); j < min(j0 + ch, kMaskN); ++j) {
                const uint32_t w = m.inb[j];
                any |= m.bnd[j] | w;
                all &= w;
            }
            in = all == cols && i0 >= 0 && i0 + cw <= kMaskN && j0 >= 0 && j0 + ch <= kMaskN;
            bnd = !in && (any & cols) != 0;
        }
        const unsigned bi = __ballot_sync(full, in), bb_ = __ballot_sync(full, bnd);
        if (in) m.cell[n_in + __popc(bi & pmh_lanemask_lt())] = off;
        if (bnd) m.cell[kPlanCells - 1 - (n_bnd + __popc(bb_ & pmh_lanemask_lt()))] = off;
        n_in += __popc(bi);
        n_bnd += __popc(bb_);
    }
    __syncwarp();
}

// Indexed form of hashes [k_begin, k_end) of polygon p (row `out` of the output).  Bound
// by issue (the exact tests of spiky rings, the mask of every polygon) and by the latency
// of the table reads, which stay in L2.  Against reading every point below a few expected
// first hits from the cells under the box: 300,000 star polygons, K = 128, 5.3 ms (9.1);
// 400,000 of the combined workload 6.4 ms (10.6).
// A __syncwarp stands between every read of a queue and the next write to it: a vote
// orders nothing in memory.
template <class Src, class W, class G>
__device__ __forceinline__ void indexed_range(UniSlice& m, const Src& src, const StreamIndexView& S, int level,
                                              int4 bb, const MaskFrame& f, float walk, uint64_t seed, uint32_t T,
                                              int64_t p, int k_begin, int k_end, const WalkQueue& wq,
                                              uint32_t* __restrict__ out, int lane, W& work, G& gc)
{
    const unsigned full = 0xffffffffu, lt = pmh_lanemask_lt();
    const uint32_t w = (uint32_t)(bb.z - bb.x), h = (uint32_t)(bb.w - bb.y);
    const IndexLevelView& L = S.lv[level];
    const int pitch = S.pitch;
    int n_in, n_bnd;
    classify_cells(m, L, pitch, bb, f, n_in, n_bnd, lane);
    // with few inside cells to bound the hashes, a first pass over the boundary cells keeps to
    // the points below ~2 expected first hits: else every cell's first point would be tried
    const uint32_t lim1 = 8 * n_in >= n_bnd ? kNoPoint : 2u * (uint32_t)fminf(2.0f * walk + 64.0f, 1.0e9f);

    for (int kc = k_begin; kc < k_end; kc += kGroup) {
        const int kn = min(kGroup, k_end - kc);
        // lane: hashes 4 * vl .. 4 * vl + 3 of the group, cells sub, sub + nsub, .. (several
        // cells at a time for few hashes)
        const int nv = (kn + 3) >> 2, lgv = 32 - __clz(nv - 1);
        const int nsub = 32 >> lgv, vl = lane & ((1 << lgv) - 1), sub = lane >> lgv;
        const bool active = vl < nv;
        const uint32_t* first = L.first + kc + 4 * (active ? vl : 0);
        if (lane == 0) gc.cells += (unsigned)((n_in + n_bnd) * kn);
        uint4 best = make_uint4(kNoPoint, kNoPoint, kNoPoint, kNoPoint);
#pragma unroll 4
        for (int i = sub; i < n_in; i += nsub) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(first + m.cell[i]));
            best.x = min(best.x, v.x);
            best.y = min(best.y, v.y);
            best.z = min(best.z, v.z);
            best.w = min(best.w, v.w);
        }
        for (int o = 1 << lgv; o < 32; o <<= 1) {
            best.x = min(best.x, __shfl_xor_sync(full, best.x, o));
            best.y = min(best.y, __shfl_xor_sync(full, best.y, o));
            best.z = min(best.z, __shfl_xor_sync(full, best.z, o));
            best.w = min(best.w, __shfl_xor_sync(full, best.w, o));
        }
        if (sub == 0) {
            m.best[4 * vl] = best.x;
            m.best[4 * vl + 1] = best.y;
            m.best[4 * vl + 2] = best.z;
            m.best[4 * vl + 3] = best.w;
        }
        __syncwarp();
        uint32_t bound = lim1;
        bool open = active;
        int nq = 0, nx = 0;  // queued candidates, queued exact tests
        const uint4 none = make_uint4(kNoPoint, kNoPoint, kNoPoint, kNoPoint);
        // an inside point bounds its hash; an outside one is followed by the next of its cell, if
        // that is still below the hash's bound
        auto settle = [&](uint2 c, bool inside, bool fail) {
            if (inside) atomicMin(&m.best[c.x & 127u], c.y);
            bool again = false;
            if (fail && (c.y & 1u)) {
                const uint32_t row = m.cell[kPlanCells - 1 - (int)((c.x >> 7) & 127u)] + (uint32_t)kc + (c.x & 127u);
                const uint32_t e = L.beg[row] + (c.x >> 16) + 1u, end = L.beg[row + (uint32_t)pitch];
                c = make_uint2(c.x + 0x10000u, 2u * L.ent[e].x + (e + 1u < end));
                again = c.y < min(m.best[c.x & 127u], bound);
                ++gc.read;
            }
            const unsigned bal = __ballot_sync(full, again);
            if (again) m.queue[nq + __popc(bal & lt)] = c;
            nq += __popc(bal);
            __syncwarp();
        };
        for (int i0 = 0;;) {
            if (i0 < n_bnd) {
                const int i = i0 + sub;
                const uint4 v = open && i < n_bnd
                                    ? __ldg(reinterpret_cast<const uint4*>(first + m.cell[kPlanCells - 1 - i]))
                                    : none;
                const uint32_t tag = (uint32_t)(i << 7 | 4 * vl);
                const uint32_t vv[4] = {v.x, v.y, v.z, v.w};
                const uint32_t bb4[4] = {best.x, best.y, best.z, best.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool cand = vv[u] < min(bb4[u], bound);
                    const unsigned bal = __ballot_sync(full, cand);
                    if (cand) m.queue[nq + __popc(bal & lt)] = make_uint2(tag + u, vv[u]);
                    nq += __popc(bal);
                }
                i0 += nsub;
                __syncwarp();
            }
            const bool scanned = i0 >= n_bnd;
            for (;;) {
                if (nx < 32 && (nq >= 32 || (scanned && nq > 0))) {
                    // look 32 candidates up
                    const int count = min(nq, 32);
                    nq -= count;
                    uint2 c = make_uint2(0u, kNoPoint);
                    uint32_t r = 0;
                    bool inside = false, fail = false, boundary = false;
                    if (lane < count) c = m.queue[nq + lane];
                    __syncwarp();
                    if (c.y < m.best[c.x & 127u]) {
                        const uint64_t sk = pmh_mix64(seed + (uint64_t)((uint32_t)kc + (c.x & 127u) + 1u) * PMH_GAMMA);
                        r = pmh_mix64_lo(sk + (uint64_t)((c.y >> 1) + 1u) * PMH_GAMMA);
                        const int px = (int)(r & 0xFFFFu), py = (int)(r >> 16);
                        fail = true;
                        if ((uint32_t)(px - bb.x) < w && (uint32_t)(py - bb.y) < h) {
                            ++gc.cand;
                            const int i = (px - f.x0) >> f.cwl, j = (py - f.y0) >> f.chl;
                            boundary = (m.bnd[j] >> i) & 1u;
                            inside = !boundary && ((m.inb[j] >> i) & 1u);
                            fail = !boundary && !inside;
                            gc.masked += boundary ? 0u : 1u;
                        }
                    }
                    const unsigned bal = __ballot_sync(full, boundary);
                    if (boundary) {
                        m.exact[nx + __popc(bal & lt)] = c;
                        m.exact_xy[nx + __popc(bal & lt)] = r;
                    }
                    nx += __popc(bal);
                    settle(c, inside, fail);
                } else if (nx >= 32 || (scanned && nx > 0)) {
                    // test 32 exactly
                    const int count = min(nx, 32);
                    nx -= count;
                    uint2 c = make_uint2(0u, kNoPoint);
                    uint32_t r = 0;
                    bool inside = false, fail = false;
                    if (lane < count) {
                        c = m.exact[nx + lane];
                        r = m.exact_xy[nx + lane];
                    }
                    if (c.y < m.best[c.x & 127u]) {
                        inside = lane_inside(src, (int)(r & 0xFFFFu), (int)(r >> 16), work);
                        fail = !inside;
                    }
                    __syncwarp();
                    settle(c, inside, fail);
                } else {
                    break;
                }
            }
            best = make_uint4(m.best[4 * vl], m.best[4 * vl + 1], m.best[4 * vl + 2], m.best[4 * vl + 3]);
            if (!scanned) continue;
            // a hash with an inside point below the bound is final: every point below it was
            // tried; the others take a second pass without one
            if (bound == kNoPoint) break;
            open = active && max(max(best.x, best.y), max(best.z, best.w)) >= bound;
            if (!__any_sync(full, open)) break;
            bound = kNoPoint;
            i0 = 0;
        }

        // hashes without an inside point below the level's limit are queued for the walks, or,
        // past the queue, marked for them in the output (no hash is above 2^31)
        for (int j0 = 0; j0 < kn; j0 += 32) {
            uint32_t v = j0 + lane < kn ? m.best[j0 + lane] : 0u;
            const unsigned todo = __ballot_sync(full, v == kNoPoint && (uint32_t)L.M < T);
            v = v == kNoPoint ? T : min(v >> 1, T);
            if (todo) {
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(wq.tickets + 1, (unsigned long long)__popc(todo));
                base = __shfl_sync(full, base, 0);
                if ((todo >> lane) & 1u) {
                    const unsigned long long pos = base + __popc(todo & lt);
                    if (pos < kWalkItems) wq.items[pos] = WalkItem{(int32_t)p, kc + j0 + lane, (uint32_t)L.M, 0u};
                    else v = kNoPoint;
                }
            }
            if (j0 + lane < kn) out[kc + j0 + lane] = v;
        }
        __syncwarp();
    }
}

// Walk form of hashes [k_begin, k_end): lane j keeps hash k0 + j of each 32.
template <int U, class Src, class W>
__device__ __forceinline__ void walk_range(const UniSlice& m, const Src& src, int4 bb, const MaskFrame& f, uint64_t seed,
                                           uint32_t T, int k_begin, int k_end,
                                           uint32_t* __restrict__ out, int lane, W& work)
{
    const uint32_t w = (uint32_t)(bb.z - bb.x), h = (uint32_t)(bb.w - bb.y);
    const MaskedWalker<Src> walker{&m, src, f.x0, f.y0, f.cwl, f.chl};
    for (int k0 = k_begin; k0 < k_end; k0 += 32) {
        const int kend = min(k_end, k0 + 32);
        uint32_t mine = T;
        for (int k = k0; k < kend; ++k) {
            const uint64_t sk = pmh_mix64(seed + (uint64_t)(k + 1) * PMH_GAMMA);
            const uint32_t hk = sign_one_t<U>(walker, bb.x, bb.y, w, h, sk, T, lane, work);
            if (lane == k - k0) mine = hk;
        }
        if (k0 + lane < kend) out[k0 + lane] = mine;
    }
}

// Walk form of a staged polygon, kept out of line so that its registers do not
// weigh on the indexed form's gather (Work by pointer: a local copy inside).
template <int U, class W>
__device__ __noinline__ void walk_staged(const UniSlice& m, StagedSrc src, int4 bb, MaskFrame f, uint64_t seed,
                                         uint32_t T, int k_begin, int k_end, uint32_t* out,
                                         int lane, W* work)
{
    W local;
    walk_range<U>(m, src, bb, f, seed, T, k_begin, k_end, out, lane, local);
    work->walk += local.walk;
    work->cand += local.cand;
    work->edges += local.edges;
    work->masked += local.masked;
    work->lane_edges += local.lane_edges;
}

// A polygon above the staged size (read from global memory): the mask, then the planned form.
template <int U, class W, class G>
__device__ __forceinline__ void sign_large(UniSlice& m, const GlobalSrc& src, int n, int4 bb, int level, float walk,
                                           const StreamIndexView& S, uint64_t seed, uint32_t T, int64_t p, int k_begin,
                                           int k_end, const WalkQueue& wq, uint32_t* out, int lane, W& work, G& gc)
{
    const MaskFrame f = mask_frame(bb);
    build_mask(m, src, n, bb, f, n <= kMaskMaxEdges, lane, work);
    // (without a mask every cell is a boundary cell: a walk of few rounds is cheaper)
    if (level >= 0 && (n <= kMaskMaxEdges || walk > 1024.0f))
        indexed_range(m, src, S, level, bb, f, walk, seed, T, p, k_begin, k_end, wq, out, lane, work, gc);
    else
        walk_range<U>(m, src, bb, f, seed, T, k_begin, k_end, out, lane, work);
}

// The same out of line, for the mixed build.
template <int U, class W, class G>
__device__ __noinline__ void sign_global(UniSlice& m, GlobalSrc src, int n, int4 bb, int level, float walk,
                                         const StreamIndexView& S, uint64_t seed, uint32_t T,
                                         int64_t p, int k_begin, int k_end, const WalkQueue& wq,
                                         uint32_t* out, int lane, W* work, G* gc)
{
    W local;
    G g;
    sign_large<U>(m, src, n, bb, level, walk, S, seed, T, p, k_begin, k_end, wq, out, lane, local, g);
    work->walk += local.walk;
    work->cand += local.cand;
    work->edges += local.edges;
    work->masked += local.masked;
    work->lane_edges += local.lane_edges;
    gc->cells += g.cells;
    gc->read += g.read;
    gc->cand += g.cand;
    gc->masked += g.masked;
}

// Builds for the classes of the class order: staged polygons of the indexed form without the
// walk and the large-polygon paths, so that the gather keeps its values in registers (a
// fraction of the mixed build's spills and no call frames); larger ones without the staged ring's
// part of the shared memory (115 of 203 KB an SM), which leaves their vertices, read many times
// from global memory, twice the L1 cache.  20,000 rings of 300 to 1,000 vertices and 2e-5 of the
// domain: K = 32 1,115 us in the mixed build, 828; K = 128 2,447, 1,601
template <int U, bool kCount, UniForm kForm>
__global__ void __launch_bounds__(kUniWarps * 32, kUniMinBlocks)
sign_unified_kernel(const int2* __restrict__ xy, const int64_t* __restrict__ off,
                    const int4* __restrict__ bbox, const int64_t* __restrict__ area2,
                    const SlabInfo* __restrict__ slabs, const int32_t* __restrict__ slab_ptr,
                    const int32_t* __restrict__ slab_edges, const int32_t* __restrict__ list,
                    int64_t n_slots, int64_t n_chunked, const int64_t* __restrict__ d_n,
                    const int* __restrict__ d_flags, uint64_t seed, int K, uint32_t T,
                    StreamIndexView S, WalkQueue wq, float brief_walk, uint32_t* __restrict__ out,
                    unsigned long long* __restrict__ work_out)
{
    using Slice = typename std::conditional<kForm == UniForm::kLarge, UniSlice, UniWarp>::type;
    __shared__ Slice smem[kUniWarps];
    __shared__ unsigned long long wsum[6];
    if (threadIdx.x < 6) wsum[threadIdx.x] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    Slice& m = smem[threadIdx.x >> 5];
    const unsigned full = 0xffffffffu;
    // work counters only in launches that report them
    using W = typename std::conditional<kCount, Work, NoWork>::type;
    using G = typename std::conditional<kCount, GatherCounts, NoGather>::type;
    W work;
    G gc;
    const bool failed = d_flags && *d_flags;  // the batch failed validation
    if (d_n) n_slots = min(n_slots, *d_n);
    n_chunked = min(n_chunked, n_slots);
    const int chunks = (K + 31) / 32;
    const int64_t n_items = failed ? 0 : n_chunked * chunks + (n_slots - n_chunked);
    // staged polygons of a small batch by their chunks too: staging, binning and mask again per
    // chunk, but on warps that had no work.  One query of at most 256 vertices, K = 128:
    // 142 -> 128 us through its graph
    const bool split = n_chunked * chunks <= (int64_t)gridDim.x * kUniWarps;
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(wq.tickets, 1ull);
        item = __shfl_sync(full, item, 0);
        if ((int64_t)item >= n_items) break;
        int64_t slot;
        int chunk = -1;  // -1: the whole polygon
        if ((int64_t)item < n_chunked * chunks) {
            slot = (int64_t)item / chunks;
            chunk = (int)((int64_t)item - slot * chunks);
        } else {
            slot = n_chunked + ((int64_t)item - n_chunked * chunks);
        }
        const int64_t p = list ? (int64_t)list[slot] : slot;
        const int64_t b = off[p];
        const int n = (int)(off[p + 1] - b);
        const bool staged = kForm == UniForm::kMixed ? n <= kSmemVerts : kForm == UniForm::kStaged;
        const bool whole = chunk < 0 || (staged && !split);
        if (whole && chunk > 0) continue;  // signed whole by its chunk 0
        const int k_begin = whole ? 0 : 32 * chunk;
        const int k_end = whole ? K : min(K, 32 * chunk + 32);
        uint32_t* row = out + p * (int64_t)K;
        const int4 bb = bbox[p];
        if (bb.z <= bb.x || bb.w <= bb.y) {  // no lattice point in the box: every hash is T
            for (int k = k_begin + lane; k < k_end; k += 32) row[k] = T;
            continue;
        }
        // the indexed form's grid level (-1: no index) and the expected walk
        const float walk = area2 ? expected_walk(area2[p]) : 0.0f;
        const int level = S.lv[0].first && area2 ? pmh_index_level(bb, K) : -1;
        if (level >= 0 && walk < brief_walk) continue;  // sign_brief_kernel's
        if constexpr (kForm != UniForm::kLarge) {
            if (staged) {
                // stage the polygon (closed: v[n] = v[0]; cp.async 8-byte copies) and bin its edges
                stage_vertices(m.v, xy + b, n, lane);
                int sh = staged_slab_shift(bb.w - bb.y);
                if (!build_staged_slabs(m.v, n, bb.y, sh, m.ids, m.beg, m.cnt, lane)) sh = single_slab(m, n, lane);
                const StagedSrc src{m.v, m.ids, m.beg, bb.y, sh};
                const MaskFrame f = mask_frame(bb);
                build_mask(m, src, n, bb, f, true, lane, work);
                if (kForm == UniForm::kStaged || level >= 0)
                    indexed_range(m, src, S, level, bb, f, walk, seed, T, p, k_begin, k_end, wq, row, lane, work, gc);
                else
                    walk_staged<U, W>(m, src, bb, f, seed, T, k_begin, k_end, row, lane, &work);
                __syncwarp();
            }
        }
        if constexpr (kForm != UniForm::kStaged) {
            if (!staged) {
                const SlabInfo si = slabs ? slabs[p] : SlabInfo{0, 0, 0, 1, 0};
                const GlobalSrc src{xy + b, n, si.S > 0 ? slab_ptr + si.slab_base : nullptr,
                                    si.S > 0 ? slab_edges + si.edge_base : nullptr, si.ymin, slab_div_magic(si.slab_h)};
                if (kForm == UniForm::kLarge)
                    sign_large<U>(m, src, n, bb, level, walk, S, seed, T, p, k_begin, k_end, wq, row, lane, work, gc);
                else
                    sign_global<U, W, G>(m, src, n, bb, level, walk, S, seed, T, p, k_begin, k_end, wq, row, lane, &work,
                                         &gc);
                __syncwarp();
            }
        }
    }
    if (kCount && work_out) {
        unsigned long long le = work.lane_edges, en = gc.read, ca = gc.cand, ma = gc.masked,
                           ce = gc.cells;  // (the gather's 32-bit lane counts, widened)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            le += __shfl_xor_sync(full, le, o);
            en += __shfl_xor_sync(full, en, o);
            ca += __shfl_xor_sync(full, ca, o);
            ma += __shfl_xor_sync(full, ma, o);
            ce += __shfl_xor_sync(full, ce, o);
        }
        if (lane == 0) {
            // Work's walk, candidates, edges and masked counts are warp-uniform; the
            // gather's counts and the lane-local edge tests are per lane
            atomicAdd(&wsum[0], work.walk);
            atomicAdd(&wsum[1], ce);
            atomicAdd(&wsum[2], en);
            atomicAdd(&wsum[3], ca + work.cand);
            atomicAdd(&wsum[4], work.edges + le);
            atomicAdd(&wsum[5], ma + work.masked);
        }
        __syncthreads();
        if (threadIdx.x < 6) atomicAdd(&work_out[threadIdx.x], wsum[threadIdx.x]);
    }
}

// Few hashes of polygons of large area (walks below kBriefWalk / K points), a warp a polygon: Algorithm 1 without
// mask, cells or slab lists for a ring that is staged -- a hash is among its first few dozen
// points, and a box point's test over all the edges is a few instructions a lane.  Bound by
// issue.  149,000 centred polygons of 9 vertices, K = 3: 378 us (763 through the index, 697 with the
// index's earlier form); 100,000 of 317: 676 (1,680, 1,525).
constexpr int kBriefWarps = 8;
constexpr int kBriefChunk = 8;  // slots looked at together, at most
template <bool kCount>
__global__ void __launch_bounds__(kBriefWarps * 32, 4)
sign_brief_kernel(const int2* __restrict__ xy, const int64_t* __restrict__ off, const int4* __restrict__ bbox,
                  const int64_t* __restrict__ area2, const SlabInfo* __restrict__ slabs,
                  const int32_t* __restrict__ slab_ptr, const int32_t* __restrict__ slab_edges,
                  const int32_t* __restrict__ list, int64_t n_slots, const int64_t* __restrict__ d_n,
                  const int* __restrict__ d_flags, uint64_t seed, int K, uint32_t T, float brief_walk,
                  uint32_t* __restrict__ out, unsigned long long* __restrict__ work_out)
{
    __shared__ int2 sv[kBriefWarps][kSmemVerts + 1];
    if (d_flags && *d_flags) return;
    if (d_n) n_slots = min(n_slots, *d_n);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    using W = typename std::conditional<kCount, Work, NoWork>::type;
    W work;
    const int64_t nwarps = (int64_t)gridDim.x * kBriefWarps;
    const int look = (int)max((int64_t)1, min((int64_t)kBriefChunk, n_slots / (2 * nwarps)));
    int64_t chunk = (int64_t)blockIdx.x * kBriefWarps + wid;
    unsigned left = 0;  // slots of the chunk to sign, a lane each
    int64_t lp = 0;     // the lane's polygon
    for (;;) {
        if (!left) {
            const int64_t slot = chunk * look + lane;
            if (chunk * look >= n_slots) break;
            chunk += nwarps;
            bool mine = false;
            if (lane < look && slot < n_slots) {
                lp = list ? (int64_t)list[slot] : slot;
                const int4 bb = bbox[lp];
                mine = bb.z > bb.x && bb.w > bb.y && expected_walk(area2[lp]) < brief_walk;
            }
            left = __ballot_sync(0xffffffffu, mine);
            continue;
        }
        const int64_t p = __shfl_sync(0xffffffffu, lp, __ffs(left) - 1);
        left &= left - 1;
        const int4 bb = bbox[p];
        const int64_t b = off[p];
        const int n = (int)(off[p + 1] - b);
        const uint32_t w = (uint32_t)(bb.z - bb.x), h = (uint32_t)(bb.w - bb.y);
        uint32_t mine = T;
        auto sign = [&](const auto& inside) {
            for (int k = 0; k < K; ++k) {
                const uint64_t sk = pmh_mix64(seed + (uint64_t)(k + 1) * PMH_GAMMA);
                const uint32_t hk = sign_one_t<kIdxU, true>(inside, bb.x, bb.y, w, h, sk, T, lane, work);
                if (lane == k) mine = hk;
            }
        };
        if (n <= kSmemVerts) {
            stage_vertices(sv[wid], xy + b, n, lane);
            sign(AllEdges{sv[wid], n});
        } else {
            const SlabInfo si = slabs ? slabs[p] : SlabInfo{0, 0, 0, 1, 0};
            const GlobalSrc src{xy + b, n, si.S > 0 ? slab_ptr + si.slab_base : nullptr,
                                si.S > 0 ? slab_edges + si.edge_base : nullptr, si.ymin, slab_div_magic(si.slab_h)};
            sign([&](int px, int py, int ln, W& wk) { return warp_inside_src(src, px, py, ln, wk); });
        }
        if (lane < K) out[p * (int64_t)K + lane] = mine;
        __syncwarp();
    }
    if (kCount && work_out && lane == 0) {  // (warp-uniform counts)
        atomicAdd(&work_out[0], work.walk);
        atomicAdd(&work_out[4], work.edges);
    }
}

// The leftover walks.  A walk is cut into segments of kWalkSegment stream points that
// warps take in turn: a warp owns the item its ticket gives it and walks it segment by
// segment; out of items, it helps with the unfinished ones, so that the last few long
// walks (2^32 / area points each: 10^5 for the smallest polygons, up to T for one without
// a lattice point) spread over the device -- walked by the warp that signed the polygon
// they were the tail of the launch: 8,000 coastlines, K = 256, took 4.8 ms and take 0.97,
// 0.10 of it here.  The smallest inside index of all segments is the hash; a segment past the best
// one so far ends the item.  Box points are tested over the polygon's slab or all its
// edges from global memory: most polygons meet a few per walk.  A thin one whose box is a
// thousand times its area meets as many: from kWalkMaskRatio on they go through the coverage
// mask first, and what is left is gathered and tested a lane each where that is cheaper than
// a warp each.  Bound by the generator's integer chain, and by those tests for thin polygons.
constexpr uint32_t kWalkSegment = 4096;
constexpr int kWalkWarps = 8;
constexpr int kWalkBuf = 32 * (kIdxU + 1);  // box points: fewer than 32 kept, and a round's
constexpr float kWalkMaskRatio = 32.0f;     // (a mask costs about as much as a segment's points)
struct WalkWarp {
    uint2 buf[kWalkBuf];  // (stream index << 1 | inside by the mask, x | y << 16), in order
    uint32_t bnd[kMaskN], inb[kMaskN];
};

// a polygon as the walks read it
struct WalkPoly {
    GlobalSrc src;
    int4 bb;
    int edges;    // of one test, about
    int batch;    // box points gathered before they are tested
    bool masked;  // box points go through the mask
    MaskFrame f;
};
template <class W>
__device__ __forceinline__ WalkPoly walk_poly(WalkWarp& m, const int2* xy, const int64_t* off, const int4* bbox,
                                              const int64_t* area2, const SlabInfo* slabs, const int32_t* slab_ptr,
                                              const int32_t* slab_edges, int64_t p, int lane, W& work)
{
    const int64_t b = off[p];
    const int n = (int)(off[p + 1] - b);
    const SlabInfo si = slabs && n > kSmemVerts ? slabs[p] : SlabInfo{0, 0, 0, 1, 0};
    WalkPoly w{{xy + b, n, si.S > 0 ? slab_ptr + si.slab_base : nullptr,
                si.S > 0 ? slab_edges + si.edge_base : nullptr, si.ymin, slab_div_magic(si.slab_h)},
               bbox[p], si.S > 0 ? min(n, 32) : n, 1, false, {}};
    // a walk meets box / area box points on average (of which the mask leaves an eighth or so): an
    // eighth of those to test at a time walks on past the hash by that much at most
    const long long a2 = area2[p];
    const float area = fmaxf(0.5f * (float)(a2 < 0 ? -a2 : a2), 1.0f);
    const float ratio = (float)(w.bb.z - w.bb.x) * (float)(w.bb.w - w.bb.y) / area;
    w.masked = ratio >= kWalkMaskRatio && n <= kMaskMaxEdges;
    w.batch = (int)fminf(fmaxf(ratio * (w.masked ? 1.0f / 64.0f : 0.125f), 1.0f), 32.0f);
    if (w.masked) {
        w.f = mask_frame(w.bb);
        build_mask(m, w.src, n, w.bb, w.f, true, lane, work);
    }
    return w;
}

// the smallest inside index of stream points [a, end), or end
template <class W>
__device__ __forceinline__ uint32_t walk_points(const WalkPoly& P, uint64_t sk, uint32_t a, uint32_t end, WalkWarp& m,
                                                int lane, W& work)
{
    const unsigned full = 0xffffffffu, lt = pmh_lanemask_lt();
    const uint32_t w = (uint32_t)(P.bb.z - P.bb.x), h = (uint32_t)(P.bb.w - P.bb.y);
    const uint64_t step = 32ull * PMH_GAMMA;
    uint64_t z = sk + (uint64_t)(a + lane + 1) * PMH_GAMMA;
    uint32_t found = end;
    int np = 0;  // gathered box points
    for (uint64_t i0 = a;; i0 += 32u * kIdxU) {
        const bool last = i0 >= end;
        bool sure = false;  // a gathered point is inside by the mask
        if (!last) {
            uint32_t pt[kIdxU];
            unsigned box = 0;
#pragma unroll
            for (int j = 0; j < kIdxU; ++j) {
                pt[j] = pmh_mix64_lo(z + (uint64_t)j * step);
                const uint32_t dx = (pt[j] & 0xFFFFu) - (uint32_t)P.bb.x, dy = (pt[j] >> 16) - (uint32_t)P.bb.y;
                box |= (unsigned)((dx < w) & (dy < h)) << j;
            }
            z += (uint64_t)kIdxU * step;
            if (!__any_sync(full, box)) continue;
#pragma unroll
            for (int j = 0; j < kIdxU; ++j) {
                const uint32_t i = (uint32_t)i0 + 32u * j + (uint32_t)lane;
                bool hit = ((box >> j) & 1u) && i < end, in = false;
                if (P.masked && hit) {
                    const int cx = ((int)(pt[j] & 0xFFFFu) - P.f.x0) >> P.f.cwl;
                    const int cy = ((int)(pt[j] >> 16) - P.f.y0) >> P.f.chl;
                    in = (m.inb[cy] >> cx) & 1u;
                    hit = in || ((m.bnd[cy] >> cx) & 1u);
                    work.masked += 1;
                }
                const unsigned bal = __ballot_sync(full, hit);
                if (hit) m.buf[np + __popc(bal & lt)] = make_uint2(2u * i + in, pt[j]);
                np += __popc(bal);
                sure |= in;
            }
            __syncwarp();
        }
        const bool all = last || __any_sync(full, sure);
        int head = 0;
        while (np - head >= P.batch || (all && np > head)) {
            const int count = min(np - head, 32);
            const uint2 c = lane < count ? m.buf[head + lane] : make_uint2(0u, 0u);
            head += count;
            unsigned in = 0;
            // (instructions of a lane's and of the warp's tests)
            if (18 * P.edges < count * (20 * ((P.edges + 31) >> 5) + 25)) {
                const bool inside = lane < count && ((c.x & 1u) || lane_inside(P.src, (int)(c.y & 0xFFFFu),
                                                                               (int)(c.y >> 16), work));
                in = __ballot_sync(full, inside);
            } else {
                for (int t = 0; t < count && !in; ++t) {
                    const uint32_t r = __shfl_sync(full, c.y, t);
                    if ((__shfl_sync(full, c.x, t) & 1u) ||
                        warp_inside_src(P.src, (int)(r & 0xFFFFu), (int)(r >> 16), lane, work)) in = 1u << t;
                }
            }
            if (in) {
                found = __shfl_sync(full, c.x, __ffs(in) - 1) >> 1;
                break;
            }
        }
        if (last || found < end) break;
        if (head > 0) {  // fewer than a batch are left: to the front
            const uint2 c = lane < np - head ? m.buf[head + lane] : make_uint2(0u, 0u);
            np -= head;
            __syncwarp();
            if (lane < np) m.buf[lane] = c;
            __syncwarp();
        }
    }
    __syncwarp();
    work.walk += (found < end ? found + 1 : end) - a;
    return found;
}

template <bool kCount>
__global__ void __launch_bounds__(kWalkWarps * 32, 3)
sign_walks_kernel(const int2* __restrict__ xy, const int64_t* __restrict__ off, const int4* __restrict__ bbox,
                  const int64_t* __restrict__ area2, const SlabInfo* __restrict__ slabs, const int32_t* __restrict__ slab_ptr,
                  const int32_t* __restrict__ slab_edges, const int32_t* __restrict__ list, int64_t n_slots,
                  const int64_t* __restrict__ d_n, const int* __restrict__ d_flags, uint64_t seed, int K, uint32_t T,
                  WalkQueue wq, uint32_t* out, unsigned long long* __restrict__ work_out)
{
    __shared__ WalkWarp smem[kWalkWarps];
    if (d_flags && *d_flags) return;
    const int lane = threadIdx.x & 31;
    WalkWarp& m = smem[threadIdx.x >> 5];
    const unsigned full = 0xffffffffu;
    using W = typename std::conditional<kCount, Work, NoWork>::type;
    W work;
    auto poly = [&](int64_t p) {
        return walk_poly(m, xy, off, bbox, area2, slabs, slab_ptr, slab_edges, p, lane, work);
    };
    auto stream = [&](int k) { return pmh_mix64(seed + (uint64_t)(k + 1) * PMH_GAMMA); };
    const unsigned long long queued = wq.tickets[1];
    const int n = (int)min(queued, (unsigned long long)kWalkItems);
    const int nwarps = (int)(gridDim.x * (blockDim.x >> 5)), warp = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    // the next segment's first index, past the walk's end when the item is finished
    auto ahead = [&](const WalkItem& it, uint32_t next, uint32_t best) {
        const uint64_t a = (uint64_t)it.start + (uint64_t)next * kWalkSegment;
        return a < (uint64_t)min(T, best);
    };
    auto walk_item = [&](int i) {
        WalkItem* it = wq.items + i;
        const WalkItem w = *it;
        uint32_t* res = out + (int64_t)w.p * K + w.k;
        const WalkPoly P = poly(w.p);
        const uint64_t sk = stream(w.k);
        for (;;) {
            uint32_t s = 0, best = 0;
            if (lane == 0) {
                s = atomicAdd(&it->next, 1u);
                best = *reinterpret_cast<volatile uint32_t*>(res);
            }
            s = __shfl_sync(full, s, 0);
            best = __shfl_sync(full, best, 0);
            if (!ahead(w, s, best)) break;
            const uint32_t a = w.start + s * kWalkSegment, end = T - a > kWalkSegment ? a + kWalkSegment : T;
            const uint32_t r = walk_points(P, sk, a, end, m, lane, work);
            if (r < end && lane == 0) atomicMin(res, r);
        }
    };
    for (;;) {
        unsigned long long i = 0;
        if (lane == 0) i = atomicAdd(wq.tickets + 2, 1ull);
        i = __shfl_sync(full, i, 0);
        if (i >= (unsigned long long)n) break;
        walk_item((int)i);
    }
    // help with unfinished items, 32 looked at a time from a place of the warp's own; done
    // after a round of the queue without one
    const int chunks = (n + 31) / 32;
    int c = chunks > 0 ? warp % chunks : 0;
    for (int idle = 0; idle < chunks; c = c + 1 == chunks ? 0 : c + 1) {
        const int i = 32 * c + lane;
        bool todo = false;
        if (i < n) {
            const WalkItem w = wq.items[i];
            todo = ahead(w, *reinterpret_cast<volatile uint32_t*>(&wq.items[i].next),
                         *reinterpret_cast<volatile uint32_t*>(out + (int64_t)w.p * K + w.k));
        }
        unsigned left = __ballot_sync(full, todo);
        if (!left) {
            ++idle;
            continue;
        }
        // (the warps of one chunk spread over its items)
        for (int skip = (warp / chunks) % __popc(left); skip > 0; --skip) left &= left - 1;
        walk_item(32 * c + __ffs(left) - 1);
        idle = 0;
        c = c == 0 ? chunks - 1 : c - 1;  // look at this chunk again
    }
    // past the queue: the marked hashes, a warp each, found in groups of `per` consecutive ones that
    // are handed out in turn: 32, or so few that every warp gets some.  5,000 thin polygons of 8
    // vertices, K = 128 (640,000 walks of 17,000 points, of which 1,400 in the box): 28 ms, 161 with
    // a polygon a warp and a warp a box point; of 64 vertices 35 and 192
    if (queued > (unsigned long long)kWalkItems) {
        if (d_n) n_slots = min(n_slots, *d_n);
        int per = 32;
        while (per > 1 && n_slots * ((K + per - 1) / per) < 4ll * nwarps) per >>= 1;
        const int groups = (K + per - 1) / per;
        for (;;) {
            unsigned long long t = 0;
            if (lane == 0) t = atomicAdd(wq.tickets + 3, 1ull);
            t = __shfl_sync(full, t, 0);
            if ((int64_t)t >= n_slots * groups) break;
            const int64_t slot = (int64_t)t / groups, p = list ? (int64_t)list[slot] : slot;
            const int k0 = (int)((int64_t)t - slot * groups) * per;
            uint32_t* row = out + p * (int64_t)K + k0;
            const bool mine = lane < per && k0 + lane < K;
            unsigned left = __ballot_sync(full, mine && row[mine ? lane : 0] == kNoPoint);
            if (!left) continue;
            const WalkPoly P = poly(p);
            const uint32_t from = (uint32_t)index_level_points(pmh_index_level(P.bb, K));
            while (left) {
                const int j = __ffs(left) - 1;
                left &= left - 1;
                const uint32_t r = walk_points(P, stream(k0 + j), from, T, m, lane, work);
                if (lane == 0) row[j] = r;
            }
        }
    }
    if (kCount && work_out) {
        unsigned long long le = work.lane_edges, ma = work.masked;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            le += __shfl_xor_sync(full, le, o);
            ma += __shfl_xor_sync(full, ma, o);
        }
        if (lane == 0) {  // (the other counts are warp-uniform)
            atomicAdd(&work_out[0], work.walk);
            atomicAdd(&work_out[4], work.edges + le);
            atomicAdd(&work_out[5], ma);
        }
    }
}

}  // namespace

// one persistent launch over `n` slots of `list` (or slot order) with its own ticket
template <UniForm kForm>
static int launch_unified(pmh_ctx ctx, int U, const int2* xy, const int64_t* off, const int4* bbox,
                          const int64_t* area2, const SlabInfo* slabs, const int32_t* slab_ptr,
                          const int32_t* slab_edges, const int32_t* list, int64_t n_slots,
                          int64_t n_chunked, const int64_t* d_n, const int* d_flags, const pmh_params* P,
                          const StreamIndexView& S, const WalkQueue& wq, uint32_t* out,
                          unsigned long long* work, cudaStream_t s)
{
    using Fn = decltype(&sign_unified_kernel<2, true, kForm>);
    // (points per lane per round of the walk form; the staged build has none)
    const Fn fns[3][2] = {{sign_unified_kernel<2, false, kForm>, sign_unified_kernel<2, true, kForm>},
                          {sign_unified_kernel<kForm == UniForm::kStaged ? 2 : 4, false, kForm>,
                           sign_unified_kernel<kForm == UniForm::kStaged ? 2 : 4, true, kForm>},
                          {sign_unified_kernel<kForm == UniForm::kStaged ? 2 : 8, false, kForm>,
                           sign_unified_kernel<kForm == UniForm::kStaged ? 2 : 8, true, kForm>}};
    const Fn fn = fns[U <= 2 ? 0 : U <= 4 ? 1 : 2][work != nullptr];
    int per_sm = 0;
    PMH_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kUniWarps * 32, 0));
    const int chunks = (int)((P->K + 31) / 32);
    const int64_t n_items = n_chunked * chunks + (n_slots - n_chunked);
    int64_t blocks = (int64_t)ctx->sm_count * std::max(per_sm, 1);
    blocks = std::max<int64_t>(1, std::min<int64_t>(blocks, (n_items + kUniWarps - 1) / kUniWarps));
    fn<<<(int)blocks, kUniWarps * 32, 0, s>>>(xy, off, bbox, area2, slabs, slab_ptr, slab_edges, list,
                                              n_slots, n_chunked, d_n, d_flags, P->seed, (int)P->K,
                                              P->T, S, wq, brief_limit((int)P->K), out, work);
    PMH_LAUNCHED(kForm == UniForm::kStaged ? "sign_unified_kernel<staged>" : "sign_unified_kernel");
    return PMH_OK;
}

int pmh_launch_sign_unified(pmh_ctx ctx, int U, const int2* xy, const int64_t* off,
                            const int4* bbox, const int64_t* area2, const SlabInfo* slabs,
                            const int32_t* slab_ptr, const int32_t* slab_edges, const int32_t* list,
                            int64_t n_slots, int64_t n_chunked, int64_t n_indexed_tail,
                            const int64_t* d_n, const int* d_flags, const pmh_params* P,
                            const StreamIndexView& S, const WalkQueue& wq, uint32_t* out,
                            unsigned long long* work, cudaStream_t s)
{
    if (n_slots <= 0) return PMH_OK;
    PMH_CUDA_TRY(cudaMemsetAsync(wq.tickets, 0, sizeof(unsigned long long) * kSignTickets, s));
    // the indexed class at the list's end goes to its own launch (needs the class list)
    const bool classes = list && !d_n;
    const int64_t tail = classes ? std::min(std::max<int64_t>(n_indexed_tail, 0), n_slots - n_chunked) : 0;
    if (S.lv[0].first && area2 && brief_limit((int)P->K) > 0.0f) {
        auto fn = work ? sign_brief_kernel<true> : sign_brief_kernel<false>;
        const int64_t blocks = std::min<int64_t>((n_slots + kBriefWarps - 1) / kBriefWarps, (int64_t)ctx->sm_count * 4);
        fn<<<(unsigned)blocks, kBriefWarps * 32, 0, s>>>(xy, off, bbox, area2, slabs, slab_ptr, slab_edges, list,
                                                         n_slots, d_n, d_flags, P->seed, (int)P->K, P->T,
                                                         brief_limit((int)P->K), out, work);
        PMH_LAUNCHED("sign_brief_kernel");
    }
    if (n_slots - tail > 0) {
        // (the class list's head holds larger rings only)
        auto launch = classes ? launch_unified<UniForm::kLarge> : launch_unified<UniForm::kMixed>;
        PMH_TRY(launch(ctx, U, xy, off, bbox, area2, slabs, slab_ptr, slab_edges, list, n_slots - tail, n_chunked, d_n,
                       d_flags, P, S, wq, out, work, s));
    }
    if (tail > 0) {
        if (n_slots - tail > 0) PMH_CUDA_TRY(cudaMemsetAsync(wq.tickets, 0, sizeof(unsigned long long), s));
        PMH_TRY(launch_unified<UniForm::kStaged>(ctx, U, xy, off, bbox, area2, slabs, slab_ptr, slab_edges,
                                                 list + (n_slots - tail), tail, 0, nullptr, d_flags, P, S, wq, out, work,
                                                 s));
    }
    if (S.lv[0].first) {
        // (three blocks of eight warps per SM: the walks are bound by the generator's integer chain)
        auto fn = work ? sign_walks_kernel<true> : sign_walks_kernel<false>;
        fn<<<ctx->sm_count * 3, kWalkWarps * 32, 0, s>>>(xy, off, bbox, area2, slabs, slab_ptr, slab_edges, list, n_slots, d_n, d_flags,
                                             P->seed, (int)P->K, P->T, wq, out, work);
        PMH_LAUNCHED("sign_walks_kernel");
    }
    return PMH_OK;
}
