// refine.cu -- step A8: exact Jaccard refinement (Sec. 5.2 refinement phase;
// J = area(A n B) / area(A u B), Sec. 1).
//
// area(A n B) by Green's theorem: the boundary of A n B is made of the pieces
// of A's edges inside B and of B's edges inside A, and area = closed integral
// of x dy over it.  Along one edge the pieces need not be sorted: with
// F(t) = dy * (x0 t + dx t^2 / 2) (x dy integrated from the edge start to
// parameter t), an edge that starts inside contributes nothing at t = 0, every
// crossing where it enters the other polygon contributes -F(t), every exit
// +F(t), and an edge that ends inside adds F(1).  Every term is independent,
// so one warp sums them for one pair in any order: each crossing of an A edge
// with a B edge is met once and adds both edges' terms with one reciprocal, and
// the "ends inside" state of an edge is the start state of the next edge.
//
// Degenerate contacts (a vertex on an edge, overlapping collinear edges,
// identical polygons) are resolved by simulation of simplicity: A is taken as
// shifted by (e1, e2), 0 < e2 << e1 infinitesimal.  Every predicate is then
// decided exactly with int64 cross products (coordinates <= 2^20), and the
// area of the shifted configuration tends to the exact one.  The terms are
// fp64 in coordinates relative to B's first vertex, summed exactly.  GB300's fp64 rate is low,
// so the fp64 work is kept to the crossings (a few per edge) and one Newton
// reciprocal each.
#include <cooperative_groups.h>

#include <algorithm>
#include <climits>

#include "pmh_internal.cuh"

namespace cg = cooperative_groups;

namespace {


__device__ __forceinline__ long long cross3(int2 o, int2 a, int2 b)
{
    return (long long)(a.x - o.x) * (b.y - o.y) - (long long)(a.y - o.y) * (b.x - o.x);
}

// sign of orient(c, d, p + e)
__device__ __forceinline__ int side_of_shifted_point(int2 c, int2 d, int2 p)
{
    long long o = cross3(c, d, p);
    if (o != 0) return o > 0 ? 1 : -1;
    int dy = d.y - c.y, dx = d.x - c.x;
    if (dy != 0) return dy > 0 ? -1 : 1;
    return dx > 0 ? 1 : -1;
}

// sign of orient(a + e, b + e, q)
__device__ __forceinline__ int side_of_point_to_shifted(int2 a, int2 b, int2 q)
{
    long long o = cross3(a, b, q);
    if (o != 0) return o > 0 ? 1 : -1;
    int dy = b.y - a.y, dx = b.x - a.x;
    if (dy != 0) return dy > 0 ? 1 : -1;
    return dx > 0 ? -1 : 1;
}

// 1/D in double precision for an integer D != 0 (|D| < 2^44): a single-precision
// reciprocal as the start, then two Newton steps y <- y + y(1 - D y), each of
// which squares the relative error (2^-23 -> 2^-46 -> below double rounding).
// Cheaper on this GPU's narrow fp64 pipe than a correctly rounded division;
// the result is within a few units in the last place, far inside the 1e-9
// relative tolerance of the refinement.
__device__ __forceinline__ double recip(long long D)
{
    const double d = (double)D;
    double y = (double)(1.0f / (float)d);
    double e = fma(-d, y, 1.0);
    y = fma(y, e, y);
    e = fma(-d, y, 1.0);
    return fma(y, e, y);
}

// exact running sum of fp64 terms |x| < 2^44: multiples of 2^-18 and of 2^-56, modulo 2^64
// (sums of integers: the order of the terms does not show)
struct ExactSum {
    unsigned long long q18 = 0, r56 = 0;
    __device__ __forceinline__ void add(double x)
    {
        const long long q = __double2ll_rn(x * 262144.0);
        const double r = fma((double)q, -1.0 / 262144.0, x);  // exact: |r| <= 2^-19
        q18 += (unsigned long long)q;
        r56 += (unsigned long long)__double2ll_rn(r * 72057594037927936.0);
    }
    __device__ __forceinline__ void reduce()  // over the warp, in every lane
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            q18 += __shfl_xor_sync(0xffffffffu, q18, o);
            r56 += __shfl_xor_sync(0xffffffffu, r56, o);
        }
    }
    // the sum plus twice_ends / 2
    __device__ __forceinline__ double total(long long twice_ends) const
    {
        return (double)(long long)(q18 + ((unsigned long long)twice_ends << 17)) * (1.0 / 262144.0) +
               (double)(long long)r56 * (1.0 / 72057594037927936.0);
    }
};

// area(A n B) for one pair, by one warp; returned in every lane.
//  * end terms: edge e_i of the shifted A ends inside B iff its end vertex
//    a_{i+1} + e is inside B (the start state of the next edge), so each lane
//    tests its vertices and adds F(1) of the edge that ends there -- no crossing
//    parity per edge is needed; likewise for B's edges and A + e;
//  * crossings: each (A edge, B edge) pair that crosses is visited by one lane,
//    which adds both boundary terms from one reciprocal: with D = de x df,
//    t = Nt / D on e and u = Nu / D on f (Nt, Nu, D exact integers),
//    F_e(t) = dy t (x0e + dx t / 2) and F_f(u) = ey u (x0f + ex u / 2).
// boundary terms of one crossing, queued as (A edge i, B edge j): with
// D = de x df, t = Nt / D on e and u = Nu / D on f (Nt, Nu, D exact integers),
// F_e(t) = dy t (x0e + dx t / 2) and F_f(u) = ey u (x0f + ex u / 2), signed by
// the direction of the crossing
__device__ __forceinline__ double crossing_terms(const int2* __restrict__ A, int na, int sA,
                                                 const int2* __restrict__ B, int nb, int sB,
                                                 int2 org, uint2 ij)
{
    const int i = (int)ij.x, j = (int)ij.y;
    const int2 a = A[i], b = A[i + 1 == na ? 0 : i + 1];
    const int2 c = B[j], d = B[j + 1 == nb ? 0 : j + 1];
    const int s2 = side_of_shifted_point(c, d, b), s4 = side_of_point_to_shifted(a, b, d);
    const long long dx = b.x - a.x, dy = b.y - a.y, ex = d.x - c.x, ey = d.y - c.y;
    const long long D = dx * ey - dy * ex;
    const long long Nt = (long long)(c.x - a.x) * ey - (long long)(c.y - a.y) * ex;
    const long long Nu = (long long)(c.x - a.x) * dy - (long long)(c.y - a.y) * dx;
    // A's edge: entering B flips the sign; B's edge: entering the shifted A
    const double sa = (((s2 > 0) == (sB > 0)) ? -1.0 : 1.0) * (sA > 0 ? 1.0 : -1.0);
    const double sb = (((s4 > 0) == (sA > 0)) ? -1.0 : 1.0) * (sB > 0 ? 1.0 : -1.0);
    const double r = recip(D);  // D != 0: the edges cross at one point
    const double t = (double)Nt * r, u = (double)Nu * r;
    const double fa = (double)dy * t * ((double)(a.x - org.x) + 0.5 * (double)dx * t);
    const double fb = (double)ey * u * ((double)(c.x - org.x) + 0.5 * (double)ex * u);
    return sa * fa + sb * fb;
}

// One warp's part of area(A n B) for a pair worked on by two warps (wip = 0, 1):
// the end terms of A's vertices (wip 0) or of B's (wip 1), and the crossings of
// the A edges in the 32-edge groups of its parity; summed over the warp.
__device__ double warp_intersection_area(const int2* __restrict__ A, int na, int sA,
                                         const int2* __restrict__ B, int nb, int sB,
                                         uint2* cq /* [64] */, int lane, int wip)
{
    const int2 org = B[0];
    double acc = 0;
    // end terms of A's edges: vertex a_i + e inside B closes edge i-1
    for (int i = wip == 0 ? lane : na; i < na; i += 32) {
        const int2 a = A[i];
        unsigned in = 0;
        for (int j = 0; j < nb; ++j) {
            const int2 c = B[j], d = B[j + 1 == nb ? 0 : j + 1];
            if ((c.y > a.y) != (d.y > a.y)) {
                const long long cr = cross3(c, d, a);
                in ^= (cr != 0) & ((cr > 0) == (d.y > c.y));
            }
        }
        if (in) {
            const int2 p = A[i == 0 ? na - 1 : i - 1];
            const double x0 = (double)(p.x - org.x), dx = (double)(a.x - p.x), dy = (double)(a.y - p.y);
            acc += (sA > 0 ? 1.0 : -1.0) * dy * (x0 + 0.5 * dx);
        }
    }
    // end terms of B's edges: vertex c_j - e inside A closes edge j-1
    for (int j = wip == 1 ? lane : nb; j < nb; j += 32) {
        const int2 c = B[j];
        unsigned in = 0;
        for (int i = 0; i < na; ++i) {
            const int2 a = A[i], b = A[i + 1 == na ? 0 : i + 1];
            if ((a.y >= c.y) != (b.y >= c.y)) {
                const long long cr = cross3(a, b, c);
                in ^= (cr == 0) | ((cr > 0) == (b.y > a.y));
            }
        }
        if (in) {
            const int2 p = B[j == 0 ? nb - 1 : j - 1];
            const double x0 = (double)(p.x - org.x), ex = (double)(c.x - p.x), ey = (double)(c.y - p.y);
            acc += (sB > 0 ? 1.0 : -1.0) * ey * (x0 + 0.5 * ex);
        }
    }
    // crossings: the lanes find them with integer predicates only and queue them
    // (edge indices); the fp64 terms are then evaluated 32 at a time, one
    // crossing per lane, so the narrow fp64 pipe never runs a mostly idle warp
    const unsigned full = 0xffffffffu;
    int nq = 0;  // warp-uniform queue length (< 32 between iterations)
    for (int i0 = 32 * wip; i0 < na; i0 += 64) {
        const int i = i0 + lane;
        int2 a = make_int2(0, 0), b = make_int2(0, 0);
        bool live = i < na;
        if (live) {
            a = A[i];
            b = A[i + 1 == na ? 0 : i + 1];
            live = a.x != b.x || a.y != b.y;
        }
        const int ax0 = min(a.x, b.x), ax1 = max(a.x, b.x), ay0 = min(a.y, b.y), ay1 = max(a.y, b.y);
        for (int j = 0; j < nb; ++j) {
            bool hit = false;
            if (live) {
                const int2 c = B[j], d = B[j + 1 == nb ? 0 : j + 1];
                if (!(max(ax0, min(c.x, d.x)) > min(ax1, max(c.x, d.x)) ||
                      max(ay0, min(c.y, d.y)) > min(ay1, max(c.y, d.y)) || (c.x == d.x && c.y == d.y))) {
                    hit = side_of_shifted_point(c, d, a) != side_of_shifted_point(c, d, b) &&
                          side_of_point_to_shifted(a, b, c) != side_of_point_to_shifted(a, b, d);
                }
            }
            const unsigned bal = __ballot_sync(full, hit);
            if (bal) {
                if (hit) cq[nq + __popc(bal & pmh_lanemask_lt())] = make_uint2((uint32_t)i, (uint32_t)j);
                nq += __popc(bal);
                __syncwarp();
                if (nq >= 32) {
                    acc += crossing_terms(A, na, sA, B, nb, sB, org, cq[lane]);
                    nq -= 32;
                    const uint2 rest = lane < nq ? cq[32 + lane] : make_uint2(0u, 0u);
                    __syncwarp();
                    if (lane < nq) cq[lane] = rest;
                    __syncwarp();
                }
            }
        }
    }
    if (lane < nq) acc += crossing_terms(A, na, sA, B, nb, sB, org, cq[lane]);
    __syncwarp();
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
}

struct PairView {
    const int2* v;
    int n;
    int sgn;
    double area;
};

__device__ __forceinline__ PairView view(const int2* xy, const int64_t* off, const int64_t* area2,
                                         int64_t p)
{
    PairView r;
    int64_t b = off[p];
    r.v = xy + b;
    r.n = (int)(off[p + 1] - b);
    long long a2 = area2[p];
    r.sgn = a2 > 0 ? 1 : (a2 < 0 ? -1 : 0);
    r.area = 0.5 * fabs((double)a2);
    return r;
}

// Cells of the two-warp form: B's edges that meet the two rings' common box, listed in
// every cell of a grid over it that their bounding box meets.  A row of cells is one
// stretch of the lists.  With cells about twice as long as an edge, an A edge meets ~2
// listed edges; y-slabs of any height leave it ~16 (a slab crosses the far side of the
// ring too).  The grid has up to 32 x 32 cells, fewer for few edges (their clearing and
// their prefix sum are paid per pair), and larger cells until the references fit
// kRefCellCap.
constexpr int kGridLog2 = 5;
constexpr int kRefCellCap = 2048;
static_assert(kRefineBigVerts <= kRefCellCap && kRefineBigVerts <= 32 * 32, "one cell holds every edge");
__device__ __forceinline__ int pair_grid_log2(int n) { return n >= 192 ? 5 : n >= 40 ? 4 : 3; }

constexpr int kRefineWarps = 4;  // two pairs per block, two warps per pair
constexpr int kWarpVerts = 1024;  // vertices of a pair's staging slice (seven blocks per SM)
static_assert(kRefineBigVerts <= kWarpVerts, "B is always staged");

// one pair's shared slice: the staged rings, a crossing queue per warp, B's cell lists,
// each ring's crossing parities by edge, and the two warps' partial sums
struct RefPair {
    int2 sv[kWarpVerts];
    // 16-bit counts of the cells, then their ends, then (filled backwards) their first
    // entries; one more holds the end of the last
    uint32_t cell[(1 << (2 * kGridLog2)) / 2 + 4];
    uint32_t cq[2][64];  // queued crossings: edge of A << 16 | edge of B
    uint16_t ids[kRefCellCap];
    uint32_t par_a[32], par_b[32];  // bit i % 32 of word i / 32: edge i is crossed an odd number of times
    int range[2][4];                // min x, max x, min y, max y of A and of B
    unsigned long long q18[2], r56[2];  // each warp's crossing terms (ExactSum)
    double part[2];
    long long ends[2];
    long long e;
    int sum[2];  // each warp's edges in the common box, references
};

// the named barrier of pair slot g (0 or 1) of the block (barrier 0 is __syncthreads;
// immediate ids, so that the block holds three barriers)
__device__ __forceinline__ void pair_sync(int g)
{
    if (g == 0) asm volatile("bar.sync 1, 64;\n" ::: "memory");
    else asm volatile("bar.sync 2, 64;\n" ::: "memory");
}

// n vertices to shared memory by asynchronous 8-byte copies, 64 threads striding
// (the caller waits)
__device__ __forceinline__ void stage_ring(int2* dst, const int2* __restrict__ src, int n, int t)
{
    for (int i = t; i < n; i += 64) {
        const unsigned d = (unsigned)__cvta_generic_to_shared(dst + i);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src + i) : "memory");
    }
}

// a + e inside B (shifted false: a is A's vertex), or c - e inside A (shifted true), by a warp
__device__ __forceinline__ int warp_point_in_ring(int2 p, const int2* v, int n, bool shifted, int lane)
{
    unsigned in = 0;
    for (int e = lane; e < n; e += 32) {
        const int2 c = v[e], d = v[e + 1 == n ? 0 : e + 1];
        if (shifted ? (c.y >= p.y) != (d.y >= p.y) : (c.y > p.y) != (d.y > p.y)) {
            const long long cr = cross3(c, d, p);
            in ^= shifted ? (cr == 0) | ((cr > 0) == (d.y > c.y)) : (cr != 0) & ((cr > 0) == (d.y > c.y));
        }
    }
    return __popc(__ballot_sync(0xffffffffu, in)) & 1;
}

// twice the end terms of a ring's edges: edge i ends inside the other ring iff its end
// vertex's state -- the first vertex's, flipped by every crossing of edges 0 .. i -- is
// inside; integers (by one warp, summed over its lanes)
__device__ __forceinline__ long long ring_ends(const int2* v, int n, const uint32_t* par, int inside, int org_x,
                                               int lane)
{
    long long sum = 0;
    const unsigned le = pmh_lanemask_lt() | (1u << lane);
    for (int i0 = 0; i0 < n; i0 += 32) {
        const uint32_t w = par[i0 >> 5];
        const int i = i0 + lane;
        if (i < n && ((inside ^ __popc(w & le)) & 1)) {
            const int2 a = v[i], b = v[i + 1 == n ? 0 : i + 1];
            sum += (long long)(b.y - a.y) * (2 * (a.x - org_x) + (b.x - a.x));
        }
        inside ^= __popc(w) & 1;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    return sum;
}

// the common box of a pair and its grid of cells
struct PairGrid {
    int rx0, rx1, ry0, ry1, lg, shx, shy;
    // cells of edge (a, b): columns c0 .. c1 of rows r0 .. r1; false: outside the box
    __device__ __forceinline__ bool cells(int2 a, int2 b, int& c0, int& c1, int& r0, int& r1) const
    {
        const int x0 = max(min(a.x, b.x), rx0), x1 = min(max(a.x, b.x), rx1);
        const int y0 = max(min(a.y, b.y), ry0), y1 = min(max(a.y, b.y), ry1);
        c0 = (x0 - rx0) >> shx;
        c1 = (x1 - rx0) >> shx;
        r0 = (y0 - ry0) >> shy;
        r1 = (y1 - ry0) >> shy;
        return x0 <= x1 && y0 <= y1;
    }
};

// B's cell lists over the common box, by the pair's 64 threads (t)
__device__ __forceinline__ void build_pair_cells(const int2* v, int n, PairGrid& G, RefPair& P, int t, int g)
{
    const unsigned full = 0xffffffffu;
    const int lane = t & 31, wip = t >> 5;
    const int words = 1 << (2 * G.lg - 1);  // two cells each
    const int per = max(words >> 6, 1);     // words per thread of the prefix sum (8, 2 or 1)
    while (((G.rx1 - G.rx0) >> G.shx) >> G.lg) ++G.shx;
    while (((G.ry1 - G.ry0) >> G.shy) >> G.lg) ++G.shy;
    for (;; ++G.shx, ++G.shy) {
        for (int i = t; i < words; i += 64) P.cell[i] = 0;
        pair_sync(g);
        for (int e = t; e < n; e += 64) {
            int c0, c1, r, r1;
            if (!G.cells(v[e], v[e + 1 == n ? 0 : e + 1], c0, c1, r, r1)) continue;
            for (; r <= r1; ++r)
                for (int c = (r << G.lg) + c0; c <= (r << G.lg) + c1; ++c)
                    atomicAdd(&P.cell[c >> 1], 1u << (16 * (c & 1)));
        }
        pair_sync(g);
        // counts to ends: each thread's words, then the warp's and the pair's prefix
        const int w0 = t * per;
        int mine = 0;
        if (w0 < words)
            for (int u = 0; u < per; ++u) {
                const uint32_t w = P.cell[w0 + u];
                mine += (int)(w & 0xFFFFu) + (int)(w >> 16);
            }
        int x = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(full, x, d);
            if (lane >= d) x += y;
        }
        if (lane == 31) P.sum[wip] = x;
        pair_sync(g);
        const int total = P.sum[0] + P.sum[1];
        if (total > kRefCellCap) {  // (one cell holds at most n <= kRefineBigVerts)
            pair_sync(g);
            continue;
        }
        int run = x - mine + (wip ? P.sum[0] : 0);
        if (w0 < words)
            for (int u = 0; u < per; ++u) {
                const uint32_t w = P.cell[w0 + u];
                const int lo = run + (int)(w & 0xFFFFu), hi = lo + (int)(w >> 16);
                P.cell[w0 + u] = (uint32_t)lo | ((uint32_t)hi << 16);
                run = hi;
            }
        if (t == 0) P.cell[words] = (uint32_t)total;
        pair_sync(g);
        break;
    }
    for (int e = t; e < n; e += 64) {
        int c0, c1, r, r1;
        if (!G.cells(v[e], v[e + 1 == n ? 0 : e + 1], c0, c1, r, r1)) continue;
        for (; r <= r1; ++r)
            for (int c = (r << G.lg) + c0; c <= (r << G.lg) + c1; ++c) {
                const uint32_t old = atomicSub(&P.cell[c >> 1], 1u << (16 * (c & 1)));
                P.ids[((old >> (16 * (c & 1))) & 0xFFFFu) - 1] = (uint16_t)e;
            }
    }
    pair_sync(g);
}

// J of one pair by two warps (wip = 0, 1; every branch is uniform over both), rings of at
// most kRefineBigVerts vertices: B staged in the pair's shared slice, A too when both fit.
// B's edges are listed by the cells of the rings' common box.  The warps take alternate
// 32-edge groups of A's edges; a group's (edge, listed edge) visits are spread over the
// lanes by a warp scan, so that no lane waits for the longest list, and the crossings
// found are queued (their fp64 terms are evaluated 32 at a time) and flip both edges'
// parities.  Each ring's first vertex is tested against the other ring; the state of
// every other vertex follows from the parities along its ring (each crossing moves an
// edge across the other boundary; the predicates are exact, so the parities are), which
// leaves the end terms as one pass of integer sums.  The crossings' terms are summed as
// integers too (ExactSum), so the lists' order (atomics of two warps) does not show.
// Bound by issue and by the latency of dependent shared-memory and integer chains.
// 77,824 pairs of 8 to 1,024 vertices (4,096 lists of 19): 0.71 ms; 1.10 with y-slabs listed
// by one warp and a lane per edge, of which the listing took a third.
__device__ double pair_jaccard(PairView A, PairView B, RefPair& P, int wip, int lane, int g)
{
    if (A.sgn == 0 || B.sgn == 0) return 0.0;
    const unsigned full = 0xffffffffu;
    const int t = 32 * wip + lane;
    double inter;
    if (max(A.n, B.n) > kRefineBigVerts) {  // (large rings where no queue takes them)
        const double part = warp_intersection_area(A.v, A.n, A.sgn, B.v, B.n, B.sgn,
                                                   reinterpret_cast<uint2*>(P.sv) + 64 * wip, lane, wip);
        if (lane == 0) P.part[wip] = part;
        pair_sync(g);
        inter = P.part[0] + P.part[1];
    } else {
        const bool sa = A.n + B.n <= kWarpVerts;
        stage_ring(P.sv, B.v, B.n, t);
        if (sa) stage_ring(P.sv + B.n, A.v, A.n, t);
        P.par_a[lane] = 0;  // (both warps write the same zeros)
        P.par_b[lane] = 0;
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        pair_sync(g);
        const int2* b = P.sv;
        const int2* a = sa ? P.sv + B.n : A.v;
        {  // warp 0: A's range; warp 1: B's
            const int2* v = wip == 0 ? a : b;
            const int n = wip == 0 ? A.n : B.n;
            int x0 = INT_MAX, x1 = INT_MIN, y0 = INT_MAX, y1 = INT_MIN;
            for (int i = lane; i < n; i += 32) {
                const int2 u = v[i];
                x0 = min(x0, u.x);
                x1 = max(x1, u.x);
                y0 = min(y0, u.y);
                y1 = max(y1, u.y);
            }
            x0 = __reduce_min_sync(full, x0);
            x1 = __reduce_max_sync(full, x1);
            y0 = __reduce_min_sync(full, y0);
            y1 = __reduce_max_sync(full, y1);
            if (lane == 0) {
                P.range[wip][0] = x0;
                P.range[wip][1] = x1;
                P.range[wip][2] = y0;
                P.range[wip][3] = y1;
            }
        }
        pair_sync(g);
        PairGrid G{max(P.range[0][0], P.range[1][0]), min(P.range[0][1], P.range[1][1]),
                   max(P.range[0][2], P.range[1][2]), min(P.range[0][3], P.range[1][3]), 0, 0, 0};
        if (G.rx0 > G.rx1 || G.ry0 > G.ry1) return 0.0;
        // B's edges in the box (the grid's size), and the first vertices' states
        int nb = 0;
        for (int e0 = 32 * wip; e0 < B.n; e0 += 64) {
            const int e = e0 + lane;
            int c0, c1, r0, r1;
            const bool in = e < B.n && G.cells(b[e], b[e + 1 == B.n ? 0 : e + 1], c0, c1, r0, r1);
            nb += __popc(__ballot_sync(full, in));
        }
        if (lane == 0) P.sum[wip] = nb;
        // (warp 0: the first vertex of A inside B; warp 1: that of B inside A)
        const int in0 = wip == 0 ? warp_point_in_ring(a[0], b, B.n, false, lane)
                                 : warp_point_in_ring(b[0], a, A.n, true, lane);
        pair_sync(g);
        G.lg = pair_grid_log2(P.sum[0] + P.sum[1]);
        build_pair_cells(b, B.n, G, P, t, g);
        const uint16_t* beg = reinterpret_cast<const uint16_t*>(P.cell);
        const int2 org = b[0];
        uint32_t* cq = P.cq[wip];
        ExactSum sum;
        int nq = 0;  // warp-uniform queue length (< 32 between iterations)
        for (int i0 = 32 * wip; i0 < A.n; i0 += 64) {
            int c0 = 0, c1 = -1, r0 = 0, r1 = -1;  // the lane's edge's cells (none)
            if (i0 + lane < A.n) {
                const int2 u = a[i0 + lane], w = a[i0 + lane + 1 == A.n ? 0 : i0 + lane + 1];
                if (!G.cells(u, w, c0, c1, r0, r1) || (u.x == w.x && u.y == w.y)) r1 = r0 - 1;
            }
            const int rows = __reduce_max_sync(full, r1 - r0 + 1);
            const int first = (r0 << 16) | c0;
            for (int dr = 0; dr < rows; ++dr) {
                int k0 = 0, len = 0;  // the row's stretch of the lists
                if (r0 + dr <= r1) {
                    const int row = (r0 + dr) << G.lg;
                    k0 = beg[row + c0];
                    len = beg[row + c1 + 1] - k0;
                }
                int excl = len;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int y = __shfl_up_sync(full, excl, d);
                    if (lane >= d) excl += y;
                }
                const int visits = __shfl_sync(full, excl, 31);
                excl -= len;
                const int shift = k0 - excl;  // list position of visit x of this lane's edge: x + shift
                for (int x0 = 0; x0 < visits; x0 += 32) {
                    const int x = x0 + lane;
                    int own = 0;  // the last lane whose first visit is <= x
#pragma unroll
                    for (int step = 16; step >= 1; step >>= 1)
                        if (__shfl_sync(full, excl, own + step) <= x) own += step;
                    const int k = x + __shfl_sync(full, shift, own);
                    const int of = __shfl_sync(full, first, own);
                    bool hit = false;
                    int j = 0;
                    const int i = i0 + own;
                    if (x < visits) {
                        j = P.ids[k];
                        const int2 c = b[j], d = b[j + 1 == B.n ? 0 : j + 1];
                        const int2 u = a[i], w = a[i + 1 == A.n ? 0 : i + 1];
                        const int dx0 = min(c.x, d.x), dy0 = min(c.y, d.y);
                        if (!(max(min(u.x, w.x), dx0) > min(max(u.x, w.x), max(c.x, d.x)) ||
                              max(min(u.y, w.y), dy0) > min(max(u.y, w.y), max(c.y, d.y)) ||
                              (c.x == d.x && c.y == d.y))) {
                            // this pair is visited once: in the first cell listed for both
                            const int ur = of >> 16, uc = of & 0xFFFF;
                            const int cell = ((ur + dr) << G.lg) + max(uc, (max(dx0, G.rx0) - G.rx0) >> G.shx);
                            if (ur + dr == max(ur, (max(dy0, G.ry0) - G.ry0) >> G.shy) && k >= beg[cell] && k < beg[cell + 1])
                                hit = side_of_shifted_point(c, d, u) != side_of_shifted_point(c, d, w) &&
                                      side_of_point_to_shifted(u, w, c) != side_of_point_to_shifted(u, w, d);
                        }
                    }
                    const unsigned bal = __ballot_sync(full, hit);
                    if (bal) {
                        if (hit) {
                            atomicXor(&P.par_a[i >> 5], 1u << (i & 31));
                            atomicXor(&P.par_b[j >> 5], 1u << (j & 31));
                            cq[nq + __popc(bal & pmh_lanemask_lt())] = ((uint32_t)i << 16) | (uint32_t)j;
                        }
                        nq += __popc(bal);
                        __syncwarp();
                        if (nq >= 32) {
                            const uint32_t ij = cq[lane];
                            sum.add(crossing_terms(a, A.n, A.sgn, b, B.n, B.sgn, org, make_uint2(ij >> 16, ij & 0xFFFFu)));
                            nq -= 32;
                            const uint32_t rest = lane < nq ? cq[32 + lane] : 0u;
                            __syncwarp();
                            if (lane < nq) cq[lane] = rest;
                            __syncwarp();
                        }
                    }
                }
            }
        }
        if (lane < nq) {
            const uint32_t ij = cq[lane];
            sum.add(crossing_terms(a, A.n, A.sgn, b, B.n, B.sgn, org, make_uint2(ij >> 16, ij & 0xFFFFu)));
        }
        sum.reduce();
        if (lane == 0) {
            P.q18[wip] = sum.q18;
            P.r56[wip] = sum.r56;
        }
        pair_sync(g);
        const long long ends = wip == 0 ? A.sgn * ring_ends(a, A.n, P.par_a, in0, org.x, lane)
                                        : B.sgn * ring_ends(b, B.n, P.par_b, in0, org.x, lane);
        if (lane == 0) P.ends[wip] = ends;
        pair_sync(g);
        inter = ExactSum{P.q18[0] + P.q18[1], P.r56[0] + P.r56[1]}.total(P.ends[0] + P.ends[1]);
    }
    const double uni = A.area + B.area - inter;
    return uni > 0 ? fmin(fmax(inter / uni, 0.0), 1.0) : 0.0;
}

__global__ void __launch_bounds__(kRefineWarps * 32, 7)
refine_pairs_kernel(const int2* __restrict__ qxy, const int64_t* __restrict__ qoff,
                    const int64_t* __restrict__ qarea2, const int4* __restrict__ qbox,
                    const int2* __restrict__ pxy, const int64_t* __restrict__ poff,
                    const int64_t* __restrict__ parea2, const int4* __restrict__ pbox,
                    const int32_t* __restrict__ ids, const int32_t* __restrict__ nlist, int m,
                    const int32_t* __restrict__ qid_list, int64_t e0, int64_t n_pairs, double* __restrict__ out,
                    unsigned long long* __restrict__ ticket /* [0]: pairs, [1]: queued pairs */,
                    int32_t* __restrict__ big, const int64_t* __restrict__ d_n)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int g = wid >> 1, wip = wid & 1;
    RefPair& P = reinterpret_cast<RefPair*>(smem_raw)[g];
    // pairs [e0, n_pairs) of the call, those of the live queries
    if (d_n && !qid_list) n_pairs = min(n_pairs, *d_n * (int64_t)m);
    // persistent warp pairs pull pairs from a ticket: pair costs differ by orders of
    // magnitude (a query against its own source vs a neighbour it barely touches)
    for (;;) {
        if (wip == 0 && lane == 0) P.e = (long long)atomicAdd(ticket, 1ull);
        pair_sync(g);
        const int64_t e = e0 + P.e;
        if (e >= n_pairs) break;  // the same for both warps
        int64_t q;
        int32_t p;
        double j = -1.0;
        bool live = true;
        if (qid_list) {  // explicit pairs
            q = qid_list[e];
            p = ids[e];
        } else {         // top-m lists: pair e = (q, slot)
            q = e / m;
            const int slot = (int)(e - q * m);
            live = slot < nlist[q];
            p = live ? ids[e] : 0;
        }
        if (live) {
            // bounding boxes (half-open lattice boxes) without a common interior point:
            // an empty intersection, J = 0 exactly, as the full computation gives
            const int4 qa = qbox[q], pb = pbox[p];
            const bool apart = !(qa.x < pb.z && pb.x < qa.z && qa.y < pb.w && pb.y < qa.w);
            const PairView A = view(qxy, qoff, qarea2, q), B = view(pxy, poff, parea2, p);
            if (!apart && big && max(A.n, B.n) > kRefineBigVerts) {
                if (wip == 0 && lane == 0) big[atomicAdd(ticket + 1, 1ull)] = (int32_t)(e - e0);
                pair_sync(g);
                continue;  // refine_big_kernel takes the pair
            }
            j = apart ? 0.0 : pair_jaccard(A, B, P, wip, lane, g);
        }
        if (wip == 0 && lane == 0) out[e] = j;
        pair_sync(g);  // the slice is free for the next pair
    }
}

// ---------------------------------------------------------------------------
// Pairs with a ring above kRefineBigVerts vertices: a cluster each.  The two-warp form
// keeps both rings' slab lists in 2,048 shared references; above ~1,700 vertices they
// overflow and every edge pair was tested (n * m predicates by 64 threads).  Here a
// ring's lists are the y-slab index of its set (slabs.cu: about n / 4 slabs, read from
// L2), or lists built in shared memory for a ring without one, so that a vertex or an
// edge meets only the few edges of its own rows.  The index lists an edge in the slabs
// of its rows [min y, max y) and leaves horizontal edges out, so
//  * a vertex a of A (+e) sees B's edges straddling the row of a.y: slab of a.y;
//  * a vertex c of B sees the shifted A's edges with min < c.y <= max: slab of c.y - 1;
//  * an A edge meets B's non-horizontal edges in the slabs from its lowest to its
//    highest row (a crossing of the shifted edge lies strictly inside B's rows, or just
//    below B's top vertex), each pair in the first slab that lists both; or every edge of B
//    once, if those lists hold more (spiky rings, whose edges are listed in hundreds of slabs:
//    1,200 pairs of stars of 1,800 to 4,000 vertices 44 ms by the lists, 7.8);
//  * a horizontal edge of B meets the A edges with min < y <= max: slab of y - 1.
// The end terms are integers (twice dy (x0 + dx / 2)), the crossings' fp64 terms are
// added as two integers (multiples of 2^-18, and the remainder's of 2^-56, modulo 2^64):
// sums of integers do not depend on their order, so neither the list order (atomics)
// nor the split over the threads shows in the result.
// Bound by the latency of list entry -> two vertices, from L1/L2, and by each vertex's own
// list.  Two blocks a pair: with one the launch ended with its largest pairs, with four or eight
// the shared set-up weighed more.  512 pairs of coastlines of 4 to 16,384 vertices: 0.53 ms;
// 0.82 with one block, 0.62 with four, 0.83 with eight; 153 ms in the two-warp form.
// ---------------------------------------------------------------------------
constexpr int kBigThreads = 512;  // per block of a pair's cluster
constexpr int kBigBlocks = 1024 / kBigThreads;  // resident an SM
constexpr int kBigCluster = 2;
constexpr int kBigWarps = kBigThreads / 32;
constexpr int kBigCap = 2048;     // shared references of a ring without a slab index
constexpr int kBigSlabs = 256;

// a ring and its edge lists: sp / se in global memory (slab index) or shared memory;
// sp == nullptr: one list of every edge
struct ListRing {
    const int2* v;
    int n;
    const int32_t* sp;
    const int32_t* se;
    int S, y0;
    uint64_t magic;
    int x0, x1;  // the ring's x-range
    __device__ __forceinline__ int2 vert(int e) const { return v[e == n ? 0 : e]; }
    // list positions of the edges whose rows [min y, max y) can hold row y
    __device__ __forceinline__ void row(int y, int& lo, int& hi) const
    {
        lo = hi = 0;
        if (!sp) {
            hi = n;
            return;
        }
        if (y < y0) return;
        const int q = slab_div(y - y0, magic);
        if (q >= S) return;
        lo = sp[q];
        hi = sp[q + 1];
    }
    __device__ __forceinline__ int edge(int t) const { return sp ? se[t] : t; }
};

struct BigSmem {
    uint2 cq[kBigWarps][64];
    int32_t ids[2][kBigCap];
    int32_t beg[2][kBigSlabs + 1];
    int cnt[2][kBigSlabs];
    int range[2][4];  // min x, max x, min y, max y of each ring
    int listed[2], sh[2];
    unsigned long long ends, q18, r56;
    long long e;
};

// the lists of a ring without a slab index (of at most kBigCap references), by one
// warp: slabs of 2^sh rows from the ring's lowest vertex
__device__ bool build_big_lists(const int2* v, int n, int y0, int y1, int32_t* ids, int32_t* beg, int* cnt,
                                int& sh_out, int lane)
{
    int sh = 0;
    while (((y1 - y0) >> sh) >= kBigSlabs) ++sh;
    for (int s = lane; s < kBigSlabs; s += 32) cnt[s] = 0;
    __syncwarp();
    for (int pass = 0; pass < 2; ++pass) {
        for (int e = lane; e < n; e += 32) {
            const int2 a = v[e], b = v[e + 1 == n ? 0 : e + 1];
            if (a.y == b.y) continue;
            const int s0 = (min(a.y, b.y) - y0) >> sh, s1 = (max(a.y, b.y) - 1 - y0) >> sh;
            for (int s = s0; s <= s1; ++s) {
                const int t = atomicAdd(&cnt[s], 1);
                if (pass) ids[t] = e;
            }
        }
        __syncwarp();
        if (pass) break;
        int carry = 0;
        for (int s0 = 0; s0 < kBigSlabs; s0 += 32) {
            const int c = cnt[s0 + lane];
            int x = c;
            for (int d = 1; d < 32; d <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, x, d);
                if (lane >= d) x += t;
            }
            beg[s0 + lane] = cnt[s0 + lane] = carry + x - c;
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
        if (carry > kBigCap) return false;
        if (lane == 0) beg[kBigSlabs] = carry;
        __syncwarp();
    }
    sh_out = sh;
    return true;
}

__device__ __forceinline__ bool edges_cross(int2 a, int2 b, int2 c, int2 d)
{
    if (max(min(a.x, b.x), min(c.x, d.x)) > min(max(a.x, b.x), max(c.x, d.x)) ||
        max(min(a.y, b.y), min(c.y, d.y)) > min(max(a.y, b.y), max(c.y, d.y)))
        return false;
    return side_of_shifted_point(c, d, a) != side_of_shifted_point(c, d, b) &&
           side_of_point_to_shifted(a, b, c) != side_of_point_to_shifted(a, b, d);
}

// queue the lanes' hits (edge of A, edge of B); evaluate 32 at a time
__device__ __forceinline__ void push_crossings(bool hit, int i, int j, uint2* cq, int& nq, const ListRing& A,
                                               int sA, const ListRing& B, int sB, int2 org, ExactSum& sum,
                                               int lane)
{
    const unsigned bal = __ballot_sync(0xffffffffu, hit);
    if (!bal) return;
    if (hit) cq[nq + __popc(bal & pmh_lanemask_lt())] = make_uint2((uint32_t)i, (uint32_t)j);
    nq += __popc(bal);
    __syncwarp();
    if (nq >= 32) {
        sum.add(crossing_terms(A.v, A.n, sA, B.v, B.n, sB, org, cq[lane]));
        nq -= 32;
        const uint2 rest = lane < nq ? cq[32 + lane] : make_uint2(0u, 0u);
        __syncwarp();
        if (lane < nq) cq[lane] = rest;
        __syncwarp();
    }
}

__global__ void __cluster_dims__(kBigCluster, 1, 1) __launch_bounds__(kBigThreads, kBigBlocks)
refine_big_kernel(const int2* __restrict__ qxy, const int64_t* __restrict__ qoff,
                  const int64_t* __restrict__ qarea2, const SlabPtrs* __restrict__ qslabs,
                  const int2* __restrict__ pxy, const int64_t* __restrict__ poff,
                  const int64_t* __restrict__ parea2, const SlabPtrs* __restrict__ pslabs,
                  const int32_t* __restrict__ ids, int m, const int32_t* __restrict__ qid_list, int64_t e0,
                  double* __restrict__ out, unsigned long long* __restrict__ ticket /* [1], [2] */,
                  const int32_t* __restrict__ big)
{
    __shared__ BigSmem s;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const long long queued = (long long)ticket[1];
    // the cluster's blocks share a pair: its vertices and edges are dealt to their threads in turn,
    // its ranges and sums are added up in their shared memories
    const cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), ctid = rank * kBigThreads + tid;
    constexpr int kStride = kBigThreads * kBigCluster;
    for (;;) {
        cl.sync();
        if (tid == 0 && rank == 0) {
            const long long next = (long long)atomicAdd(ticket + 2, 1ull);
            for (int r = 0; r < kBigCluster; ++r) *cl.map_shared_rank(&s.e, r) = next;
        }
        if (tid < 2) {
            s.range[tid][0] = s.range[tid][2] = INT_MAX;
            s.range[tid][1] = s.range[tid][3] = INT_MIN;
        }
        if (tid == 0) s.ends = s.q18 = s.r56 = 0;
        cl.sync();
        if (s.e >= queued) break;
        const int64_t e = e0 + big[s.e];
        const int64_t q = qid_list ? (int64_t)qid_list[e] : e / m;
        const int64_t p = ids[e];
        const PairView va = view(qxy, qoff, qarea2, q), vb = view(pxy, poff, parea2, p);
        if (va.sgn == 0 || vb.sgn == 0) {  // (uniform over the cluster)
            if (ctid == 0) out[e] = 0.0;
            continue;
        }
        // both rings' ranges
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int2* v = r ? vb.v : va.v;
            const int n = r ? vb.n : va.n;
            int x0 = INT_MAX, x1 = INT_MIN, y0 = INT_MAX, y1 = INT_MIN;
#pragma unroll 4
            for (int i = ctid; i < n; i += kStride) {
                const int2 u = v[i];
                x0 = min(x0, u.x);
                x1 = max(x1, u.x);
                y0 = min(y0, u.y);
                y1 = max(y1, u.y);
            }
            x0 = __reduce_min_sync(0xffffffffu, x0);
            x1 = __reduce_max_sync(0xffffffffu, x1);
            y0 = __reduce_min_sync(0xffffffffu, y0);
            y1 = __reduce_max_sync(0xffffffffu, y1);
            if (lane < kBigCluster) {
                int* range = cl.map_shared_rank(s.range[r], lane);
                atomicMin(range + 0, x0);
                atomicMax(range + 1, x1);
                atomicMin(range + 2, y0);
                atomicMax(range + 3, y1);
            }
        }
        cl.sync();
        ListRing A{va.v, va.n, nullptr, nullptr, 0, 0, 0, s.range[0][0], s.range[0][1]};
        ListRing B{vb.v, vb.n, nullptr, nullptr, 0, 0, 0, s.range[1][0], s.range[1][1]};
        // lists: the set's slab index, else shared lists (warp r builds ring r's), else
        // every edge
        const SlabInfo sia = qslabs && qslabs->info ? qslabs->info[q] : SlabInfo{0, 0, 0, 1, 0};
        const SlabInfo sib = pslabs && pslabs->info ? pslabs->info[p] : SlabInfo{0, 0, 0, 1, 0};
        if (wid < 2 && (wid ? sib.S : sia.S) == 0) {
            int sh = 0;
            const bool ok = build_big_lists(wid ? B.v : A.v, wid ? B.n : A.n, s.range[wid][2], s.range[wid][3],
                                            s.ids[wid], s.beg[wid], s.cnt[wid], sh, lane);
            if (lane == 0) {
                s.listed[wid] = ok;
                s.sh[wid] = sh;
            }
        }
        __syncthreads();
        auto lists = [&](ListRing& R, const SlabInfo& si, const SlabPtrs* sl, int r) {
            if (si.S > 0) {
                R.sp = sl->ptr + si.slab_base;
                R.se = sl->edges + si.edge_base;
                R.S = si.S;
                R.y0 = si.ymin;
                R.magic = slab_div_magic(si.slab_h);
            } else if (s.listed[r]) {
                R.sp = s.beg[r];
                R.se = s.ids[r];
                R.S = kBigSlabs;
                R.y0 = s.range[r][2];
                R.magic = slab_div_magic(1 << s.sh[r]);
            }
        };
        lists(A, sia, qslabs, 0);
        lists(B, sib, pslabs, 1);
        const int ya0 = s.range[0][2], ya1 = s.range[0][3], yb0 = s.range[1][2], yb1 = s.range[1][3];
        const int2 org = B.v[0];
        long long ends = 0;  // twice the end terms
        ExactSum sum;
        // end terms of A's edges: vertex a_i + e inside B closes edge i - 1
        for (int i = ctid; i < A.n; i += kStride) {
            const int2 a = A.v[i];
            if (a.y < yb0 || a.y > yb1 || a.x < B.x0 || a.x > B.x1) continue;
            int lo, hi;
            B.row(a.y, lo, hi);
            unsigned in = 0;
#pragma unroll 2
            for (int t = lo; t < hi; ++t) {
                const int j = B.edge(t);
                const int2 c = B.v[j], d = B.vert(j + 1);
                if ((c.y > a.y) != (d.y > a.y)) {
                    const long long cr = cross3(c, d, a);
                    in ^= (cr != 0) & ((cr > 0) == (d.y > c.y));
                }
            }
            if (in) {
                const int2 u = A.v[i == 0 ? A.n - 1 : i - 1];
                ends += va.sgn * (long long)(a.y - u.y) * (2 * (u.x - org.x) + (a.x - u.x));
            }
        }
        // end terms of B's edges: vertex c_j - e inside A closes edge j - 1
        for (int j = ctid; j < B.n; j += kStride) {
            const int2 c = B.v[j];
            if (c.y < ya0 || c.y > ya1 || c.x < A.x0 || c.x > A.x1) continue;
            int lo, hi;
            A.row(c.y - 1, lo, hi);
            unsigned in = 0;
#pragma unroll 2
            for (int t = lo; t < hi; ++t) {
                const int i = A.edge(t);
                const int2 a = A.v[i], b = A.vert(i + 1);
                if ((a.y >= c.y) != (b.y >= c.y)) {
                    const long long cr = cross3(a, b, c);
                    in ^= (cr == 0) | ((cr > 0) == (b.y > a.y));
                }
            }
            if (in) {
                const int2 u = B.v[j == 0 ? B.n - 1 : j - 1];
                ends += vb.sgn * (long long)(c.y - u.y) * (2 * (u.x - org.x) + (c.x - u.x));
            }
        }
        // crossings of A's edges with B's non-horizontal edges
        int nq = 0;  // warp-uniform queue length
        for (int i0 = ctid & ~31; i0 < A.n; i0 += kStride) {
            const int i = i0 + lane;
            int2 a = make_int2(0, 0), b = make_int2(0, 0);
            int k0 = 0, cntk = 0, q0 = 0;
            bool all = !B.sp;  // every edge of B, instead of the lists
            if (i < A.n) {
                a = A.v[i];
                b = A.vert(i + 1);
                const int lo = max(min(a.y, b.y), yb0), hi = min(max(a.y, b.y), yb1);
                if ((a.x != b.x || a.y != b.y) && hi >= lo && max(a.x, b.x) >= B.x0 && min(a.x, b.x) <= B.x1) {
                    cntk = B.n;
                    if (B.sp) {
                        q0 = slab_div(lo - B.y0, B.magic);
                        const int q1 = min(slab_div(hi - B.y0, B.magic), B.S - 1);
                        const int listed = q0 <= q1 ? B.sp[q1 + 1] - B.sp[q0] : 0;
                        // (long edges of both rings, as of spiky ones: an edge is listed in every slab
                        // it meets, and its lists exceed the ring)
                        all = listed > B.n;
                        if (!all) {
                            k0 = listed > 0 ? B.sp[q0] : 0;
                            cntk = listed;
                        }
                    }
                }
            }
            const int steps = __reduce_max_sync(0xffffffffu, cntk);
            int qs = q0;  // slab of list position k0 + t
            for (int t = 0; t < steps; ++t) {
                bool hit = false;
                int j = 0;
                if (t < cntk) {
                    const int k = k0 + t;
                    j = all ? t : B.se[k];
                    const int2 c = B.v[j], d = B.vert(j + 1);
                    bool once = c.y != d.y;
                    if (!all) {
                        while (k >= B.sp[qs + 1]) ++qs;
                        once = once && qs == max(q0, slab_div(min(c.y, d.y) - B.y0, B.magic));
                    }
                    hit = once && edges_cross(a, b, c, d);
                }
                push_crossings(hit, i, j, s.cq[wid], nq, A, va.sgn, B, vb.sgn, org, sum, lane);
            }
        }
        // crossings of B's horizontal edges with A's edges
        for (int j0 = ctid & ~31; j0 < B.n; j0 += kStride) {
            const int j = j0 + lane;
            int2 c = make_int2(0, 0), d = make_int2(0, 0);
            int lo = 0, hi = 0;
            if (j < B.n) {
                c = B.v[j];
                d = B.vert(j + 1);
                if (c.y == d.y && c.x != d.x && c.y >= ya0 && c.y <= ya1) A.row(c.y - 1, lo, hi);
            }
            const int steps = __reduce_max_sync(0xffffffffu, hi - lo);
            for (int t = 0; t < steps; ++t) {
                bool hit = false;
                int i = 0;
                if (t < hi - lo) {
                    i = A.edge(lo + t);
                    const int2 a = A.v[i], b = A.vert(i + 1);
                    hit = (a.x != b.x || a.y != b.y) && edges_cross(a, b, c, d);
                }
                push_crossings(hit, i, j, s.cq[wid], nq, A, va.sgn, B, vb.sgn, org, sum, lane);
            }
        }
        if (lane < nq) sum.add(crossing_terms(A.v, A.n, va.sgn, B.v, B.n, vb.sgn, org, s.cq[wid][lane]));
        unsigned long long en = (unsigned long long)ends;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            en += __shfl_xor_sync(0xffffffffu, en, o);
        }
        sum.reduce();
        if (lane == 0) {
            BigSmem* first = cl.map_shared_rank(&s, 0);
            atomicAdd(&first->ends, en);
            atomicAdd(&first->q18, sum.q18);
            atomicAdd(&first->r56, sum.r56);
        }
        cl.sync();
        if (ctid == 0) {
            const double inter = ExactSum{s.q18, s.r56}.total((long long)s.ends);
            const double uni = va.area + vb.area - inter;
            out[e] = uni > 0 ? fmin(fmax(inter / uni, 0.0), 1.0) : 0.0;
        }
    }
}

struct JKey {
    double j;
    int32_t id;
};

__device__ __forceinline__ bool jkey_before(JKey a, JKey b)  // (J desc, id asc)
{
    return a.j > b.j || (a.j == b.j && (uint32_t)a.id < (uint32_t)b.id);
}

__global__ void topk_by_j_kernel(const int32_t* __restrict__ ids, const int32_t* __restrict__ nlist,
                                 const double* __restrict__ jv, int m, int cap, int k,
                                 int32_t* __restrict__ top_ids, double* __restrict__ top_j,
                                 const int64_t* __restrict__ d_n)
{
    extern __shared__ JKey s[];
    const int64_t q = blockIdx.x;
    if (d_n && q >= *d_n) return;  // past the live batch
    const int n = nlist[q];
    for (int i = threadIdx.x; i < cap; i += blockDim.x) {
        JKey x;
        if (i < n) {
            x.j = jv[q * m + i];
            x.id = ids[q * m + i];
        } else {
            x.j = -1.0;
            x.id = -1;  // as unsigned: largest id, sorts last
        }
        s[i] = x;
    }
    __syncthreads();
    for (int kk = 2; kk <= cap; kk <<= 1)
        for (int jj = kk >> 1; jj > 0; jj >>= 1) {
            for (int i = threadIdx.x; i < cap; i += blockDim.x) {
                int l = i ^ jj;
                if (l > i) {
                    JKey a = s[i], b = s[l];
                    bool up = (i & kk) == 0;
                    if (jkey_before(b, a) == up) {
                        s[i] = b;
                        s[l] = a;
                    }
                }
            }
            __syncthreads();
        }
    for (int i = threadIdx.x; i < k; i += blockDim.x) {
        bool ok = i < n;
        top_ids[q * k + i] = ok ? s[i].id : -1;
        top_j[q * k + i] = ok ? s[i].j : -1.0;
    }
}

}  // namespace

// pairs of one launch: the queue of large rings holds a launch's pairs
constexpr int64_t kRefineSlice = 1 << 20;

size_t pmh_refine_queue_bytes(int64_t n_pairs)
{
    return sizeof(int32_t) * (size_t)std::min(std::max<int64_t>(n_pairs, 1), kRefineSlice);
}

const void* pmh_refine_big_func() { return reinterpret_cast<const void*>(refine_big_kernel); }

// persistent grids (SM count x resident blocks) over the pairs, kRefineSlice at a time; with
// a queue, the pairs of large rings are left to refine_big_kernel
static int launch_refine(pmh_ctx ctx, const RefineQueries& qs, pmh_polys db, const int32_t* ids,
                         const int32_t* nlist, int m, const int32_t* qid_list, int64_t n_pairs, double* out,
                         unsigned long long* tickets, int32_t* big, const int64_t* d_n, cudaStream_t s)
{
    const size_t smem = sizeof(RefPair) * (kRefineWarps / 2);
    PMH_CUDA_TRY(cudaFuncSetAttribute(refine_pairs_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem));
    int per_sm = 0;
    PMH_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, refine_pairs_kernel,
                                                               kRefineWarps * 32, smem));
    for (int64_t e0 = 0; e0 < n_pairs; e0 += kRefineSlice) {
        const int64_t e1 = std::min(n_pairs, e0 + kRefineSlice);
        const int blocks = (int)std::min<int64_t>((e1 - e0 + 1) / 2,
                                                  (int64_t)ctx->sm_count * std::max(per_sm, 1));
        PMH_CUDA_TRY(cudaMemsetAsync(tickets, 0, 3 * sizeof(unsigned long long), s));
        refine_pairs_kernel<<<blocks, kRefineWarps * 32, smem, s>>>(
            qs.xy, qs.off, qs.area2, qs.box, db->xy, db->offsets, db->area2, db->bbox, ids, nlist, m, qid_list,
            e0, e1, out, tickets, big, d_n);
        PMH_LAUNCHED("refine_pairs_kernel");
        if (!big) continue;
        const int bblocks = kBigCluster * (int)std::min<int64_t>(e1 - e0, std::max(ctx->sm_count * kBigBlocks / kBigCluster, 1));
        refine_big_kernel<<<bblocks, kBigThreads, 0, s>>>(qs.xy, qs.off, qs.area2, qs.slabs, db->xy, db->offsets,
                                                          db->area2, db->d_slabs, ids, m, qid_list, e0, out,
                                                          tickets, big);
        PMH_LAUNCHED("refine_big_kernel");
    }
    return PMH_OK;
}

// first of the three context ticket slots of the refinement grids
constexpr int kRefineTicket = 40;

int pmh_launch_refine_topk(pmh_ctx ctx, const RefineQueries& qs, pmh_polys db, const int32_t* ids,
                           const int32_t* nlist, int64_t Q, const int64_t* d_n, int32_t m, int32_t k,
                           double* jv, unsigned long long* tickets, int32_t* big, int32_t* top_ids,
                           double* top_j, cudaStream_t s)
{
    if (Q <= 0) return PMH_OK;
    PMH_TRY(launch_refine(ctx, qs, db, ids, nlist, m, nullptr, Q * m, jv, tickets, big, d_n, s));
    int cap = 1;
    while (cap < m) cap <<= 1;
    const size_t smem = sizeof(JKey) * cap;
    topk_by_j_kernel<<<(unsigned)Q, 256, smem, s>>>(ids, nlist, jv, m, cap, k, top_ids, top_j, d_n);
    PMH_LAUNCHED("topk_by_j_kernel");
    return PMH_OK;
}

// scratch of a library call: `doubles` exact Jaccards, then the queue of large rings when
// either set has one
static int refine_scratch(pmh_ctx ctx, pmh_polys queries, pmh_polys db, int64_t doubles, int64_t n_pairs,
                          double** jv, int32_t** big)
{
    const bool large = std::max(queries->max_n, db->max_n) > kRefineBigVerts;
    void* buf = nullptr;
    PMH_TRY(pmh_scratch(ctx, SCR_REFINE, sizeof(double) * (size_t)doubles +
                                             (large ? pmh_refine_queue_bytes(n_pairs) : 0), &buf));
    *jv = static_cast<double*>(buf);
    *big = large ? reinterpret_cast<int32_t*>(*jv + doubles) : nullptr;
    return PMH_OK;
}

static RefineQueries refine_queries(pmh_polys q)
{
    return RefineQueries{q->xy, q->offsets, q->area2, q->bbox, q->d_slabs};
}

extern "C" int pmh_refine_topk(pmh_ctx ctx, pmh_polys queries, pmh_polys db, const int32_t* d_ids,
                               const int32_t* d_n, int64_t Q, int32_t m, int32_t k,
                               int32_t* d_top_ids, double* d_top_j, void* stream)
{
    PMH_TRY(pmh_check_device(ctx));
    if (!queries || !db || Q < 0 || Q > queries->n || m < 1 || m > 1024 || k < 1 || k > m ||
        (Q > 0 && (!d_ids || !d_n || !d_top_ids || !d_top_j)))
        return pmh_set_error(PMH_ERR_ARG, "bad arguments (1 <= k <= m <= 1024)");
    if (Q == 0) return PMH_OK;
    double* jv = nullptr;
    int32_t* big = nullptr;
    PMH_TRY(refine_scratch(ctx, queries, db, Q * m, Q * m, &jv, &big));
    return pmh_launch_refine_topk(ctx, refine_queries(queries), db, d_ids, d_n, Q, nullptr, m, k, jv,
                                  ctx->d_tickets + kRefineTicket, big, d_top_ids, d_top_j,
                                  (cudaStream_t)stream);
}

extern "C" int pmh_pair_jaccard(pmh_ctx ctx, pmh_polys queries, pmh_polys db, const int32_t* d_qid,
                                const int32_t* d_pid, int64_t n_pairs, double* d_j, void* stream)
{
    PMH_TRY(pmh_check_device(ctx));
    if (!queries || !db || n_pairs < 0 || (n_pairs > 0 && (!d_qid || !d_pid || !d_j)))
        return pmh_set_error(PMH_ERR_ARG, "bad arguments");
    if (n_pairs == 0) return PMH_OK;
    double* none = nullptr;
    int32_t* big = nullptr;
    PMH_TRY(refine_scratch(ctx, queries, db, 0, n_pairs, &none, &big));
    return launch_refine(ctx, refine_queries(queries), db, d_pid, nullptr, 1, d_qid, n_pairs, d_j,
                         ctx->d_tickets + kRefineTicket, big, nullptr, (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------
// Brute-force candidate set of the exact search (the paper's BF baseline,
// Sec. 5.2): every database polygon whose bounding box overlaps the query's
// with positive area -- the only ones with J > 0.  The database is cut into
// segments; a warp takes kBoxQueries queries over one segment, 64 boxes at a
// time, one read of a box serving all of its queries; ballots keep ids
// ascending.  The counting pass leaves every (query, segment)'s hits in seg;
// the filling pass starts behind the sum of the segments before.  (A warp per
// query over the whole set left a batch of 96 queries to 96 warps: 1.27 ms a
// pass over 100,000 boxes, bound by the latency of one load at a time;
// 22 us now.)
// ---------------------------------------------------------------------------
namespace {

constexpr int kBoxQueries = 4;
constexpr int kBoxWarps = 8;

template <bool kWrite>
__global__ void __launch_bounds__(kBoxWarps * 32)
bbox_join_kernel(const int4* __restrict__ qbox, int64_t Q, const int4* __restrict__ pbox, int64_t N, int segs,
                 int32_t* __restrict__ seg, int64_t* __restrict__ counts,
                 const int64_t* __restrict__ row_ptr, int32_t* __restrict__ cand)
{
    const int lane = threadIdx.x & 31;
    const int64_t groups = (Q + kBoxQueries - 1) / kBoxQueries;
    const int64_t nwarps = (int64_t)gridDim.x * kBoxWarps;
    for (int64_t w = (int64_t)blockIdx.x * kBoxWarps + (threadIdx.x >> 5); w < groups * segs; w += nwarps) {
        const int64_t g = w / segs;
        const int i = (int)(w - g * segs);
        const int64_t q0 = g * kBoxQueries;
        const int nq = (int)min((int64_t)kBoxQueries, Q - q0);
        int4 a[kBoxQueries];
        int64_t out[kBoxQueries];
        int cnt[kBoxQueries];
#pragma unroll
        for (int t = 0; t < kBoxQueries; ++t) {
            a[t] = t < nq ? qbox[q0 + t] : make_int4(0, 0, 0, 0);
            out[t] = cnt[t] = 0;
            if (kWrite && t < nq) {
                int64_t before = 0;
                for (int u = lane; u < i; u += 32) before += seg[(q0 + t) * segs + u];
                for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
                out[t] = row_ptr[q0 + t] + before;
            }
        }
        const int64_t b = N * i / segs, e = N * (i + 1) / segs;
        for (int64_t x0 = b; x0 < e; x0 += 64) {
            int4 box[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int64_t x = x0 + 32 * u + lane;
                // (an empty box at the far corner overlaps nothing)
                box[u] = x < e ? pbox[x] : make_int4(INT_MAX, INT_MAX, INT_MIN, INT_MIN);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int4 p = box[u];
#pragma unroll
                for (int t = 0; t < kBoxQueries; ++t) {
                    const bool hit = t < nq && a[t].x < p.z && p.x < a[t].z && a[t].y < p.w && p.y < a[t].w;
                    const unsigned m = __ballot_sync(0xffffffffu, hit);
                    if (kWrite && hit)
                        cand[out[t] + cnt[t] + __popc(m & pmh_lanemask_lt())] = (int32_t)(x0 + 32 * u + lane);
                    cnt[t] += __popc(m);
                }
            }
        }
        if (!kWrite && lane == 0) {
#pragma unroll
            for (int t = 0; t < kBoxQueries; ++t)
                if (t < nq) {
                    seg[(q0 + t) * segs + i] = cnt[t];
                    atomicAdd(reinterpret_cast<unsigned long long*>(&counts[q0 + t]), (unsigned long long)cnt[t]);
                }
        }
    }
}

}  // namespace

extern "C" int pmh_bbox_join(pmh_ctx ctx, pmh_polys queries, pmh_polys db, int64_t* d_row_ptr,
                             int32_t* d_cand, int64_t cand_capacity, int64_t* h_total, void* stream)
{
    PMH_TRY(pmh_check_device(ctx));
    if (!queries || !db || !d_row_ptr || !h_total || cand_capacity < 0)
        return pmh_set_error(PMH_ERR_ARG, "bad arguments");
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t Q = queries->n;
    *h_total = 0;
    if (Q == 0) {
        PMH_CUDA_TRY(cudaMemsetAsync(d_row_ptr, 0, sizeof(int64_t), s));
        return PMH_OK;
    }
    // segments of the database: enough (query group, segment) items for the device, at least
    // 64 boxes and at most 1,024 segments each
    const int64_t groups = (Q + kBoxQueries - 1) / kBoxQueries;
    const int64_t full = (int64_t)ctx->sm_count * 8, want = (full * kBoxWarps + groups - 1) / groups;
    const int segs = (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(want, 1024), db->n / 64));
    int64_t* counts = nullptr;
    PMH_TRY(pmh_scratch(ctx, SCR_QUERY, (sizeof(int64_t) + sizeof(int32_t) * segs) * (size_t)Q, (void**)&counts));
    int32_t* seg = reinterpret_cast<int32_t*>(counts + Q);
    const unsigned blocks = (unsigned)std::min<int64_t>((groups * segs + kBoxWarps - 1) / kBoxWarps, full);
    PMH_CUDA_TRY(cudaMemsetAsync(counts, 0, sizeof(int64_t) * (size_t)Q, s));
    bbox_join_kernel<false><<<blocks, kBoxWarps * 32, 0, s>>>(queries->bbox, Q, db->bbox, db->n, segs, seg,
                                                              counts, nullptr, nullptr);
    PMH_LAUNCHED("bbox_join_kernel<count>");
    PMH_TRY(pmh_exclusive_scan_i64(ctx, counts, d_row_ptr, Q, s));
    PMH_CUDA_TRY(cudaMemcpyAsync(ctx->h_pinned, d_row_ptr + Q, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    PMH_CUDA_TRY(cudaStreamSynchronize(s));
    const int64_t total = ctx->h_pinned[0];
    *h_total = total;
    if (total > cand_capacity)
        return pmh_set_error(PMH_ERR_CAPACITY, "%lld pairs > capacity %lld", (long long)total,
                             (long long)cand_capacity);
    if (total == 0) return PMH_OK;
    if (!d_cand) return pmh_set_error(PMH_ERR_ARG, "null candidate buffer");
    bbox_join_kernel<true><<<blocks, kBoxWarps * 32, 0, s>>>(queries->bbox, Q, db->bbox, db->n, segs, seg,
                                                             nullptr, d_row_ptr, d_cand);
    PMH_LAUNCHED("bbox_join_kernel<fill>");
    return PMH_OK;
}
