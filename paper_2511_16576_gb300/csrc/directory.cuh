// directory.cuh -- the bucket index's directory over its sorted composites (lsh.cu): sizes,
// filling and lookup, in host and device code alike.
//
// A composite is (band j in the top band_bits bits, the key's top bits below).  Valid ones lie
// in [0, cmax) with cmax = bands << (32 - band_bits); invalid entries (all ones) sort last and
// are never looked up.  dir[s] = first sorted entry whose composite >> shift is >= s, for s
// in [0, top] with top = ceil(cmax / 2^shift), and dir[top + 1] = the number of entries: the
// end of a bucket is looked up as the lower bound of its composite + 1, which for the last
// valid composite is cmax itself, whose slot may be top.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define PMH_HD __host__ __device__ __forceinline__
#else
#define PMH_HD inline
#endif

// bits of the band index, below 2^bits - 1 for every band (no valid composite is all ones)
PMH_HD int pmh_band_bits(uint32_t bands)
{
    int bits = 1;
    while ((1u << bits) - 1 < bands) ++bits;
    return bits;
}

PMH_HD int64_t pmh_dir_cmax(uint32_t bands, int band_bits) { return (int64_t)bands << (32 - band_bits); }

// about eight sorted entries per slot over [0, cmax), at most 2^24 slots
PMH_HD int pmh_dir_shift(int64_t entries, int64_t cmax)
{
    int sh = 31;
    while (sh > 0 && (cmax >> (sh - 1)) <= (int64_t)1 << 24 && (cmax >> (sh - 1)) * 8 <= entries) --sh;
    return sh;
}

PMH_HD int64_t pmh_dir_top(int64_t cmax, int sh) { return (cmax + ((int64_t)1 << sh) - 1) >> sh; }
PMH_HD int64_t pmh_dir_len(int64_t cmax, int sh) { return pmh_dir_top(cmax, sh) + 2; }

// The slots [from, to] that entry e of m writes with its own number: those after its
// predecessor's, up to its own (e = m: up to the last), so every slot is written once.
PMH_HD void pmh_dir_slots(const uint32_t* comp, int64_t m, int64_t e, int sh, int64_t cmax, int64_t* from,
                          int64_t* to)
{
    const int64_t before = e > 0 ? ((int64_t)comp[e - 1] < cmax ? (int64_t)comp[e - 1] : cmax) : 0;
    const int64_t own = e < m ? ((int64_t)comp[e] < cmax ? (int64_t)comp[e] : cmax) : 0;
    *from = e > 0 ? (before >> sh) + 1 : 0;
    *to = e < m ? own >> sh : pmh_dir_top(cmax, sh) + 1;
}

// first sorted entry whose composite is >= c, for c in [0, cmax]
template <class Dir>
PMH_HD int64_t pmh_comp_lower_bound(const uint32_t* comp, const Dir& dir, int sh, uint32_t c)
{
    const uint32_t s = c >> sh;
    int64_t lo = dir[s], hi = dir[s + 1];
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (comp[mid] < c) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}
