// The range arithmetic of the allocation's selection (skim_allocate.cu): unsigned 64-bit keys in a closed range, split
// into at most 2048 equal parts.  Plain C++ without CUDA, so that it can be run over all kinds of keys on the host too.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define SKIM_HD __host__ __device__ __forceinline__
#else
#define SKIM_HD inline
#endif

struct SkimKeyRange {
    static constexpr int PART_BITS = 11;
    uint64_t lo, hi;      // the live keys lie in [lo, hi]

    // parts are 2^shift keys wide: the fewest bits that leave at most 2^PART_BITS parts
    SKIM_HD int shift() const
    {
        const uint64_t span = hi - lo;
#ifdef __CUDA_ARCH__
        const int bits = 64 - __clzll((long long)span);
#else
        const int bits = span ? 64 - __builtin_clzll(span) : 0;
#endif
        return bits > PART_BITS ? bits - PART_BITS : 0;
    }
    // (a key below the range wraps round to a large number)
    SKIM_HD bool holds(uint64_t key) const { return key - lo <= hi - lo; }
    SKIM_HD unsigned part_of(uint64_t key, int sh) const { return (unsigned)((key - lo) >> sh); }
    // Part p, cut off at the range's end.  Its last key is formed as an offset from lo, whose low `sh` bits are free: the sum
    // lo + (p << sh) + 2^sh - 1 can pass 2^64 in the last part (infinite gains beside a negative one span nearly all keys).
    SKIM_HD SkimKeyRange part(unsigned p, int sh) const
    {
        const uint64_t first = (uint64_t)p << sh, last = first | (((uint64_t)1 << sh) - 1), span = hi - lo;
        SkimKeyRange r;
        r.lo = lo + first;
        r.hi = lo + (last < span ? last : span);
        return r;
    }
};
