// Where the unpacking kernels (skim_unpack.cu) read a lane's eight codes at width 3.  Plain C++ without CUDA, so that the addresses can be
// checked for every row length on the host too.
#pragma once

#ifdef __CUDACC__
#define SKIM_HD __host__ __device__ __forceinline__
#else
#define SKIM_HD inline
#endif

// Lane L of a step of 32 lanes owns bits 24 L .. 24 L + 23 of the step's 24 words: they begin in word `first`, at bit `shift`.
struct SkimLaneWords3 {
    int first, shift;
    SKIM_HD explicit SkimLaneWords3(int lane) : first(3 * lane >> 2), shift(8 * (3 * lane & 3)) {}
    // Whether the next word holds bits of the lane's first `columns` codes.  It is read only then: at the end of a row whose last codes fill a
    // word of the 16-byte padded row's last four, the next word is another row's, or behind the buffer.
    SKIM_HD bool reaches_next(int columns) const { return shift + 3 * (columns < 8 ? columns : 8) > 32; }
};
