// Labels of eight consecutive elements of a row by the midpoint rule (number of boundaries strictly below the value),
// shared by the packer and the residual kernel.
#pragma once

#include "skim_internal.cuh"

namespace skiml {

// The boundaries of one row's width block in shared memory: tf[j] is the midpoint of centroids j and j + 1 rounded down to
// binary32 (x > midpoint exactly when x > tf), +inf past the last; th[j] the same rounded down to binary16, twice.
struct RowBounds {
    float tf[16];
    __half2 th[16];
};

// Thread j < 16 fills entry j; c: the row's k = 2^b centroids, cj its own (or the last).
__device__ __forceinline__ void fill_bounds(RowBounds &rb, int j, const float *c, float cj, int k)
{
    float t = __int_as_float(0x7f800000);
    if (j < k - 1) {
        t = __double2float_rd(0.5 * ((double)cj + (double)c[j + 1]));
        if (t == 0.0f) t = 0.0f;
    }
    rb.tf[j] = t;
    rb.th[j] = __half2half2(__float2half_rd(t));
}

// No scale installed: a binary16 weight is above a boundary exactly when it is above the boundary rounded down to binary16,
// so two weights are compared per instruction and the label is the running sum of the 0/1 results.  Label u in bits
// [u B, (u + 1) B).
template <int B>
__device__ __forceinline__ uint32_t labels8_half(const uint4 &raw, const __half2 *th)
{
    const __half2 *p = reinterpret_cast<const __half2 *>(&raw);
    const __half2 magic = __floats2half2_rn(1024.0f, 1024.0f);   // 1024 + n has n in its low mantissa bits
    uint32_t v = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        __half2 cnt = magic;
#pragma unroll
        for (int j = 0; j < (1 << B) - 1; ++j) cnt = __hadd2(cnt, __hgt2(p[u], th[j]));
        const uint32_t bits = *reinterpret_cast<const uint32_t *>(&cnt);
        v |= (bits & 0xfu) << ((2 * u) * B);
        v |= ((bits >> 16) & 0xfu) << ((2 * u + 1) * B);
    }
    return v;
}

// A scale vector installed: B probes of the binary32 boundaries in shared memory for each of the eight values.
template <int B>
__device__ __forceinline__ uint32_t labels8_float(const float *x, const float *tf)
{
    uint32_t v = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        int code = 0;
#pragma unroll
        for (int step = 1 << (B - 1); step >= 1; step >>= 1) code += (x[u] > tf[code + step - 1]) ? step : 0;
        v |= (uint32_t)code << (u * B);
    }
    return v;
}

// Elements e0 .. e0 + 7 of a row of binary16 weights, zeros past cols.  The row may start at any even address: two aligned
// 16-byte blocks are then shifted together (both inside the row), single loads only where the row ends.
__device__ __forceinline__ uint4 load8_weights(const uint16_t *row, int e0, int cols)
{
    const uint32_t mis = (uint32_t)(reinterpret_cast<uintptr_t>(row) & 15u);             // the same for the whole row
    if (mis == 0) {
        if (e0 + 8 <= cols) return __ldg(reinterpret_cast<const uint4 *>(row + e0));
    } else if (e0 >= 8 && e0 + 16 <= cols) {
        const uint4 *p = reinterpret_cast<const uint4 *>(reinterpret_cast<uintptr_t>(row + e0) & ~(uintptr_t)15);
        const uint4 a = __ldg(p), b = __ldg(p + 1);
        const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        const uint32_t q = mis >> 2, s = (mis & 3u) * 8u;                                 // whole words, then bits
        uint32_t t[5];
#pragma unroll
        for (int u = 0; u < 5; ++u) t[u] = q == 0 ? w[u] : q == 1 ? w[u + 1] : q == 2 ? w[u + 2] : w[u + 3 < 8 ? u + 3 : 7];
        return make_uint4(__funnelshift_r(t[0], t[1], s), __funnelshift_r(t[1], t[2], s), __funnelshift_r(t[2], t[3], s), __funnelshift_r(t[3], t[4], s));
    }
    uint32_t r[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int u = 0; u < 8; ++u)
        if (e0 + u < cols) r[u >> 1] |= (uint32_t)row[e0 + u] << (16 * (u & 1));
    return make_uint4(r[0], r[1], r[2], r[3]);
}

// The eight weights as binary32, times r (1 / alpha) where given.
__device__ __forceinline__ void values8(const uint4 &raw, const float *r, int e0, int cols, float *x)
{
    const __half2 *h2 = reinterpret_cast<const __half2 *>(&raw);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const float2 f = __half22float2(h2[u]);
        x[2 * u] = f.x;
        x[2 * u + 1] = f.y;
    }
    if (r) {
        if (e0 + 8 <= cols) {
            const float4 r0 = *reinterpret_cast<const float4 *>(r + e0), r1 = *reinterpret_cast<const float4 *>(r + e0 + 4);
            x[0] = __fmul_rn(x[0], r0.x); x[1] = __fmul_rn(x[1], r0.y);
            x[2] = __fmul_rn(x[2], r0.z); x[3] = __fmul_rn(x[3], r0.w);
            x[4] = __fmul_rn(x[4], r1.x); x[5] = __fmul_rn(x[5], r1.y);
            x[6] = __fmul_rn(x[6], r1.z); x[7] = __fmul_rn(x[7], r1.w);
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (e0 + u < cols) x[u] = __fmul_rn(x[u], r[e0 + u]);
        }
    }
}

}  // namespace skiml
