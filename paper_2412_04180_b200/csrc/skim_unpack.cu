// Consumers of the packed form (SKIM Section 4.2, last paragraph: rows of equal width are stored and
// processed together; Section 4 overview and Section 4.3: a dequantised weight is its codebook
// entry times the scaling vector, Wq = Quant(W * alpha^-1) * alpha):
//   skim_dequantize  packed codes + per-row codebooks (+ alpha) -> fp16 matrix in source-row order
//   skim_matvec      y = Wq x taken straight from the packed codes, never forming Wq
//
// The codebook of a warp's row sits in registers, as planes of its entries' low and high bytes: a byte permutation takes four codes at
// once out of eight entries, so that a lookup costs two permutations per four elements (four at width 4) and no memory access.  (A load
// from the warp's copy in shared memory, as before, is a wavefront of the L1 data path per 32 elements, and its address two more
// operations per element.)  A warp takes 256 columns of a row at a time, eight a lane; the per-column vector (alpha, or z = alpha x) sits
// in shared memory.  What a warp needs of its first row is on its way while that vector is staged.
// Both kernels are programmatic dependents of whatever runs before them.  us, call after call, with codebooks in shared memory / in registers / and as
// a dependent, on one packed matrix (in L2) and, in brackets, on ten in turn (165 MB, more than L2 holds):
//   mat-vec      4096 x 11008 at 3.0 bits 19.7 / 17.5 / 14.5 (18.9 / 16.8 / 14.3), 22016 x 8192 54 and now 43 either way.  Bound by the integer
//                pipe (16 lanes a clock and scheduler: about 3 operations per element there), then by its start and end
//   dequantiser  4096 x 11008 scaled 26.6 / 27.4 / 24.9 (25.9 / 26.9 / 24.9), unscaled 23.2 and now 21.4.  b/8 B in and 2 B out per element, 1.6
//                times as long as a plain fill of the output: issue is 59 % busy, and a warp has one row, eleven batches of codes one
//                after another, with every eighth warp idle
// Lanes that own 32 columns and walk rows, the codes brought by bulk copies: 24.7 us for the unscaled dequantiser where this took 23.7, and 22.6 for the
// mat-vec (too few warps for the chain of a row).  Requesting whole rows into L2 first: slower by 5 % at 22016 x 8192.
#include "skim_internal.cuh"
#include "skim_lane_words.h"

namespace {

struct UnpackArgs {
    const uint32_t *packed;
    const int32_t *row_order;
    const long long *group_info;    // [nb + 1] first packed row of every group, then [nb + 1] word offsets
    const uint16_t *lut;            // [rows][kmax] binary16
    const float *s;                 // [cols] or nullptr
    const uint16_t *x;              // [cols] binary16 (mat-vec only)
    int64_t rows;
    int cols;
    int nb, bmin, kmax;
    uint16_t *out;                  // dequantiser: [rows][ld]
    int64_t ld;
    int out_vec;                    // rows of `out` are 16-byte aligned
    float *y;                       // mat-vec: [rows]
};

// The groups' first packed rows and word offsets, in registers (uniform loads, all at once).
struct Groups {
    int start[SKIM_MAX_NBITS + 1];
    long long word[SKIM_MAX_NBITS];
    int placed;                     // packed rows (a width outside the bit set was skipped)
    __device__ __forceinline__ explicit Groups(const UnpackArgs &a)
    {
        placed = 0;
#pragma unroll
        for (int u = 0; u <= SKIM_MAX_NBITS; ++u) {
            start[u] = u <= a.nb ? (int)__ldg(a.group_info + u) : 0;
            if (u < SKIM_MAX_NBITS) word[u] = u < a.nb ? __ldg(a.group_info + a.nb + 1 + u) : 0;
            if (u == a.nb) placed = start[u];
        }
    }
};

// Eight codes of B bits (the low 8 B bits of x; above them anything) as the eight nibbles of a word.
template <int B>
__device__ __forceinline__ uint32_t nibbles(uint32_t x)
{
    if constexpr (B == 4) {
        return x;
    } else if constexpr (B == 3) {
        // halves of 12 bits, bytes of 6, nibbles of 3; what comes along above each is cleared at the end
        const uint32_t y = (x & 0x00000fffu) | ((x << 4) & 0xfffff000u);
        const uint32_t z = (y & 0x00ff00ffu) | ((y << 2) & 0xff00ff00u);
        return ((z & 0x0f0f0f0fu) | ((z << 1) & 0xf0f0f0f0u)) & 0x77777777u;
    } else if constexpr (B == 2) {
        const uint32_t y = __byte_perm(x, 0u, 0x4140);
        const uint32_t z = (y | (y << 4)) & 0x0f0f0f0fu;
        return (z | (z << 2)) & 0x33333333u;
    } else {
        const uint32_t y = (x | (x << 12)) & 0x000f000fu;
        const uint32_t z = (y | (y << 6)) & 0x03030303u;
        return (z | (z << 3)) & 0x11111111u;
    }
}

// A codebook in registers, as byte planes: lo[i], hi[i] hold the low and high bytes of entries 4 i .. 4 i + 3.
template <int B>
struct Book {
    static constexpr int N = B == 4 ? 4 : B == 3 ? 2 : 1;
    uint32_t lo[N], hi[N];
    // entries: binary16, 8-byte aligned
    __device__ __forceinline__ explicit Book(const uint16_t *entries)
    {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const uint2 e = reinterpret_cast<const uint2 *>(entries)[i];
            lo[i] = __byte_perm(e.x, e.y, 0x6420);
            hi[i] = __byte_perm(e.x, e.y, 0x7531);
        }
    }
    // The entries of eight codes, two a word.
    __device__ __forceinline__ void look_up(uint32_t n, uint32_t (&h)[4]) const
    {
        // a permutation takes four selectors of 4 bits, whose top bit must be clear
        const uint32_t s = B == 4 ? n & 0x77777777u : n;
        const uint32_t top = B == 4 ? (n >> 3) & 0x11111111u : 0u;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const uint32_t su = u ? s >> 16 : s;
            uint32_t l, g;
            if constexpr (B == 4) {
                const uint32_t upper = __byte_perm(0x0000ff00u, 0u, u ? top >> 16 : top);       // the bytes of codes 8 .. 15
                l = (__byte_perm(lo[0], lo[1], su) & ~upper) | (__byte_perm(lo[2], lo[3], su) & upper);
                g = (__byte_perm(hi[0], hi[1], su) & ~upper) | (__byte_perm(hi[2], hi[3], su) & upper);
            } else {
                l = __byte_perm(lo[0], lo[N - 1], su);
                g = __byte_perm(hi[0], hi[N - 1], su);
            }
            h[2 * u] = __byte_perm(l, g, 0x5140);
            h[2 * u + 1] = __byte_perm(l, g, 0x7362);
        }
    }
};

// Two binary32 operations in one instruction; the same results as two.
__device__ __forceinline__ unsigned long long pack2(float a, float b)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

constexpr int UT = 1024;            // threads per block, one block per SM
constexpr int UW = UT / 32;
constexpr int STEP = 256;           // columns a warp takes at a time

// The lane's codes of a row, from step t on: those of a step are 8 B bits at byte (32 t + lane) B, asked for with `ask` and put together with `get` when
// they are used, so that the load does not have to be waited for before.
template <int B>
struct LaneCodes {
    const unsigned char *at, *at2;  // for B = 3 the word that holds its first byte, and the next one if the bits reach into it
    SkimLaneWords3 words;           // B = 3
    __device__ __forceinline__ LaneCodes(const uint32_t *row, int lane, int t) : words(lane)
    {
        at = reinterpret_cast<const unsigned char *>(row) + t * (32 * B) + (B == 3 ? 4 * words.first : B * lane);
        at2 = at + (words.reaches_next(8) ? 4 : 0);
    }
    // of the t-th step from here, of which the row has `columns` columns from the lane's first one on (8: or more)
    __device__ __forceinline__ uint2 ask(int t, int columns = 8) const
    {
        const int o = t * (32 * B);
        if (B == 4) return make_uint2(__ldg(reinterpret_cast<const uint32_t *>(at + o)), 0u);
        if (B == 2) return make_uint2(__ldg(reinterpret_cast<const uint16_t *>(at + o)), 0u);
        if (B == 1) return make_uint2(__ldg(at + o), 0u);
        // (whole: read without a branch; else 0, the code of the columns past the row's end)
        const bool second = columns >= 8 || words.reaches_next(columns);
        return make_uint2(__ldg(reinterpret_cast<const uint32_t *>(at + o)), second ? __ldg(reinterpret_cast<const uint32_t *>(at2 + o)) : 0u);
    }
    __device__ __forceinline__ void advance(int t)
    {
        at += t * (32 * B);
        at2 += t * (32 * B);
    }
    __device__ __forceinline__ uint32_t get(const uint2 &v) const { return B == 3 ? __funnelshift_r(v.x, v.y, words.shift) : v.x; }
};

// How a lane's eight values leave: one aligned 16-byte store; or, for rows that are not 16-byte aligned, through the warp's stretch of
// shared memory, so that the stores are whole words next to one another; or one by one.
enum Mode { STORE_VEC, STORE_STAGED, STORE_SINGLE, MATVEC };

template <int MODE>
__device__ __forceinline__ void store8(uint16_t *dst, int j0, int cols, const uint32_t (&h)[4], uint32_t *stage)
{
    if (MODE == STORE_VEC && j0 + 8 <= cols) {
        *reinterpret_cast<uint4 *>(dst + j0) = make_uint4(h[0], h[1], h[2], h[3]);
        return;
    }
    if (MODE != STORE_STAGED) {
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (j0 + u < cols) dst[j0 + u] = (uint16_t)((u & 1) ? (h[u >> 1] >> 16) : (h[u >> 1] & 0xffffu));
        return;
    }
    const int lane = threadIdx.x & 31;
    const uint16_t *s16 = reinterpret_cast<const uint16_t *>(stage);
    const int base = j0 - lane * 8, n = min(STEP, cols - base);            // the warp's first element, and how many
    *reinterpret_cast<uint4 *>(stage + lane * 4) = make_uint4(h[0], h[1], h[2], h[3]);
    __syncwarp();
    const int odd = (int)((reinterpret_cast<uintptr_t>(dst + base) >> 1) & 1u);        // elements before the first whole word
    if (odd && lane == 0) dst[base] = s16[0];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int e = odd + 2 * (u * 32 + lane);
        if (e + 1 < n) *reinterpret_cast<uint32_t *>(dst + base + e) = (uint32_t)s16[e] | ((uint32_t)s16[e + 1] << 16);
        else if (e < n) dst[base + e] = s16[e];
    }
    __syncwarp();
}

// Where the vector's entry of column j sits: inside a block of 256 columns the first quads of all 32 lanes come first, then the second
// quads, so that a lane's eight are two 16-byte loads that are contiguous across the warp.
__device__ __forceinline__ int vec_slot(int j)
{
    const int in = j & (STEP - 1), lane = in >> 3, u = in & 7;
    return (j & ~(STEP - 1)) + (u >> 2) * 128 + lane * 4 + (u & 3);
}

// Steps [s0, s1) of one row; MATVEC: returns the lane's sum.
template <int B, int MODE>
__device__ __forceinline__ float unpack_row(const UnpackArgs &a, const uint32_t *words, uint16_t *dst, int s0, int s1, const float *vec, const uint16_t *entries,
                                            uint32_t *stage)
{
    constexpr int AHEAD = 4;                // steps whose codes are in flight
    const int lane = threadIdx.x & 31;
    const Book<B> book(entries);
    LaneCodes<B> codes(words, lane, s0);
    const float *v4 = vec + s0 * STEP + lane * 4;
    int j0 = s0 * STEP + lane * 8;
    unsigned long long acc[2] = {0ull, 0ull};
    auto step = [&](int u0, const uint2 &raw, bool whole) {
        uint32_t h[4];
        book.look_up(nibbles<B>(codes.get(raw)), h);
        if (MODE == MATVEC || a.s) {
            const ulonglong2 va = *reinterpret_cast<const ulonglong2 *>(v4 + u0 * STEP), vb = *reinterpret_cast<const ulonglong2 *>(v4 + u0 * STEP + 128);
            const unsigned long long v[4] = {va.x, va.y, vb.x, vb.y};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&h[u]));
                if constexpr (MODE == MATVEC) {
                    acc[u & 1] = fma2(pack2(f.x, f.y), v[u], acc[u & 1]);
                } else {
                    float p, q;
                    unpack2(mul2(pack2(f.x, f.y), v[u]), p, q);
                    const __half2 r = __floats2half2_rn(p, q);
                    h[u] = *reinterpret_cast<const uint32_t *>(&r);
                }
            }
        }
        if constexpr (MODE != MATVEC) {
            const int j = j0 + u0 * STEP;
            if (MODE == STORE_VEC && whole)
                *reinterpret_cast<uint4 *>(dst + j) = make_uint4(h[0], h[1], h[2], h[3]);
            else
                store8<MODE>(dst, j, a.cols, h, stage);
        }
    };
    // By AHEAD steps: two batches take turns, the next one requested as a whole before the current one is worked on (one step at a
    // time, a load shares its scoreboard with later ones and is waited for with them).  The last batch holds what is left, and the row's
    // ragged end: lanes past it have nothing (STORE_STAGED: they help with the stores).
    const int batches = max(min(s1, a.cols / STEP) - s0, 0) / AHEAD, left = s1 - s0 - batches * AHEAD;
    uint2 now[AHEAD], next[AHEAD];
    auto ask_left = [&](int j, uint2 (&to)[AHEAD]) {
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) to[u] = u < left && j + u * STEP < a.cols ? codes.ask(u, a.cols - j - u * STEP) : make_uint2(0u, 0u);
    };
    if (batches) {
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) now[u] = codes.ask(u);
    } else {
        ask_left(j0, now);
    }
    for (int b = 1; b <= batches; ++b) {
        codes.advance(AHEAD);
        if (b < batches) {
#pragma unroll
            for (int u = 0; u < AHEAD; ++u) next[u] = codes.ask(u);
        } else {
            ask_left(j0 + AHEAD * STEP, next);
        }
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) step(u, now[u], true);
        v4 += AHEAD * STEP;
        j0 += AHEAD * STEP;
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) now[u] = next[u];
    }
#pragma unroll
    for (int u = 0; u < AHEAD; ++u)
        if (u < left && (MODE == STORE_STAGED || j0 + u * STEP < a.cols)) step(u, now[u], j0 + u * STEP - lane * 8 + STEP <= a.cols);
    float p, q, r, v;
    unpack2(acc[0], p, q);
    unpack2(acc[1], r, v);
    return (p + q) + (r + v);
}

// Packed rows are dealt round-robin to the blocks, so that every SM gets the same number (within one); `parts` warps share a
// row, each with a stretch of its steps (the mat-vec then adds their sums in order).
template <int MODE>
__global__ void __launch_bounds__(UT) skim_unpack_kernel(UnpackArgs a, int steps, int parts)
{
    extern __shared__ __align__(16) float vec[];          // [steps][STEP] (scaled, or the mat-vec), then (STORE_STAGED) [UW][STEP / 2] words
    __shared__ __align__(16) uint16_t books[UW][16];
    __shared__ float sums[UW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool use_vec = MODE == MATVEC || a.s;
    uint32_t *stage = reinterpret_cast<uint32_t *>(vec + (use_vec ? steps * STEP : 0)) + (MODE == STORE_STAGED ? warp * (STEP / 2) : 0);
    skim_let_next_kernel_start();
    skim_wait_for_previous_kernel();
    const Groups g(a);
    const int part = warp % parts, hop = UW / parts * (int)gridDim.x;
    const int s0 = steps * part / parts, s1 = steps * (part + 1) / parts;
    int p = (int)blockIdx.x + warp / parts * (int)gridDim.x;
    int src = p < g.placed ? __ldg(a.row_order + p) : 0;
    if (!SKIM_IDX(src, a.rows, nullptr)) src = 0;
    uint16_t entry = p < g.placed ? __ldg(a.lut + (int64_t)src * a.kmax + min(lane, a.kmax - 1)) : (uint16_t)0;
    if (use_vec) {
        for (int j = tid * 4; j < steps * STEP; j += UT * 4) {
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                v[u] = 0.0f;
                if (j + u < a.cols) {
                    v[u] = a.s ? a.s[j + u] : 1.0f;
                    if (MODE == MATVEC) {
                        const float x = __half2float(__ushort_as_half(a.x[j + u]));
                        v[u] = a.s ? __fmul_rn(x, v[u]) : x;
                    }
                }
            }
            *reinterpret_cast<float4 *>(vec + vec_slot(j)) = make_float4(v[0], v[1], v[2], v[3]);
        }
        __syncthreads();
    }
    // every warp goes through the same number of rounds: warps that share a row meet at a barrier
    for (int first_p = (int)blockIdx.x; first_p < g.placed; first_p += hop, p += hop) {
        float acc = 0.0f;
        if (p < g.placed) {
            __syncwarp();
            if (lane < 16) books[warp][lane] = entry;
            __syncwarp();
            const uint16_t *book = books[warp];
            const int nsrc = p + hop < g.placed ? __ldg(a.row_order + p + hop) : 0;      // the next row's, one row early
            int u = 0, first = g.start[0];
            long long word = g.word[0];
#pragma unroll
            for (int v = 1; v < SKIM_MAX_NBITS; ++v)
                if (v < a.nb && p >= g.start[v]) { u = v; first = g.start[v]; word = g.word[v]; }
            const int width = a.bmin + u;
            const uint32_t *words = a.packed + word + (int64_t)(p - first) * skim_row_stride_words(a.cols, width);
            uint16_t *dst = a.out + (int64_t)src * a.ld;
            switch (width) {
            case 1: acc = unpack_row<1, MODE>(a, words, dst, s0, s1, vec, book, stage); break;
            case 2: acc = unpack_row<2, MODE>(a, words, dst, s0, s1, vec, book, stage); break;
            case 3: acc = unpack_row<3, MODE>(a, words, dst, s0, s1, vec, book, stage); break;
            default: acc = unpack_row<4, MODE>(a, words, dst, s0, s1, vec, book, stage); break;
            }
            if (MODE == MATVEC) {
#pragma unroll
                for (int off = 16; off; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
                if (parts == 1 && lane == 0) a.y[src] = acc;
            }
            if (MODE == MATVEC && parts > 1) {
                if (lane == 0) sums[warp] = acc;
            }
            if (MODE != MATVEC || parts == 1) {
                src = SKIM_IDX(nsrc, a.rows, nullptr) ? nsrc : 0;
                entry = __ldg(a.lut + (int64_t)src * a.kmax + min(lane, a.kmax - 1));
            }
        }
        if (MODE == MATVEC && parts > 1) {
            __syncthreads();
            if (p < g.placed) {
                if (part == 0 && lane == 0) {
                    for (int q = 1; q < parts; ++q) acc += sums[warp + q];
                    a.y[src] = acc;
                }
                src = p + hop < g.placed ? __ldg(a.row_order + p + hop) : 0;
                if (!SKIM_IDX(src, a.rows, nullptr)) src = 0;
                entry = __ldg(a.lut + (int64_t)src * a.kmax + min(lane, a.kmax - 1));
            }
            __syncthreads();
        }
    }
}

constexpr size_t UNPACK_STATIC_SMEM = UW * 17 * sizeof(float);      // (more than the 1152 bytes in use: the longest row taken stays 57 344 columns)

// with few rows several warps share one
int unpack_parts(const skim_ctx *ctx, int64_t rows, int steps)
{
    int parts = 1;
    while (parts < UW && parts * 2 <= steps && rows * parts * 2 <= (int64_t)ctx->sm_count * UW) parts *= 2;
    return parts;
}

int launch_unpack(skim_ctx *ctx, void (*kernel)(UnpackArgs, int, int), const UnpackArgs &a, int steps, size_t smem)
{
    // Set on every launch that needs it, to the same value: no state shared between contexts.  The calls on small matrices are bound
    // by the host, and this one is a twelfth of their time, so it is left out within the 48 KB that need no permission.
    if (smem + UNPACK_STATIC_SMEM > 48 * 1024)
        SKIM_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ctx->max_smem_optin - (int)UNPACK_STATIC_SMEM));
    const unsigned blocks = (unsigned)(a.rows < ctx->sm_count ? a.rows : ctx->sm_count);      // one block per SM
    return skim_launch_dependent(ctx, kernel, dim3(blocks), UT, smem, a, steps, unpack_parts(ctx, a.rows, steps));
}

}  // namespace

int skim_launch_dequantize(skim_ctx *ctx, const uint32_t *packed, const int32_t *row_order, const int64_t *group_info,
                           const uint16_t *lut, const float *s, int64_t rows, int64_t cols, const SkimBits &bs,
                           uint16_t *out, int64_t ld_out)
{
    if (rows == 0) return SKIM_OK;
    UnpackArgs a;
    a.packed = packed; a.row_order = row_order; a.group_info = (const long long *)group_info; a.lut = lut;
    a.s = s; a.x = nullptr; a.rows = rows; a.cols = (int)cols; a.nb = bs.n_bits; a.bmin = bs.b_min; a.kmax = 1 << bs.b_max;
    a.out = out; a.ld = ld_out; a.y = nullptr;
    a.out_vec = ((reinterpret_cast<uintptr_t>(out) & 15u) == 0 && (ld_out % 8) == 0) ? 1 : 0;
    const int steps = (int)((cols + STEP - 1) / STEP);
    const size_t vec = s ? (size_t)steps * STEP * sizeof(float) : 0, stage = (size_t)UW * STEP * 2;
    if (vec + UNPACK_STATIC_SMEM > (size_t)ctx->max_smem_optin) return SKIM_ERR_SHAPE;
    if (a.out_vec) return launch_unpack(ctx, skim_unpack_kernel<STORE_VEC>, a, steps, vec);
    // very long unaligned rows leave no room for the staging of the stores: single 16-bit stores then
    if (vec + stage + UNPACK_STATIC_SMEM <= (size_t)ctx->max_smem_optin) return launch_unpack(ctx, skim_unpack_kernel<STORE_STAGED>, a, steps, vec + stage);
    return launch_unpack(ctx, skim_unpack_kernel<STORE_SINGLE>, a, steps, vec);
}

int skim_launch_matvec(skim_ctx *ctx, const uint32_t *packed, const int32_t *row_order, const int64_t *group_info,
                       const uint16_t *lut, const float *s, const uint16_t *x, int64_t rows, int64_t cols,
                       const SkimBits &bs, float *y)
{
    if (rows == 0) return SKIM_OK;
    UnpackArgs a;
    a.packed = packed; a.row_order = row_order; a.group_info = (const long long *)group_info; a.lut = lut;
    a.s = s; a.x = x; a.rows = rows; a.cols = (int)cols; a.nb = bs.n_bits; a.bmin = bs.b_min; a.kmax = 1 << bs.b_max;
    a.out = nullptr; a.ld = 0; a.out_vec = 0; a.y = y;
    const int steps = (int)((cols + STEP - 1) / STEP);
    const size_t vec = (size_t)steps * STEP * sizeof(float);
    if (vec + UNPACK_STATIC_SMEM > (size_t)ctx->max_smem_optin) return SKIM_ERR_SHAPE;
    return launch_unpack(ctx, skim_unpack_kernel<MATVEC>, a, steps, vec);
}
