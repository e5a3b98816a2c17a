// Consumers of the packed form (SKIM Section 4.2, last paragraph: rows of equal width are stored and
// processed together; Section 4 overview and Section 4.3: a dequantised weight is its codebook
// entry times the scaling vector, Wq = Quant(W * alpha^-1) * alpha):
//   skim_dequantize  packed codes + per-row codebooks (+ alpha) -> fp16 matrix in source-row order
//   skim_matvec      y = Wq x taken straight from the packed codes, never forming Wq
//
// Codebook lookups go to the warp's copy of the row's codebook in shared memory, 16 consecutive words: no bank conflicts,
// one wavefront of the L1 data path per 32 elements (a shuffle takes that path for twice as long).
// A warp takes 256 columns of a row at a time; the per-column vector (alpha, or z = alpha x) sits in shared memory.  What a
// warp needs of its first row is on its way while that vector is staged.
//   dequantiser  bound by its writes: b/8 B in and 2 B out per element (4096 x 11008 24.4 us, a plain fill of the output 24.3)
//   mat-vec      bound by the L1 data path (2.7 wavefronts per 32 elements: a lookup each, the reads of z and the packed words; busy
//                13.2 of 17.3 us at 4096 x 11008), then by issue and, at the usual sizes, by its start and end
#include "skim_internal.cuh"

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

// The shared address of a codebook as the lookups take it.  The lookups are assembly that the compiler does not see as reads of the
// array: this call, before and after the array is written, keeps them on their side of the stores.
__device__ __forceinline__ uint32_t codebook_address(const float *book)
{
    uint32_t r;
    asm volatile("mov.u32 %0, %1;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(book)) : "memory");
    return r;
}

// Codebook entry of a code, the codebook at shared address `book` (64-byte aligned).  `code4` holds the code in bits 2 .. B + 1
// among others: one logic operation makes the address.
template <int B>
__device__ __forceinline__ float lookup(uint32_t book, uint32_t code4)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"((code4 & (((1u << B) - 1u) << 2)) | book));
    return v;
}

constexpr int UT = 1024;            // threads per block, one block per SM
constexpr int UW = UT / 32;
constexpr int STEP = 256;           // columns a warp takes at a time

// The eight codes of the lane's elements (8 B bits at byte `at` B of the row), as loaded: at width 3 they may lie in two words, which
// are only put together when they are used, so that the load does not have to be waited for before.
template <int B>
struct LaneCodes {
    uint32_t lo, hi;
    __device__ __forceinline__ void load(const uint8_t *row, int at)
    {
        hi = 0u;
        if (B == 4) lo = __ldg(reinterpret_cast<const uint32_t *>(row) + at);
        else if (B == 2) lo = __ldg(reinterpret_cast<const uint16_t *>(row) + at);
        else if (B == 1) lo = __ldg(row + at);
        else {
            // the row is padded to 16 bytes, and the second word is only asked for where the bits reach into it
            const uint32_t *w = reinterpret_cast<const uint32_t *>(row) + (3 * at >> 2);
            lo = __ldg(w);
            if ((3 * at & 3) > 1) hi = __ldg(w + 1);
        }
    }
    __device__ __forceinline__ uint32_t get(int at) const { return B == 3 ? __funnelshift_r(lo, hi, 8 * (3 * at & 3)) : lo; }
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
__device__ __forceinline__ float unpack_row(const UnpackArgs &a, const uint8_t *words, uint16_t *dst, int s0, int s1, const float *vec, uint32_t book,
                                            uint32_t *stage)
{
    constexpr int AHEAD = 4;                // steps whose codes are in flight
    const int lane = threadIdx.x & 31, last = (a.cols - 1) / 8;      // the row's last group of eight
    // two batches take turns: the next one is requested as a whole before the current one is worked on (one step at a time, a
    // load shares its scoreboard with later ones and is waited for with them)
    LaneCodes<B> codes[AHEAD], next[AHEAD];
    float acc = 0.0f;
#pragma unroll
    for (int u = 0; u < AHEAD; ++u) codes[u].load(words, min((s0 + u) * 32 + lane, last));
    for (int t0 = s0; t0 < s1; t0 += AHEAD) {
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) next[u].load(words, min((t0 + AHEAD + u) * 32 + lane, last));
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            const int t = t0 + u;
            if (t < s1) {
                const uint32_t c = codes[u].get(min(t * 32 + lane, last));
                float r[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) r[e] = lookup<B>(book, e * B >= 2 ? c >> (e * B - 2) : c << (2 - e * B));
                if (MODE == MATVEC || a.s) {
                    const float4 va = *reinterpret_cast<const float4 *>(vec + t * STEP + lane * 4), vb = *reinterpret_cast<const float4 *>(vec + t * STEP + 128 + lane * 4);
                    const float v[8] = {va.x, va.y, va.z, va.w, vb.x, vb.y, vb.z, vb.w};
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        if (MODE == MATVEC) acc = fmaf(r[e], v[e], acc);
                        else r[e] = __fmul_rn(r[e], v[e]);
                    }
                }
                if constexpr (MODE == MATVEC) continue;
                else {
                uint32_t h[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const __half2 v = __floats2half2_rn(r[2 * e], r[2 * e + 1]);
                    h[e] = *reinterpret_cast<const uint32_t *>(&v);
                }
                const int j0 = t * STEP + lane * 8;
                if (MODE == STORE_STAGED || j0 < a.cols) store8<MODE>(dst, j0, a.cols, h, stage);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) codes[u] = next[u];
    }
    return acc;
}

// Packed rows are dealt round-robin to the blocks, so that every SM gets the same number (within one); `parts` warps share a
// row, each with a stretch of its steps (the mat-vec then adds their sums in order).
template <int MODE>
__global__ void __launch_bounds__(UT) skim_unpack_kernel(UnpackArgs a, int steps, int parts)
{
    extern __shared__ __align__(16) float vec[];          // [steps][STEP] (scaled, or the mat-vec), then (STORE_STAGED) [UW][STEP / 2] words
    __shared__ __align__(128) float books[UW][16];
    __shared__ float sums[UW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool use_vec = MODE == MATVEC || a.s;
    uint32_t *stage = reinterpret_cast<uint32_t *>(vec + (use_vec ? steps * STEP : 0)) + (MODE == STORE_STAGED ? warp * (STEP / 2) : 0);
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
            if (lane < 16) books[warp][lane] = __half2float(__ushort_as_half(entry));
            __syncwarp();
            const uint32_t book = codebook_address(books[warp]);
            const int nsrc = p + hop < g.placed ? __ldg(a.row_order + p + hop) : 0;      // the next row's, one row early
            int u = 0, first = g.start[0];
            long long word = g.word[0];
#pragma unroll
            for (int v = 1; v < SKIM_MAX_NBITS; ++v)
                if (v < a.nb && p >= g.start[v]) { u = v; first = g.start[v]; word = g.word[v]; }
            const int width = a.bmin + u;
            const uint8_t *words = reinterpret_cast<const uint8_t *>(a.packed + word + (int64_t)(p - first) * skim_row_stride_words(a.cols, width));
            uint16_t *dst = a.out + (int64_t)src * a.ld;
            switch (width) {
            case 1: acc = unpack_row<1, MODE>(a, words, dst, s0, s1, vec, book, stage); break;
            case 2: acc = unpack_row<2, MODE>(a, words, dst, s0, s1, vec, book, stage); break;
            case 3: acc = unpack_row<3, MODE>(a, words, dst, s0, s1, vec, book, stage); break;
            default: acc = unpack_row<4, MODE>(a, words, dst, s0, s1, vec, book, stage); break;
            }
            codebook_address(books[warp]);
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

constexpr size_t UNPACK_STATIC_SMEM = UW * 17 * sizeof(float);

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
    kernel<<<blocks, UT, smem, ctx->stream>>>(a, steps, unpack_parts(ctx, a.rows, steps));
    SKIM_CUDA_OK(cudaGetLastError());
    ctx->launches += 1;
    return SKIM_OK;
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
