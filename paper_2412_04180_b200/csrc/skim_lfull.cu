// L-full error of every row (SKIM Section 3.4: the layer-wise objective written per row,
// err_i = (w_i - wq_i) X X^T (w_i - wq_i)^T; Section 4.2 and Algorithm 3 fill the error table with it; the
// paper's scaling vector enters through wq = replace(c, l) * alpha, Section 4.3).
//
//   skim_residual_kernel      D = binary16((float(w) - c[label] * alpha) * 2^e): one block per row, labels by the
//                             same midpoint rule as the packer.  Streaming: 2 B in, 2 B out per element.
//   skim_lfull_gemm_kernel    Y = D H (H = X X^T, symmetric, binary16) on the tensor cores and, fused into the
//                             epilogue, the row-wise dot  sum_n Y_in D_in  of every output tile, so Y never
//                             leaves the SM.  This is the one dense contraction of the method.  Where only the errors are
//                             asked for it runs over the upper half of H with weight 2 (half the products; the kernel's
//                             spare warps check that H is symmetric, and the full contraction follows if not):
//                             bound by the tensor pipe, 4096 x 11008 x 11008 0.374 ms per width against 0.709 ms in full.
//   skim_lfull_reduce_kernel  adds the per-tile partial sums of a row in a fixed order, divides 4^e out.
//
// GEMM kernel: persistent, one CTA per SM, CTAs in pairs (cluster of two, tcgen05 cta_group::2), tile 256 x 256 x 64
// per pair, tcgen05.mma (kind::f16, binary32 accumulators in tensor memory, two accumulator stages of 256 columns),
// operands brought in by TMA (cp.async.bulk.tensor, 128-byte swizzle) through a 6-stage shared-memory ring.  A CTA
// fetches its 128 rows of D and half of the tile's rows of H (32 KB per K block of 64; a tile of its own of 128 x 256
// took 48 KB for the same MMA time, more than the L2 delivers to an SM meanwhile).  Warp 0 issues the TMA loads, warp 1
// allocates tensor memory and, in the first CTA, issues the MMAs of both, eight warps read the accumulators back
// (tcgen05.ld) and do the dot product with the matching D tile.  No TMA multicast: every CTA fetches its own operands.
// Every wait on an mbarrier is bounded: after WAIT_LIMIT_CYCLES the waiting role raises the block's abort flag,
// sets SKIM_STATUS_TIMEOUT, and all roles leave their loops; tensor memory is freed on every path.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <vector>

#include "skim_internal.cuh"
#include "skim_labels.cuh"

namespace {

// ---------------------------------------------------------------- residual

constexpr int RES_T = 256;

struct ResidualArgs {
    const uint16_t *W;
    const float *rscale;     // 1 / alpha (installed scale), or nullptr
    const float *s;          // alpha itself, or nullptr
    const float *centroids;
    const uint8_t *row_bits; // nullptr: every row at `width`
    int width;
    int64_t ld, ldd;
    int cols;
    int nb, bmin, sumk;
    int exp2;
    int vec;                 // rows of D (and of the scale vector) allow 128-bit accesses
    uint16_t *D;
    unsigned long long *status;
};

// Eight elements per thread and step, the next step's weights in flight.  The label's centroid is one conflict-free lookup in
// shared memory; the labels themselves come from packed compares (unscaled), so that a narrow width costs little.  Plain stores:
// what fits stays in L2 for the contraction.
template <int B>
__device__ __forceinline__ void residual_row(const ResidualArgs &a, const uint16_t *Wr, uint16_t *Dr, const skiml::RowBounds &rb, const float *cs, uint4 raw)
{
    __half2 th[(1 << B) - 1];
#pragma unroll
    for (int j = 0; j < (1 << B) - 1; ++j) th[j] = rb.th[j];
    const float scale = __int_as_float((127 + a.exp2) << 23);       // 2^exp2, exact
    for (int e0 = threadIdx.x * 8; e0 < a.cols; e0 += RES_T * 8) {
        uint4 next = make_uint4(0u, 0u, 0u, 0u);
        if (e0 + RES_T * 8 < a.cols) next = skiml::load8_weights(Wr, e0 + RES_T * 8, a.cols);
        float w[8];
        skiml::values8(raw, nullptr, e0, a.cols, w);
        uint32_t code;
        if (a.rscale) {
            float x[8];
            skiml::values8(raw, a.rscale, e0, a.cols, x);
            code = skiml::labels8_float<B>(x, rb.tf);
        } else {
            code = skiml::labels8_half<B>(raw, th);
        }
        float q[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) q[u] = cs[(code >> (u * B)) & ((1u << B) - 1u)];
        if (a.s) {
            if (a.vec) {
                const float4 s0 = *reinterpret_cast<const float4 *>(a.s + e0), s1 = *reinterpret_cast<const float4 *>(a.s + e0 + 4);
                const float sv[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
#pragma unroll
                for (int u = 0; u < 8; ++u) q[u] = __fmul_rn(q[u], sv[u]);
            } else {
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (e0 + u < a.cols) q[u] = __fmul_rn(q[u], a.s[e0 + u]);
            }
        }
        uint32_t out[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const __half2 h = __floats2half2_rn(__fmul_rn(__fsub_rn(w[2 * u], q[2 * u]), scale), __fmul_rn(__fsub_rn(w[2 * u + 1], q[2 * u + 1]), scale));
            out[u] = *reinterpret_cast<const uint32_t *>(&h);
        }
        if (a.vec) {
            *reinterpret_cast<uint4 *>(Dr + e0) = make_uint4(out[0], out[1], out[2], out[3]);
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (e0 + u < a.cols) Dr[e0 + u] = (uint16_t)((u & 1) ? (out[u >> 1] >> 16) : (out[u >> 1] & 0xffffu));
        }
        raw = next;
    }
}

__global__ void __launch_bounds__(RES_T) skim_residual_kernel(ResidualArgs a)
{
    __shared__ skiml::RowBounds rb;
    __shared__ float cs[16];
    const int tid = threadIdx.x;
    const int64_t row = blockIdx.x;
    skim_wait_for_previous_kernel();
    skim_let_next_kernel_start();
    const uint16_t *Wr = a.W + row * a.ld;
    const uint4 raw = skiml::load8_weights(Wr, tid * 8, a.cols);
    const int b = a.row_bits ? (int)a.row_bits[row] : a.width;
    const int bi = b - a.bmin;
    if (bi < 0 || bi >= a.nb) {
        if (tid == 0) atomicOr(a.status, (unsigned long long)SKIM_STATUS_BAD_BITS);
        return;
    }
    const int k = 1 << b;
    const int off = (1 << a.bmin) * ((1 << bi) - 1);
    const float *c = a.centroids + row * a.sumk + off;
    if (tid < 16) {
        const float cj = c[min(tid, k - 1)];
        cs[tid] = cj;
        skiml::fill_bounds(rb, tid, c, cj, k);
    }
    __syncthreads();
    uint16_t *Dr = a.D + row * a.ldd;
    switch (b) {
    case 1: residual_row<1>(a, Wr, Dr, rb, cs, raw); break;
    case 2: residual_row<2>(a, Wr, Dr, rb, cs, raw); break;
    case 3: residual_row<3>(a, Wr, Dr, rb, cs, raw); break;
    default: residual_row<4>(a, Wr, Dr, rb, cs, raw); break;
    }
}

// ---------------------------------------------------------------- GEMM with fused row-wise dot

constexpr int BM = 256, BN = 256, BK = 64;      // a tile belongs to a pair of CTAs: each has half of its rows
constexpr int CM = BM / 2;                      // rows of D (and of the accumulator) in a CTA
constexpr int CB = 64;                          // rows of H in a TMA box; a CTA holds BN / 2 = two boxes
constexpr int STAGES = 6;                       // ring of the half contraction; the full one gives a stage up for EpilogueSmem
constexpr int UMMA_K = 16;
constexpr int A_BYTES = CM * BK * 2, BOX_BYTES = CB * BK * 2, STAGE_BYTES = A_BYTES + 2 * BOX_BYTES;     // per CTA
constexpr int EPI_WARPS = 8;                    // two for every quarter of the accumulator's rows, each with half of the columns
constexpr int GEMM_THREADS = (2 + EPI_WARPS) * 32;
constexpr int LEAVE_POLL = 8;                   // the producer of the half contraction looks at the leave flag every so many K blocks
constexpr int CHECK_WARPS = 4;                  // further warps of the half contraction: they compare H with its transpose
constexpr int SPLIT_MAX = 8;                    // ranges of K a tile of the last round is cut into, at most
constexpr int HALF_MIN_ROWS = 768, HALF_MIN_NT = 4;
constexpr double HALF_MIN_SAVING = 14.0;         // K blocks of a pair (6 us) that the half contraction must save
constexpr double EPILOGUE_KB = 10.0;             // K blocks' worth of MMA time of an epilogue (256 columns read back and multiplied)
constexpr size_t HALF_FLAG_BYTES = 4096;         // symmetry flags of up to 1024 blocks
constexpr int TMEM_COLS = 512;                  // two accumulator stages of BN binary32 columns
constexpr long long WAIT_LIMIT_CYCLES = 400000000ll;   // about 0.2 s; a whole launch takes milliseconds
constexpr int KC = 16;                          // clusters of a row at most

// What the epilogue warps of a CTA exchange.
struct EpilogueSmem {
    double slot[2][KC][CM];      // per half of the columns and row: sums of y alpha by cluster (full contraction with Y only)
    double alpha[BN];
};
__host__ __device__ constexpr int ring_stages(bool half) { return half ? STAGES : STAGES - 1; }
__host__ __device__ constexpr size_t gemm_smem(bool half)
{
    return (size_t)ring_stages(half) * STAGE_BYTES + 1024 /* alignment slack */ + 256 /* barriers */ + CM * sizeof(float) + (half ? 0 : sizeof(EpilogueSmem));
}

struct GemmSync {
    uint64_t full[STAGES];
    uint64_t empty[STAGES];
    uint64_t tmem_full[2];
    uint64_t tmem_empty[2];
    uint64_t drained;            // half contraction: the MMAs issued are done (both CTAs)
    uint32_t tmem_base;
    int abort;                   // a wait ran out
    int asym;                    // half contraction: this CTA's warps have found (or been told) that H is not symmetric
    int leave;                   // half contraction: both CTAs stop where they are
    int issued[2];               // half contraction: K blocks that the CTAs' producers have issued
};
static_assert(sizeof(GemmSync) <= 256, "the barriers' part of gemm_smem");

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// Address of `p` (this CTA's shared memory) in the pair's CTA of rank `rank`.
__device__ __forceinline__ uint32_t cluster_addr(const void *p, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(smem_u32(bar)), "r"(parity)
                 : "memory");
    return ok != 0;
}
// Bounded wait.  False when the block is aborting (this wait ran out, or another role's did) or, with LEAVES, leaving.
template <bool LEAVES>
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, GemmSync &sync)
{
    volatile int *abort_flag = &sync.abort, *leave_flag = &sync.leave;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (*abort_flag || (LEAVES && *leave_flag)) return false;
        if (clock64() - t0 > WAIT_LIMIT_CYCLES) {
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}
__device__ __forceinline__ void store_cluster(uint32_t addr, int v)
{
    asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// A flag in global memory that other blocks of the launch may set.
__device__ __forceinline__ unsigned flag_load(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void flag_set(unsigned *p) { asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(1u) : "memory"); }

// Into this CTA's shared memory; the bytes are counted by the mbarrier at `bar` (an address in either CTA of the pair).
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint32_t bar, int x, int y)
{
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
                     smem_u32(dst)),
                 "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y)
                 : "memory");
}

// Shared-memory operand descriptor: K-major tile whose rows are 64 binary16 = 128 bytes, 128-byte swizzle,
// 8-row groups 1024 bytes apart (the layout TMA writes with CU_TENSOR_MAP_SWIZZLE_128B); tiles are 1024-byte
// aligned, and a step of UMMA_K elements along K inside the swizzle row is a plain 32-byte address offset.
__device__ __forceinline__ uint64_t umma_desc(uint32_t smem_addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3ffffu) >> 4);          // start address
    d |= (uint64_t)1 << 16;                                // leading byte offset (unused for this layout)
    d |= (uint64_t)(1024 >> 4) << 32;                      // stride byte offset: 8 rows x 128 bytes
    d |= (uint64_t)1 << 46;                                // descriptor version of this architecture
    d |= (uint64_t)2 << 61;                                // 128-byte swizzle
    return d;
}

// Instruction descriptor of kind::f16: D binary32, A and B binary16, both K-major, M = 256 (a pair of CTAs), N columns.
__host__ __device__ constexpr uint32_t umma_idesc(int n) { return (1u << 4) | (0u << 7) | (0u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24); }

// One lane of the pair's first CTA issues for both: each contributes its rows of A and its half of the rows of B from
// its own shared memory (same offsets) and accumulates its rows of D in its own tensor memory.
__device__ __forceinline__ void umma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
                 "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
                 : "memory");
}
// D = A B + D / 2
__device__ __forceinline__ void umma_f16_halve(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.b32 p, 0, 0;\n\ttcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p, 1;\n\t}" ::"r"(tmem_d),
                 "l"(adesc), "l"(bdesc), "r"(idesc)
                 : "memory");
}
// Arrives on the mbarrier at this offset in both CTAs once the MMAs issued so far are done.
__device__ __forceinline__ void umma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(smem_u32(bar)),
                 "h"((uint16_t)3)
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 32 consecutive binary32 columns of this thread's tensor-memory lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t *v)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Whole 32-byte sectors in one access: a lane of the epilogue has a row of its own, so that narrower ones take the L1 data path once per
// lane each (and a store of half a sector the L2 twice).
__device__ __forceinline__ void ld_sector(const void *p, uint4 &a, uint4 &b)
{
    asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
                 : "l"(p));
}
__device__ __forceinline__ void st_sector(void *p, const uint32_t *v)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]),
                 "r"(v[6]), "r"(v[7])
                 : "memory");
}

struct GemmArgs {
    const uint16_t *D;       // [rows][ldd] binary16 (also operand A, through its tensor map)
    int64_t ldd;
    int rows, cols;
    int mt, nt;              // tiles along rows and along columns
    int full_tiles, split;   // tiles [full_tiles, mt * nt) are cut into `split` parts (see unit_of)
    float *partial;          // [mt * BM][split][nt]
    float *Y;                // optional [rows][ldy]: the product D H itself (the scaling-vector update needs it)
    int64_t ldy;
    SkimLfullClusters cl;    // with Y, optional: sums of Y alpha by cluster
    int *asym;               // [asym_n] per block of the half contraction: H is not symmetric in the part it compared, or the block left
    int asym_n;
    int sectors;             // rows of D (and labels) start at whole sectors, and cols is a multiple of 32
    unsigned *leave;         // half contraction: some block has found H not symmetric (zero between calls)
    int piece_kb;            // half contraction: a tile's list of K blocks is cut into pieces of about this length
    unsigned long long *status;
};

// Work units.  Tiles are taken round-robin by the persistent pairs of CTAs; the tiles of the last, partly filled round
// would leave most pairs idle for a whole tile time, so each of them is cut into `split` parts that run side by side:
// ranges of K (the fused row-wise dot is linear in the accumulator, so a range simply leaves one more partial dot per
// row), or, where the product Y itself is asked for, the two halves of its columns.
struct GemmUnit {
    int tile, slice, kb0, kb1;
    int n_off, n;            // columns of the tile
};
__device__ __forceinline__ GemmUnit unit_of(const GemmArgs &a, int u, int nkb)
{
    GemmUnit w;
    w.tile = u; w.slice = 0; w.kb0 = 0; w.kb1 = nkb; w.n_off = 0; w.n = BN;
    if (u >= a.full_tiles) {
        const int r = u - a.full_tiles;
        w.tile = a.full_tiles + r / a.split;
        w.slice = r % a.split;
        if (a.Y) {
            w.n = BN / a.split;
            w.n_off = w.slice * w.n;
        } else {
            w.kb0 = (int)((long long)nkb * w.slice / a.split);
            w.kb1 = (int)((long long)nkb * (w.slice + 1) / a.split);
        }
    }
    return w;
}

// The quadratic form of a symmetric H needs half of its products:  d H d^T = sum_n d_n (H_nn d_n + 2 sum_{k>n} H_nk d_k).
// In tiles: column tile nb takes the K blocks of its own diagonal block with weight 1 and those beyond it (k >= n0 + BN)
// with weight 2, so its K list is simply n0/BK .. nkb-1.  The diagonal part comes first and is halved by the first MMA
// of the rest (the tensor core's own scaling of the accumulator input, exact); the epilogue doubles the dot.  (The
// upper half, not the lower: a large residual then meets as many later roundings of the accumulator as in the full
// contraction.)  Lists shrink from nkb blocks to one: tiles are taken in descending length, every other round of blocks
// in reverse order, so that the blocks end together; a list may be cut into pieces (their dots add up).  Row tiles vary
// fastest, so the blocks of a round share the panels of H.
struct HalfList {
    int nb, base, pieces;    // cursor: units base .. base + mt * pieces - 1 belong to column tile nb
};
constexpr int HALF_DIAG = BN / BK;                  // K blocks of a diagonal block (the last one may have fewer)
__host__ __device__ __forceinline__ int half_len(int nb, int nkb) { return nkb - nb * HALF_DIAG; }
__host__ __device__ __forceinline__ int half_pieces(int nb, int nkb, int piece_kb)
{
    const int p = (half_len(nb, nkb) + piece_kb - 1) / piece_kb;
    return p < SPLIT_MAX ? p : SPLIT_MAX;
}
// The GemmUnit of unit u (kb0, kb1 are list positions); units are asked for in ascending order.
__device__ __forceinline__ GemmUnit half_unit(const GemmArgs &a, HalfList &h, int u, int nkb)
{
    while (u >= h.base + a.mt * h.pieces) {
        h.base += a.mt * h.pieces;
        ++h.nb;
        h.pieces = half_pieces(h.nb, nkb, a.piece_kb);
    }
    const int r = u - h.base, len = half_len(h.nb, nkb);
    GemmUnit w;
    w.slice = r / a.mt;
    w.tile = h.nb * a.mt + r % a.mt;
    w.kb0 = len * w.slice / h.pieces;
    w.kb1 = len * (w.slice + 1) / h.pieces;
    w.n_off = 0;
    w.n = BN;
    return w;
}

// Unit of this pair in round t, or -1: round-robin (HALF: every other round reversed).
template <bool HALF>
__device__ __forceinline__ int unit_index(int t, int nunits)
{
    const int pairs = (int)gridDim.x / 2, pair = (int)blockIdx.x / 2;
    const int u = t * pairs + ((HALF && (t & 1)) ? pairs - 1 - pair : pair);
    return u < nunits ? u : -1;
}

// Compares H with its transpose, one warp per pair of blocks H[32 I .. +32][64 J .. +64] and H[64 J ..][32 I ..] at or
// above the diagonal.  A lane compares an 8 x 8 sub-block against its mirror image in registers; whole sectors on either side.
// The ragged end (fewer than 8 rows or columns cannot occur: cols is a multiple of 8).  True, and *leave set, at the first
// difference; true as well as soon as some other warp of the launch has set it.
__device__ __forceinline__ bool compare_transpose(const uint16_t *H, int64_t ldh, int cols, int first, int step, unsigned *leave)
{
    const int lane = threadIdx.x & 31;
    const int ni = (cols + 31) / 32, nj = (cols + 63) / 64;
    for (long long t = first; t < (long long)ni * nj; t += step) {
        const int I = (int)(t % ni), J = (int)(t / ni);
        if (64 * J + 64 <= 32 * I) continue;                  // below the diagonal: the mirror pair is compared
        const unsigned left = flag_load(leave);
        uint32_t diff = 0u;
        const int r0 = 32 * I + (lane >> 3) * 8, c0 = 64 * J + (lane & 7) * 8;
        if (r0 < cols && c0 < cols) {
            uint4 x[8], y[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = __ldg(reinterpret_cast<const uint4 *>(H + (int64_t)(r0 + u) * ldh + c0));
#pragma unroll
            for (int u = 0; u < 8; ++u) y[u] = __ldg(reinterpret_cast<const uint4 *>(H + (int64_t)(c0 + u) * ldh + r0));
#pragma unroll
            for (int r = 0; r < 8; r += 2) {
                const uint32_t a0[4] = {x[r].x, x[r].y, x[r].z, x[r].w}, a1[4] = {x[r + 1].x, x[r + 1].y, x[r + 1].z, x[r + 1].w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint4 b0 = y[2 * q], b1 = y[2 * q + 1];
                    const uint32_t v0 = r == 0 ? b0.x : r == 2 ? b0.y : r == 4 ? b0.z : b0.w;
                    const uint32_t v1 = r == 0 ? b1.x : r == 2 ? b1.y : r == 4 ? b1.z : b1.w;
                    diff |= __byte_perm(a0[q], a1[q], 0x5410) ^ v0;
                    diff |= __byte_perm(a0[q], a1[q], 0x7632) ^ v1;
                }
            }
        }
        if (__any_sync(0xffffffffu, (diff | left) != 0u)) {
            if (lane == 0) flag_set(leave);
            return true;
        }
    }
    return false;
}

// Adds y_j alpha_j of 32 consecutive columns to the row's sums by cluster (slot k of this thread at slot[k * CM]).  The
// slots of four elements are read together and the additions run in element order in registers, an element whose
// cluster matches an earlier one of the four continuing from that one's result, so that the round trips through shared
// memory do not follow one another.
__device__ __forceinline__ void add_by_cluster(double *slot, const uint32_t *y, const uint2 *labels, const double *alpha)
{
#pragma unroll
    for (int u0 = 0; u0 < 32; u0 += 4) {
        const uint32_t l4 = (u0 & 4) ? labels[u0 / 8].y : labels[u0 / 8].x;
        const double2 a0 = *reinterpret_cast<const double2 *>(alpha + u0), a1 = *reinterpret_cast<const double2 *>(alpha + u0 + 2);
        const double al[4] = {a0.x, a0.y, a1.x, a1.y};
        int l[4];
        double v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            l[u] = (int)((l4 >> (8 * u)) & (KC - 1));
            v[u] = slot[l[u] * CM];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            double base = v[u];
#pragma unroll
            for (int t = 0; t < u; ++t)
                if (l[t] == l[u]) base = v[t];
            v[u] = fma((double)__uint_as_float(y[u0 + u]), al[u], base);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) slot[l[u] * CM] = v[u];      // where clusters repeat the last store holds the full sum
    }
}

__device__ __forceinline__ bool epilogue_barrier_or(bool v)
{
    uint32_t r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(r)
                 : "r"((uint32_t)v), "n"(EPI_WARPS * 32)
                 : "memory");
    return r != 0;
}
__device__ __forceinline__ void epilogue_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory"); }

// HALF: the half contraction for a symmetric H, launched first; a.asym then says whether H was.  At the first difference that
// the checking warps find all pairs stop where they are (within a few K blocks), so that an H that is symmetric up to rounding
// only costs little more than the full contraction.  !HALF: the full contraction; with a.asym given it is the fallback of a
// half launch and returns at once unless H was not symmetric.
template <bool HALF>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GEMM_THREADS + (HALF ? CHECK_WARPS * 32 : 0), 1)
skim_lfull_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, GemmArgs a, const uint16_t *H, int64_t ldh)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char *tiles = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    constexpr int NST = ring_stages(HALF);
    GemmSync &sy = *reinterpret_cast<GemmSync *>(tiles + (size_t)NST * STAGE_BYTES);
    float *dot_s = reinterpret_cast<float *>(tiles + (size_t)NST * STAGE_BYTES + 256);                           // [CM]
    EpilogueSmem &ep = *reinterpret_cast<EpilogueSmem *>(tiles + (size_t)NST * STAGE_BYTES + 256 + CM * sizeof(float));   // not for HALF
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nkb = (a.cols + BK - 1) / BK;
    const int ntiles = a.mt * a.nt;
    int nunits = a.full_tiles + (ntiles - a.full_tiles) * a.split;
    HalfList half = {0, 0, HALF ? half_pieces(0, nkb, a.piece_kb) : 1};
    // Behind the half form the full one lets its reduction start as it ends: usually it has nothing to do and ends at once, and where H is not symmetric,
    // reduction blocks that wait beside it cost more than the launch (a table, us, let in at once and now: 4096 x 4096 symmetric 366 and 358, not
    // symmetric 633 and 614, 4096 x 2048 153 and 148, 289 and 276; with ordinary launches 410, 596, 185 and 313).
    if (!a.Y && (HALF || !a.asym)) skim_let_next_kernel_start();
    if (!HALF && a.asym) skim_wait_for_previous_kernel();
    if (HALF) {
        nunits = 0;
        for (int nb = 0; nb < a.nt; ++nb) nunits += a.mt * half_pieces(nb, nkb, a.piece_kb);
    } else if (a.asym) {
        int any = 0;
        for (int i = threadIdx.x; i < a.asym_n; i += GEMM_THREADS) any |= a.asym[i];
        if (blockIdx.x == 0 && threadIdx.x == 0) *a.leave = 0u;
        if (!__syncthreads_or(any)) return;
    }

    const uint32_t rank = cluster_rank();
    if (threadIdx.x == 0) {
        // full and tmem_empty are used in the first CTA only; the other two in both
        for (int s = 0; s < NST; ++s) { mbar_init(&sy.full[s], 1); mbar_init(&sy.empty[s], 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(&sy.tmem_full[s], 1); mbar_init(&sy.tmem_empty[s], 2 * EPI_WARPS); }
        mbar_init(&sy.drained, 1);
        sy.abort = 0;
        sy.asym = 0;
        sy.leave = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sy.tmem_base)), "r"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    if (HALF || !a.asym) skim_wait_for_previous_kernel();      // nothing is read or written before it
    const uint32_t tmem_base = sy.tmem_base;

    // one K block of operands: this CTA's half of either
    auto load_block = [&](int stage, int k, int m0, int b0, int boxes) {
        unsigned char *sa = tiles + (size_t)stage * STAGE_BYTES;
        if (rank == 0) mbar_expect_tx(&sy.full[stage], 2 * (A_BYTES + boxes * BOX_BYTES));
        const uint32_t bar = cluster_addr(&sy.full[stage], 0);
        tma_load_2d(sa, &map_a, bar, k, m0);
        for (int b = 0; b < boxes; ++b) tma_load_2d(sa + A_BYTES + b * BOX_BYTES, &map_b, bar, k, b0 + b * CB);
    };
    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (one lane)
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            int issued = 0;
            unsigned left = 0u;                               // the leave flag as it was LEAVE_POLL blocks ago: its load is never waited for
            for (int t = 0; t * ((int)gridDim.x / 2) < nunits && ok; ++t) {
                const int u = unit_index<HALF>(t, nunits);
                if (u < 0) continue;
                const GemmUnit w = HALF ? half_unit(a, half, u, nkb) : unit_of(a, u, nkb);
                const int m0 = (w.tile % a.mt) * BM + (int)rank * CM, n0 = (w.tile / a.mt) * BN;
                const int boxes = w.n / (2 * CB), b0 = n0 + w.n_off + (int)rank * (w.n / 2);
                for (int l = w.kb0; l < w.kb1; ++l) {
                    const int kb = HALF ? n0 / BK + l : l;
                    if (HALF && issued % LEAVE_POLL == 0) {
                        if (left) {
                            *(volatile int *)&sy.leave = 1;
                            store_cluster(cluster_addr(&sy.leave, rank ^ 1u), 1);
                            ok = false;
                            break;
                        }
                        left = flag_load(a.leave);
                    }
                    if (!(ok = mbar_wait<HALF>(&sy.empty[stage], phase ^ 1u, sy))) break;
                    load_block(stage, kb * BK, m0, b0, boxes);
                    ++issued;
                    if (++stage == NST) { stage = 0; phase ^= 1u; }
                }
            }
            if (HALF)
                for (uint32_t r = 0; r < 2; ++r) store_cluster(cluster_addr(&sy.issued[rank], r), issued);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (one lane of the first CTA)
        if (lane == 0 && rank == 0) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            int it = 0;
            for (int t = 0; t * ((int)gridDim.x / 2) < nunits && ok; ++t) {
                const int u = unit_index<HALF>(t, nunits);
                if (u < 0) continue;
                const GemmUnit w = HALF ? half_unit(a, half, u, nkb) : unit_of(a, u, nkb);
                const int as = it & 1;
                if (!(ok = mbar_wait<HALF>(&sy.tmem_empty[as], (((uint32_t)it >> 1) & 1u) ^ 1u, sy))) break;
                tc_fence_after();
                const uint32_t tmem_d = tmem_base + (uint32_t)(as * BN), idesc = umma_idesc(w.n);
                for (int kb = w.kb0; kb < w.kb1; ++kb) {          // HALF: list positions
                    if (!(ok = mbar_wait<HALF>(&sy.full[stage], phase, sy))) break;
                    tc_fence_after();
                    const uint32_t sa = smem_u32(tiles + (size_t)stage * STAGE_BYTES), sb = sa + A_BYTES;
#pragma unroll
                    for (int k = 0; k < BK / UMMA_K; ++k)
                        if (HALF && k == 0 && kb == HALF_DIAG && kb > w.kb0) umma_f16_halve(tmem_d, umma_desc(sa), umma_desc(sb), idesc);
                        else umma_f16(tmem_d, umma_desc(sa + k * UMMA_K * 2), umma_desc(sb + k * UMMA_K * 2), idesc, (kb > w.kb0 || k) ? 1u : 0u);
                    umma_commit(&sy.empty[stage]);           // the stage is free, in both CTAs, once these MMAs have read it
                    if (++stage == NST) { stage = 0; phase ^= 1u; }
                }
                if (ok) umma_commit(&sy.tmem_full[as]);      // the accumulator is complete once all MMAs are
                ++it;
            }
            if (HALF && !ok) umma_commit(&sy.drained);       // leaving
        }
    } else if (HALF && warp >= GEMM_THREADS / 32) {
        // ------------------------------------------------------------ H against its transpose, under the contraction
        if (compare_transpose(H, ldh, a.cols, (int)blockIdx.x * CHECK_WARPS + warp - GEMM_THREADS / 32, (int)gridDim.x * CHECK_WARPS, a.leave))
            sy.asym = 1;
    } else {
        // ------------------------------------------------------------ epilogue: one row per thread, half of the tile's columns
        const int q = warp & 3;                               // the tensor-memory lane quarter this warp may read
        const int ch = (warp - 2) >> 2, r = q * 32 + lane;    // half of the columns, row of the CTA
        const bool by_cluster = !HALF && a.cl.labels != nullptr;
        double *slot = &ep.slot[ch][0][r];
        bool ok = true;
        int it = 0;
        for (int t = 0; t * ((int)gridDim.x / 2) < nunits; ++t) {
            const int u = unit_index<HALF>(t, nunits);
            if (u < 0) continue;
            const GemmUnit w = HALF ? half_unit(a, half, u, nkb) : unit_of(a, u, nkb);
            const int as = it & 1;
            const int mb = w.tile % a.mt, nb = w.tile / a.mt;
            const int row = mb * BM + (int)rank * CM + r;
            const int n0 = nb * BN + w.n_off, c0 = ch * (w.n / 2);
            const int64_t lrow = min(row, a.rows - 1);
            const uint16_t *drow = a.D + lrow * a.ldd;
            if (by_cluster) {
                const int j = threadIdx.x - 64;
                if (j < w.n) ep.alpha[j] = n0 + j < a.cols ? a.cl.alpha[n0 + j] : 0.0;
#pragma unroll
                for (int k = 0; k < KC; ++k) slot[k * CM] = 0.0;
            }
            // the operands of the dot (and the labels) do not depend on the accumulator: the next 32 columns' are in flight
            uint4 dv[4], dn[4];
            uint2 lv[4], ln[4];
            auto fetch = [&](int c, uint4 (&d)[4], uint2 (&l)[4]) {
                if (a.sectors) {
                    const int col = n0 + c;
                    const bool in = c < c0 + w.n / 2 && col < a.cols;                 // cols is a multiple of 32
#pragma unroll
                    for (int v = 0; v < 4; v += 2) {
                        d[v] = d[v + 1] = make_uint4(0u, 0u, 0u, 0u);
                        if (in) ld_sector(drow + col + v * 8, d[v], d[v + 1]);
                    }
                    if (by_cluster) {
                        uint4 x = make_uint4(0u, 0u, 0u, 0u), y = x;
                        if (in) ld_sector(a.cl.labels + lrow * a.cols + col, x, y);
                        l[0] = make_uint2(x.x, x.y); l[1] = make_uint2(x.z, x.w); l[2] = make_uint2(y.x, y.y); l[3] = make_uint2(y.z, y.w);
                    }
                    return;
                }
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const int col = n0 + c + v * 8;
                    const bool in = c < c0 + w.n / 2 && col < a.cols;             // cols is a multiple of 8
                    d[v] = in ? __ldg(reinterpret_cast<const uint4 *>(drow + col)) : make_uint4(0u, 0u, 0u, 0u);
                    if (by_cluster) l[v] = in ? __ldg(reinterpret_cast<const uint2 *>(a.cl.labels + lrow * a.cols + col)) : make_uint2(0u, 0u);
                }
            };
            fetch(c0, dv, lv);
            epilogue_barrier();                               // alpha is in place
            ok = mbar_wait<HALF>(&sy.tmem_full[as], ((uint32_t)it >> 1) & 1u, sy);
            ok = __all_sync(0xffffffffu, ok);
            float acc = 0.0f;
            if (ok) {
                tc_fence_after();
#pragma unroll 1
                for (int c = c0; c < c0 + w.n / 2; c += 32) {
                    const int col = n0 + c;
                    fetch(c + 32, dn, ln);
                    uint32_t v[32];
                    tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(as * BN + c), v);
                    if (!HALF && a.Y && row < a.rows) {
                        float *yrow = a.Y + (int64_t)row * a.ldy + col;
#pragma unroll
                        for (int g = 0; g < 4; ++g)
                            if (col + g * 8 + 8 <= a.cols) st_sector(yrow + g * 8, v + g * 8);
                    }
                    // columns past the matrix have a zero accumulator and a zero alpha
                    if (by_cluster) add_by_cluster(slot, v, lv, ep.alpha + c);
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        const uint32_t w4[4] = {dv[g].x, dv[g].y, dv[g].z, dv[g].w};
#pragma unroll
                        for (int h = 0; h < 4; ++h) {
                            const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&w4[h]));
                            acc = fmaf(__uint_as_float(v[g * 8 + 2 * h]), f.x, acc);
                            acc = fmaf(__uint_as_float(v[g * 8 + 2 * h + 1]), f.y, acc);
                        }
                    }
#pragma unroll
                    for (int g = 0; g < 4; ++g) { dv[g] = dn[g]; lv[g] = ln[g]; }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(cluster_addr(&sy.tmem_empty[as], 0));
            }
            if (ch) dot_s[r] = acc;
            // the other half's dots and sums are in place; a warp whose wait ran out takes all of them out of the loop
            if (epilogue_barrier_or(!ok)) break;
            if (ch == 0 && row < a.rows) {
                acc += dot_s[r];
                // a piece that reaches past its diagonal blocks holds half the dot (the diagonal blocks' part was halved)
                if (HALF && w.kb1 > HALF_DIAG) acc *= 2.0f;
                a.partial[((int64_t)row * (HALF ? SPLIT_MAX : a.split) + w.slice) * a.nt + nb] = acc;
            }
            if (by_cluster && row < a.rows) {
                // this thread's half of the row's clusters
                double2 *rp = reinterpret_cast<double2 *>(a.cl.rpart + (((int64_t)row * a.nt + nb) * 2 + w.slice) * KC) + ch * (KC / 4);
#pragma unroll
                for (int k = 0; k < KC / 2; k += 2) {
                    const int kk = ch * (KC / 2) + k;
                    rp[k / 2] = make_double2(ep.slot[0][kk][r] + ep.slot[1][kk][r], ep.slot[0][kk + 1][r] + ep.slot[1][kk + 1][r]);
                }
            }
            epilogue_barrier();                               // before the slots, alpha and dots are written again
            ++it;
        }
    }
    // ---------------------------------------------------------------- teardown (every path comes here)
    tc_fence_before();
    __syncthreads();
    if (HALF) {
        // A pair that leaves has copies and MMAs in flight, and one of its producers may be ahead of the other, whose bytes
        // the pair's mbarriers then still expect.  Both issue as many blocks as the one ahead has (of anything; their stages
        // are free for both: one commit frees a stage in both CTAs), and wait until all of it has landed and the MMAs are done.
        cluster_sync();                // the counts and the leave flag are in place
        if (threadIdx.x == 0) {
            a.asym[blockIdx.x] = sy.asym | sy.leave;
            // (a producer that has issued its last block never raises the flag, so a pair that leaves has not finished)
            bool ok = sy.leave && !sy.abort;
            const int most = max(sy.issued[0], sy.issued[1]);
            for (int b = sy.issued[rank]; b < most && ok; ++b) {
                ok = mbar_wait<false>(&sy.empty[b % NST], (((uint32_t)(b / NST)) & 1u) ^ 1u, sy);
                if (ok) load_block(b % NST, 0, 0, 0, BN / (2 * CB));
            }
            if (rank == 0)
                for (int b = max(0, most - NST); b < most && ok; ++b) ok = mbar_wait<false>(&sy.full[b % NST], ((uint32_t)(b / NST)) & 1u, sy);
            if (ok) mbar_wait<false>(&sy.drained, 0u, sy);
        }
        __syncthreads();
    }
    if (sy.abort) {
        // a wait ran out: give the bulk copies that may still be in flight time to land before the block's
        // shared memory is released (about a millisecond), and report
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
        if (threadIdx.x == 0) atomicOr(a.status, (unsigned long long)SKIM_STATUS_TIMEOUT);
    }
    cluster_sync();                    // the other CTA may still read this one's shared memory, or arrive on its mbarriers
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS));
    }
}

constexpr int RED_WARPS = 8;

// Adds a row's partial dots in a fixed order, one warp per row: a lane takes every 32nd column tile, then a tree.  After a
// half contraction whose H was symmetric a tile has half_pieces() dots; after a full one slice 0 of every tile was
// written, and the further slices of the tiles that were cut along K.
__global__ void __launch_bounds__(RED_WARPS * 32)
skim_lfull_reduce_kernel(GemmArgs a, int exp2, float *__restrict__ err, int64_t err_stride, double *__restrict__ err64)
{
    skim_wait_for_previous_kernel();
    if (!a.Y) skim_let_next_kernel_start();
    bool half = false;
    if (a.asym) {
        int any = 0;
        for (int i = threadIdx.x; i < a.asym_n; i += RED_WARPS * 32) any |= a.asym[i];
        half = !__syncthreads_or(any);
    }
    const int i = blockIdx.x * RED_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= a.rows) return;
    const int mb = i / BM, nkb = (a.cols + BK - 1) / BK;
    double s = 0.0;
    for (int t = lane; t < a.nt; t += 32) {
        const int split = half ? SPLIT_MAX : a.split;
        const int pieces = half ? half_pieces(t, nkb, a.piece_kb) : t * a.mt + mb >= a.full_tiles ? a.split : 1;
        for (int sl = 0; sl < pieces; ++sl) s += (double)a.partial[((int64_t)i * split + sl) * a.nt + t];
    }
    if (a.cl.labels) {
        // R_k = sum_{j in k} Y_ij alpha_j over the column tiles, q_k = 2 R_k / (2^exp2 G_k) into the row's table
        const int k = lane & (KC - 1);
        double r = 0.0;
        for (int t = lane / KC; t < a.nt; t += 32 / KC) {
            const double *p = a.cl.rpart + ((int64_t)i * a.nt + t) * 2 * KC + k;
            r += p[0];
            if (a.split == 2 && t * a.mt + mb >= a.full_tiles) r += p[KC];
        }
        r += __shfl_down_sync(0xffffffffu, r, KC);
        if (lane < KC) {
            const double gk = a.cl.tconst[(int64_t)i * KC + lane].x;
            a.cl.tq[(int64_t)i * KC + lane].y = gk > 0.0 ? ldexp(2.0 * r, -exp2) / gk : 0.0;
        }
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) {
        if (err) err[(int64_t)i * err_stride] = (float)ldexp(s, -2 * exp2);
        if (err64) err64[i] = ldexp(s, -2 * exp2);
    }
}

// Length of the busiest pair of CTAs in a half contraction, in K blocks, if lists are cut into pieces of about piece_kb: a
// piece also costs its epilogue, which hides under the next piece's MMAs unless that one is shorter.
double half_makespan(int mt, int nt, int nkb, int piece_kb, int pairs)
{
    std::vector<double> load(pairs, 0.0);
    int u = 0;
    for (int nb = 0; nb < nt; ++nb) {
        const int p = half_pieces(nb, nkb, piece_kb);
        const double len = (double)half_len(nb, nkb) / p;
        for (int r = 0; r < p * mt; ++r, ++u) {
            const int t = u / pairs, b = u % pairs;
            load[(t & 1) ? pairs - 1 - b : b] += len > EPILOGUE_KB ? len : EPILOGUE_KB;
        }
    }
    double most = 0.0;
    for (double v : load) most = v > most ? v : most;
    return most + EPILOGUE_KB;
}

int encode_map(CUtensorMap *map, const uint16_t *base, int64_t rows, int64_t cols, int64_t ld, int box_rows)
{
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess || !fn)
        return SKIM_ERR_CUDA;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn)(
        map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<uint16_t *>(base), dims, strides, box, estr,
        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? SKIM_OK : SKIM_ERR_CUDA;
}

}  // namespace

int skim_launch_residual(skim_ctx *ctx, const uint16_t *W, int64_t rows, int64_t cols, int64_t ld, const float *centroids,
                         const uint8_t *row_bits, int width, const SkimBits &bs, const float *s, int exp2, uint16_t *D,
                         int64_t ldd)
{
    if (rows == 0) return SKIM_OK;
    SkimWorkspace ws = skim_carve(ctx->ws, rows, cols);
    ResidualArgs a;
    a.W = W;
    a.rscale = ctx->scaled ? ws.rscale : nullptr;
    a.s = s;
    a.centroids = centroids;
    a.row_bits = row_bits;
    a.width = width;
    a.ld = ld;
    a.ldd = ldd;
    a.cols = (int)cols;
    a.nb = bs.n_bits;
    a.bmin = bs.b_min;
    a.sumk = bs.sumk;
    a.exp2 = exp2;
    a.vec = ((reinterpret_cast<uintptr_t>(D) & 15u) == 0 && ldd % 8 == 0 && cols % 8 == 0 && (!s || (reinterpret_cast<uintptr_t>(s) & 15u) == 0)) ? 1 : 0;
    a.D = D;
    a.status = ws.status;
    return skim_launch_dependent(ctx, skim_residual_kernel, dim3((unsigned)rows), RES_T, 0, a);
}

size_t skim_lfull_cluster_bytes(int64_t rows, int64_t cols)
{
    return skim_align256((size_t)rows * ((cols + BN - 1) / BN) * 2 * KC * sizeof(double));
}

size_t skim_lfull_scratch_bytes(int64_t rows, int64_t cols)
{
    const int64_t mt = (rows + BM - 1) / BM, nt = (cols + BN - 1) / BN;
    return skim_align256((size_t)(mt * BM) * (size_t)nt * SPLIT_MAX * sizeof(float)) + HALF_FLAG_BYTES;
}

int skim_launch_err_lfull(skim_ctx *ctx, const uint16_t *D, int64_t rows, int64_t cols, int64_t ldd, const uint16_t *H,
                          int64_t ldh, int exp2, void *scratch, float *err, int64_t err_stride, float *Y, int64_t ldy,
                          double *err64, const SkimLfullClusters *clusters)
{
    if (rows == 0) return SKIM_OK;
    CUtensorMap map_a, map_b;
    int rc = encode_map(&map_a, D, rows, cols, ldd, CM);
    if (rc) return rc;
    rc = encode_map(&map_b, H, cols, cols, ldh, CB);
    if (rc) return rc;
    GemmArgs a;
    a.D = D;
    a.ldd = ldd;
    a.rows = (int)rows;
    a.cols = (int)cols;
    a.mt = (int)((rows + BM - 1) / BM);
    a.nt = (int)((cols + BN - 1) / BN);
    a.partial = (float *)scratch;
    a.Y = Y;
    a.ldy = ldy;
    a.cl = clusters ? *clusters : SkimLfullClusters{};
    a.sectors = cols % 32 == 0 && ((reinterpret_cast<uintptr_t>(D) | (uintptr_t)ldd * 2) & 31u) == 0 && (!clusters || (reinterpret_cast<uintptr_t>(clusters->labels) & 31u) == 0);
    const size_t smem = gemm_smem(false);
    a.status = (unsigned long long *)ctx->ws;
    SKIM_CUDA_OK(cudaFuncSetAttribute(skim_lfull_gemm_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int tiles = a.mt * a.nt;
    // the tiles of the last round, if it is not full, are cut along K into as many ranges as fit the SMs
    const int nkb = (int)((cols + BK - 1) / BK);
    const int pairs = ctx->sm_count / 2;
    const int rest = tiles % pairs;
    a.full_tiles = tiles;
    a.split = 1;
    if (Y && rest > 0 && 2 * rest <= pairs) {
        a.full_tiles = tiles - rest;
        a.split = 2;
    } else if (!Y && rest > 0) {
        // `rest` tiles in s ranges each take ceil(rest s / pairs) sub-rounds of 1/s tile time: the least, the smaller s on a tie
        int sp = 1;
        double best = 1.0;
        for (int c = 2; c <= SPLIT_MAX && c <= nkb; ++c) {
            const double cost = (double)((rest * c + pairs - 1) / pairs) / c;
            if (cost < best - 1e-9) { best = cost; sp = c; }
        }
        if (sp > 1) {
            a.full_tiles = tiles - rest;
            a.split = sp;
        }
    }
    // Half the contraction where H turns out symmetric, as a Gram matrix is.  The comparison of H with its transpose
    // reads all of H (2 B per entry) under a contraction of rows MACs per entry: at the measured rates the two take equally long
    // near 700 rows (512 x 11008 145 us in full, 158 halved; 768 x 11008 204 and 161).  The further launch, the longer start and
    // the pair's teardown cost 6 us, so the busiest pair must save more than that.  us per call in full and halved where the rule
    // says full: 1536 x 1536 16.6 and 22.7, 1298 x 3072 31.6 and 37.0, 8192 x 1280 32.0 and 37.0, 768 x 6144 51.8 and 55.6; and
    // where it says halved: 1298 x 3216 39.1 and 35.0, 4096 x 1792 39.1 and 30.9, 6000 x 1280 40.7 and 28.8, 1024 x 4096 47.3 and 41.1.
    a.asym = nullptr;
    a.asym_n = 0;
    a.leave = skim_lfull_leave_flag(ctx->ws);
    a.piece_kb = nkb;
    bool halved = !Y && rows >= HALF_MIN_ROWS && a.nt >= HALF_MIN_NT && ctx->sm_count * sizeof(int) <= HALF_FLAG_BYTES;
    if (halved) {
        // pieces of about the full contraction's length (the accumulator's rounding errors grow with it), or half of that
        // where it balances the blocks clearly better
        double best = 0.0;
        const int c0 = a.full_tiles == 0 ? a.split : 1;
        for (int c = c0; c <= 2 * c0 && c <= SPLIT_MAX; ++c) {
            const int piece = (nkb + c - 1) / c;
            const double v = half_makespan(a.mt, a.nt, nkb, piece, pairs);
            if (c == c0 || v < best * 0.95) { best = v; a.piece_kb = piece; }
        }
        // the full contraction's rounds of whole tiles, then of cut ones (a piece takes an epilogue's time at least)
        const int cut = (tiles - a.full_tiles) * a.split;
        auto round_kb = [](double kb) { return kb > EPILOGUE_KB ? kb : EPILOGUE_KB; };
        const double full = (a.full_tiles + pairs - 1) / pairs * round_kb(nkb) + (cut + pairs - 1) / pairs * round_kb((double)nkb / a.split) + EPILOGUE_KB;
        halved = full - best >= HALF_MIN_SAVING;
    }
    if (halved) {
        a.asym = (int *)((char *)scratch + skim_lfull_scratch_bytes(rows, cols) - HALF_FLAG_BYTES);
        a.asym_n = 2 * pairs;
        SKIM_CUDA_OK(cudaFuncSetAttribute(skim_lfull_gemm_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem(true)));
        rc = skim_launch_dependent(ctx, skim_lfull_gemm_kernel<true>, dim3((unsigned)(2 * pairs)), GEMM_THREADS + CHECK_WARPS * 32, gemm_smem(true), map_a, map_b, a, H, ldh);
        if (rc) return rc;
    }
    const int units = a.full_tiles + (tiles - a.full_tiles) * a.split;
    const unsigned blocks = (unsigned)(2 * (units < pairs ? units : pairs));    // persistent: one CTA per SM
    const dim3 red((unsigned)((rows + RED_WARPS - 1) / RED_WARPS));
    if (Y) {
        // In the scaling-vector update the dependents' blocks, moving in under the contraction and its reduction, cost more than the
        // launches they save (a step of 4096 x 4096: 257 us so, 249 with ordinary launches).
        skim_lfull_gemm_kernel<false><<<blocks, GEMM_THREADS, smem, ctx->stream>>>(map_a, map_b, a, H, ldh);
        SKIM_CUDA_OK(cudaGetLastError());
        skim_lfull_reduce_kernel<<<red, RED_WARPS * 32, 0, ctx->stream>>>(a, exp2, err, err_stride, err64);
        SKIM_CUDA_OK(cudaGetLastError());
        ctx->launches += 2;
        return SKIM_OK;
    }
    rc = skim_launch_dependent(ctx, skim_lfull_gemm_kernel<false>, dim3(blocks), GEMM_THREADS, smem, map_a, map_b, a, H, ldh);
    if (rc) return rc;
    return skim_launch_dependent(ctx, skim_lfull_reduce_kernel, red, RED_WARPS * 32, 0, a, exp2, err, err_stride, err64);
}
