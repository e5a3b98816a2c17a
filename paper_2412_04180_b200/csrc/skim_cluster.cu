// Row clustering: weighted 1-D K-means of every matrix row at every candidate width (SKIM
// Algorithm 3, error pre-recording loop; objective of Section 3.2, diagonal form), in two kernels
// per chunk of rows: a sort kernel (one block per row) that leaves the sorted row, its group index
// and its block prefix sums in a row record in global memory, and the Lloyd kernel (skim_lloyd.cu,
// one warp per row, thousands of rows in flight) that iterates on the records.  The split exists
// because the Lloyd iteration is a long chain of dependent small steps: inside the sort block it ran
// on one warp while two rows filled an SM's shared memory; from global memory (the hot lines stay in
// L1) every SM keeps 28 rows in flight.
//
// Long unscaled rows are sorted by skim_cluster16.cu, the others by skim_bucket.cu.  Rows that the bucket kernel cannot spread (few
// distinct values, clumps) go on a list: unscaled ones to skim_cluster16.cu, scaled ones to the radix sort kernel of this
// file.  With it the host-side launcher of the whole clustering.
//
// One thread block owns one row at a time.
//   1. load   the row's (value, importance) pairs into registers; the value is turned into an
//             order-preserving unsigned key.
//   2. sort   block-wide LSD radix sort (8-bit digits, warp-private digit counters, ballot-based
//             stable ranking), exchanging through one shared-memory buffer.  Afterwards every
//             1-D cluster is a contiguous interval of the sorted row.
//   3.        one pass over the sorted row writes its row record (skim_cluster_phases.cuh).
#include "skim_cluster_phases.cuh"

namespace {

using namespace skimk;

// Unscaled rows up to this length go to the bucket kernel too.  The fp16-key kernel clears and scans its counters twice whatever
// the row length, and places every element twice: us for 4096 rows there and in buckets, 700 columns 70 and 33, 4096 129.6 and 102, 8192 238.8 and
// 215 (rows that the buckets refuse: skim_bucket.cu).  Beyond, the buckets' counters leave fewer blocks on an SM: 11 008 columns 289.4 and
// 308.1, 2000 rows of 22 016 334 and 365 (of 16 000 263 and 255).
constexpr int BUCKET_UNSCALED_COLS = 8192;
constexpr int RADIX_BITS = 8;
constexpr int RADIX = 1 << RADIX_BITS;

constexpr int PASSES = 32 / RADIX_BITS;

// Shared-memory layout, computed identically on host and device.
struct SmemLayout {
    size_t keys, gs, uni, dbase, phase, total;
};

__host__ __device__ inline SmemLayout smem_layout(int cap, int nwarps)
{
    SmemLayout L;
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off += (b + 15) & ~(size_t)15; return o; };
    L.keys = take((size_t)cap * 4);
    L.gs = take((size_t)cap * 4);
    L.uni = take((size_t)nwarps * RADIX * 4);
    L.dbase = take(RADIX * 4);
    L.phase = take(sizeof(PhaseSmem));
    L.total = off;
    return L;
}

// Takes the rows of a.sort_list (blocks leave at once when it is empty, the usual case).  The kernel after this one may start as the blocks leave, no
// earlier: the Lloyd blocks of few rows, moving in beside blocks that sort, waited there with their split of shared memory and L1 (clustering of rows
// that are all listed, us, let in at once and now: 1000 x 11008 scaled 384 and 353, 300 x 8192 scaled 114 and 111, 500 x 1500 unscaled 39 and 35).
template <int THREADS, int ITEMS>
__global__ void __launch_bounds__(THREADS) skim_sort_kernel(ClusterArgs a)
{
    using K = KeyOps<uint32_t>;
    constexpr int NW = THREADS / 32;
    constexpr int CAP = THREADS * ITEMS;
    extern __shared__ __align__(16) unsigned char smem[];
    const SmemLayout L = smem_layout(CAP, NW);
    uint32_t *skeys = reinterpret_cast<uint32_t *>(smem + L.keys);
    float *sg = reinterpret_cast<float *>(smem + L.gs);
    uint32_t *cnt = reinterpret_cast<uint32_t *>(smem + L.uni);
    uint32_t *dbase = reinterpret_cast<uint32_t *>(smem + L.dbase);
    PhaseSmem &ps = *reinterpret_cast<PhaseSmem *>(smem + L.phase);

    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    const int m = a.m;
    skim_wait_for_previous_kernel();
    const int listed = min(*a.sort_count, a.chunk_rows);
    for (int at = blockIdx.x; at < listed; at += gridDim.x) {
    const int local = a.sort_list[at];
    const int64_t row = a.row0 + local;
    const uint16_t *Wr = a.W + row * a.ld;
    const float *Gr = a.G + row * a.ld;

    // ---------------------------------------------------------------- 1. load
    uint32_t key[ITEMS];
    float val[ITEMS];
    unsigned bad = 0;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int e = warp * (ITEMS * 32) + i * 32 + lane;
        if (e < m) {
            const uint16_t h = Wr[e];
            const float g = Gr[e];
            if ((h & 0x7c00u) == 0x7c00u) bad |= 1u;
            if (!(g >= 0.0f) || g > 3.0e38f) bad |= 2u;
            float x = __half2float(__ushort_as_half(h));
            x = __fmul_rn(x, a.rscale[e]);
            if (x == 0.0f) x = 0.0f;
            key[i] = K::from_float(x);
            val[i] = g;
        } else {
            key[i] = K::PAD;
            val[i] = 0.0f;
        }
    }
    if (bad) atomicOr(a.status, (unsigned long long)bad);

    // ---------------------------------------------------------------- 2. sort
    const unsigned lt_mask = (1u << lane) - 1u;
#pragma unroll 1
    for (int pass = 0; pass < PASSES; ++pass) {
        const int shift = pass * RADIX_BITS;
        for (int d = tid; d < NW * RADIX; d += THREADS) cnt[d] = 0;
        __syncthreads();
        // count: warp-private histogram of this digit
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const unsigned d = ((unsigned)key[i] >> shift) & (RADIX - 1);
            atomicAdd(&cnt[warp * RADIX + d], 1u);
        }
        __syncthreads();
        // scan: per digit over warps (exclusive, in place), then over digits
        for (int d = tid; d < RADIX; d += THREADS) {
            uint32_t run = 0;
            for (int w = 0; w < NW; ++w) {
                const uint32_t c = cnt[w * RADIX + d];
                cnt[w * RADIX + d] = run;
                run += c;
            }
            dbase[d] = run;
        }
        __syncthreads();
        if (warp == 0) {
            uint32_t loc[RADIX / 32];
            uint32_t s = 0;
#pragma unroll
            for (int u = 0; u < RADIX / 32; ++u) { loc[u] = dbase[lane * (RADIX / 32) + u]; s += loc[u]; }
            uint32_t inc = s;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, inc, off);
                if (lane >= off) inc += t;
            }
            uint32_t run = inc - s;
#pragma unroll
            for (int u = 0; u < RADIX / 32; ++u) { dbase[lane * (RADIX / 32) + u] = run; run += loc[u]; }
        }
        __syncthreads();
        // rank and scatter: items of one warp are taken in position order, so the pass is stable
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const unsigned d = ((unsigned)key[i] >> shift) & (RADIX - 1);
            unsigned peers = 0xffffffffu;   // lanes of this warp whose item has the same digit
#pragma unroll
            for (int b = 0; b < RADIX_BITS; ++b) {
                const bool bit = (d >> b) & 1u;
                const unsigned bal = __ballot_sync(0xffffffffu, bit);
                peers &= bit ? bal : ~bal;
            }
            const uint32_t base = cnt[warp * RADIX + d];
            const unsigned rank = __popc(peers & lt_mask);
            __syncwarp();
            if (rank == 0) cnt[warp * RADIX + d] = base + __popc(peers);
            __syncwarp();
            const uint32_t pos = dbase[d] + base + rank;
            if (SKIM_IDX(pos, CAP, a.status)) {
                skeys[pos] = key[i];
                sg[pos] = val[i];
            }
        }
        __syncthreads();
        if (pass + 1 < PASSES) {
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                const int e = warp * (ITEMS * 32) + i * 32 + lane;
                key[i] = skeys[e];
                val[i] = sg[e];
            }
            // the next pass re-zeroes the counters and syncs before anyone scatters again
        }
    }

    // ---------------------------------------------------------------- 3. row record for the Lloyd kernel
    if (tid == 0) { ps.misc[0] = 0; ps.misc[1] = 0; }
    __syncthreads();
    const SortedArrays<uint32_t> src{skeys, sg};
    const int nd = write_row_record<uint32_t, THREADS, true>(a, src, ps, 0, local);
    if (nd <= 16) {
        collect_distinct<uint32_t, THREADS>(src, m, nd, ps);
        write_distinct_values(a, nd, ps.dvals, local);
    }
    __syncthreads();
    }
}

struct Variant {
    int cap;
    int threads;
    void (*kernel)(ClusterArgs);
};

#define SKIM_VARIANT(T, I) {T * I, T, skim_sort_kernel<T, I>}

// A row pays for the whole size: with 512 x 8, 22 and 44 only, 4096 refused rows of 5600 columns took 1167 us, with 512 x 16 890.
const Variant kVariants32[] = {SKIM_VARIANT(256, 2), SKIM_VARIANT(256, 8), SKIM_VARIANT(512, 8), SKIM_VARIANT(512, 16), SKIM_VARIANT(512, 22),
                               SKIM_VARIANT(512, 32), SKIM_VARIANT(512, 44)};
constexpr int kNumVariants = sizeof(kVariants32) / sizeof(kVariants32[0]);

// Picks the smallest variant that holds `cols` and fits shared memory.
const Variant *pick_variant(const Variant *table, int64_t cols, int max_smem, size_t *smem)
{
    for (int v = 0; v < kNumVariants; ++v) {
        if (table[v].cap < cols) continue;
        const SmemLayout L = smem_layout(table[v].cap, table[v].threads / 32);
        if (L.total <= (size_t)max_smem) { *smem = L.total; return &table[v]; }
    }
    return nullptr;
}

}  // namespace

int skim_cluster_max_cols(int max_smem_optin, int64_t *out)
{
    int64_t best = 0;
    for (int v = 0; v < kNumVariants; ++v) {
        size_t b;
        if (pick_variant(kVariants32, kVariants32[v].cap, max_smem_optin, &b)) best = kVariants32[v].cap;
    }
    *out = best;
    return SKIM_OK;
}

int skim_launch_cluster(skim_ctx *ctx, const uint16_t *W, const float *importance, int64_t rows,
                        int64_t cols, int64_t ld, const uint8_t *row_bits, const SkimBits &bits,
                        int iters, float *centroids, uint8_t *codes, float *err, void *exact_scratch)
{
    if (rows == 0) return SKIM_OK;
    SkimWorkspace ws = skim_carve(ctx->ws, rows, cols);
    const bool scaled = ctx->scaled;
    ClusterArgs a;
    a.W = W;
    a.G = importance;
    a.rscale = scaled ? ws.rscale : nullptr;
    a.row_bits = row_bits;
    a.rows = rows;
    a.ld = ld;
    a.m = (int)cols;
    a.nb = bits.n_bits;
    a.bmin = bits.b_min;
    a.sumk = bits.sumk;
    a.iters = iters;
    a.centroids = centroids;
    a.codes = codes;
    a.err = err;
    a.status = ws.status;
    a.scratch = ws.cluster_scratch;
    a.row0 = 0;
    a.early_exit = ctx->early_exit ? 1 : 0;
    a.iter_stats = ctx->timing ? ws.status + 1 : nullptr;

    // unscaled rows get compact records (the exact kernel reads the full ones with their g*x^2 prefixes)
    a.rec_half = (!scaled && !exact_scratch) ? 1 : 0;
    a.rec_stride = (long long)row_record(a.m, a.rec_half != 0).total;
    a.full_order = exact_scratch ? 1 : 0;
    a.sort_list = ws.sort_list;
    a.sort_count = (int *)(ws.status + 4);
    size_t smem = 0;
    const Variant *v = nullptr;
    const bool bucket = scaled || (a.rec_half && cols <= BUCKET_UNSCALED_COLS);
    a.unordered = bucket ? 1 : 0;
    if (scaled) {
        v = pick_variant(kVariants32, cols, ctx->max_smem_optin, &smem);
        if (!v) return SKIM_ERR_SHAPE;
        SKIM_CUDA_OK(cudaFuncSetAttribute(v->kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    }
    if ((size_t)a.rec_stride > skim_cluster_record_bytes(cols)) return SKIM_ERR_WORKSPACE;

    for (int64_t row0 = 0; row0 < rows; row0 += SKIM_CLUSTER_CHUNK_ROWS) {
        const int64_t n = rows - row0 < SKIM_CLUSTER_CHUNK_ROWS ? rows - row0 : SKIM_CLUSTER_CHUNK_ROWS;
        a.row0 = row0;
        cudaEvent_t *tev = (ctx->timing && ctx->timing_used < SKIM_TIMING_SLOTS) ? ctx->timing_ev[ctx->timing_used] : nullptr;
        if (tev) SKIM_CUDA_OK(cudaEventRecord(tev[0], ctx->stream));
        a.chunk_rows = (int)n;
        bool lists = false;
        int rc = bucket ? skim_launch_sort_bucket(ctx, a, n, &lists) : skim_launch_sort16(ctx, a, n);
        if (rc) return rc;
        if (lists) {
            // the rows the buckets could not spread: usually none
            if (scaled) rc = skim_launch_dependent(ctx, v->kernel, dim3(skim_list_blocks(ctx, v->threads, n)), v->threads, smem, a);
            else rc = skim_launch_sort16(ctx, a, n, true);
            if (rc) return rc;
        }
        if (tev) SKIM_CUDA_OK(cudaEventRecord(tev[1], ctx->stream));
        rc = exact_scratch ? skim_launch_exact(ctx, a, n, exact_scratch, skim_exact_slots(ctx, rows, cols))
                                     : skim_launch_lloyd(ctx, a, n);
        if (rc) return rc;
        if (tev) {
            SKIM_CUDA_OK(cudaEventRecord(tev[2], ctx->stream));
            ctx->timing_used += 1;
        }
    }
    return SKIM_OK;
}
