// Internal declarations shared by the translation units of libskim.so.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "skim.h"

#define SKIM_MAX_NBITS SKIM_MAX_BIT
#define SKIM_HOST_CHUNKS 8   // row chunks of the host-buffer entry point, and how many with the last one cut further
#define SKIM_HOST_EVENTS 14
#define SKIM_MAX_SUMK 30  // 2 + 4 + 8 + 16: one warp lane per centroid
#define SKIM_TIMING_SLOTS 256   // clustering chunks whose kernel times skim_kernel_timing can hold

struct skim_ctx {
    int device;
    cudaStream_t stream;
    int sm_count;
    int max_smem_optin;   // bytes of dynamic shared memory one block may opt into
    void *ws;             // caller's workspace
    size_t ws_bytes;
    bool scaled;          // a scale vector is installed
    int64_t scale_cols;
    int64_t launches;
    // host-buffer entry point: a second stream for the host-to-device copies, so that the copy
    // of one row chunk runs under the clustering of the previous one (created on first use)
    cudaStream_t copy_stream;
    cudaEvent_t copy_done[SKIM_HOST_EVENTS];
    cudaEvent_t main_idle;
    bool copy_ready;
    // optional kernel timing: events before the sort kernel, between the two kernels and after
    // the Lloyd kernel of every clustering chunk, on the context's stream
    bool early_exit;      // rows stop iterating once no boundary moved (default)
    bool timing;
    bool timing_ready;
    int timing_used;
    cudaEvent_t timing_ev[SKIM_TIMING_SLOTS][3];
};

// Workspace layout (all offsets 256-byte aligned), carved per call for the call's (rows, cols).
// The status word and the reciprocal scale sit at fixed offsets, so they persist across calls.
struct SkimWorkspace {
    unsigned long long *status;  // word 0: status bits; words 1, 2: Lloyd iterations run and rows counted (skim_lloyd_iterations); word 4: length of sort_list; word 5: skim_lfull_leave_flag
    float *rscale;               // [cols]     reciprocal of the installed scale vector
    int32_t *row_pos;            // [rows]     packed-row index of every source row
    double *alpha64;             // [cols]     scale-update master copy of alpha
    double *adam_m;              // [cols]
    double *adam_v;              // [cols]
    double *loss_part;           // [rows]     scale update: loss of every row
    double *grad_part;           // [SKIM_SCALE_MAX_CTAS][cols]  partial gradients of the row ranges
    double *scale_const;         // [rows][16][2]  scale update: per-cluster constants (sum g, sum g w^2)
    double *scale_cq;            // [rows][16][2]  scale update: per-cluster centroid and gradient factor
    uint16_t *scale_ord_end;     // [rows][16]  scale update: steps of the clusters in the label-ordered rows
    int *sort_list;              // [min(rows, SKIM_CLUSTER_CHUNK_ROWS)] rows the bucket sort kernel leaves to the radix kernel
    unsigned char *cluster_scratch;  // [min(rows, SKIM_CLUSTER_CHUNK_ROWS)] row records of the clustering; during a scale update the label-ordered matrix
    size_t bytes;                // enough for every call
    size_t bytes_no_update;      // enough for every call but the scale updates (the records, not the label-ordered matrix)
};

#define SKIM_SCALE_MAX_CTAS 296
#define SKIM_CLUSTER_CHUNK_ROWS 8192   // rows clustered per sort-kernel / Lloyd-kernel pair

// Upper bound of one row record of the clustering: 128-byte header, 96 bytes per group of 8
// elements, group index 0.5 B per element, segment table, plus rounding.
__host__ __device__ static inline size_t skim_cluster_record_bytes(int64_t cols)
{
    const size_t m8 = ((size_t)cols + 7) & ~(size_t)7;
    return (13 * m8 + 1024 + 127) & ~(size_t)127;
}

// The label-ordered matrix of the scale update (skim_scale.cu): elements (8 bytes each) of a row, at most -- rows of up to
// SKIM_ORDER_SHORT_COLS have no padding (an even number of elements), the others have 16 clusters padded to whole units of
// 64 -- and the bytes behind the last row that its readers may fetch.
#define SKIM_ORDER_UNIT 64
#define SKIM_ORDER_SHORT_COLS 512
#define SKIM_ORDER_SLACK 8192
__host__ __device__ static inline int64_t skim_ordered_stride(int64_t cols)
{
    if (cols <= SKIM_ORDER_SHORT_COLS) return (cols + 1) / 2 * 2;
    return (cols + SKIM_ORDER_UNIT - 1) / SKIM_ORDER_UNIT * SKIM_ORDER_UNIT + 16 * SKIM_ORDER_UNIT;
}

// The half contraction's leave flag (skim_lfull.cu), in the status words at the start of the workspace: zero between calls.
static inline unsigned *skim_lfull_leave_flag(void *ws) { return (unsigned *)((unsigned long long *)ws + 5); }

static inline size_t skim_align256(size_t v) { return (v + 255) & ~(size_t)255; }

static inline SkimWorkspace skim_carve(void *base, int64_t rows, int64_t cols)
{
    SkimWorkspace w;
    char *p = (char *)base;
    size_t off = 0;
    auto take = [&](size_t bytes) { char *q = p ? p + off : nullptr; off += skim_align256(bytes); return q; };
    w.status = (unsigned long long *)take(256);
    w.rscale = (float *)take((size_t)cols * 4);
    w.row_pos = (int32_t *)take((size_t)rows * 4);
    w.alpha64 = (double *)take((size_t)cols * 8);
    w.adam_m = (double *)take((size_t)cols * 8);
    w.adam_v = (double *)take((size_t)cols * 8);
    w.loss_part = (double *)take((size_t)(rows > SKIM_SCALE_MAX_CTAS ? rows : SKIM_SCALE_MAX_CTAS) * 8);
    w.grad_part = (double *)take((size_t)SKIM_SCALE_MAX_CTAS * (size_t)cols * 8);
    w.scale_const = (double *)take((size_t)rows * 16 * 2 * 8);
    w.scale_cq = (double *)take((size_t)rows * 16 * 2 * 8);
    w.scale_ord_end = (uint16_t *)take((size_t)rows * 16 * 2);
    w.sort_list = (int *)take((size_t)(rows < SKIM_CLUSTER_CHUNK_ROWS ? rows : SKIM_CLUSTER_CHUNK_ROWS) * 4);
    const size_t records = (size_t)(rows < SKIM_CLUSTER_CHUNK_ROWS ? rows : SKIM_CLUSTER_CHUNK_ROWS) * skim_cluster_record_bytes(cols);
    const size_t ordered = (size_t)rows * (size_t)skim_ordered_stride(cols) * 8 + SKIM_ORDER_SLACK;
    w.bytes_no_update = off + skim_align256(records);
    w.cluster_scratch = (unsigned char *)take(records > ordered ? records : ordered);
    w.bytes = off;
    return w;
}

// Index checks of the checked build (nvcc -DSKIM_CHECK_BOUNDS; build.py builds it as libskim_checked.so).
// Every index into shared memory, a row record or a scratch list that is COMPUTED from data (a scatter
// position, a counter slot, a searched group, a gathered column) goes through SKIM_IDX: in the checked
// build an index outside [0, n) sets SKIM_STATUS_BOUNDS in the status word and the access is skipped
// (never a trap); in the normal build the macro is the constant true and costs nothing.
#ifdef SKIM_CHECK_BOUNDS
__device__ __forceinline__ bool skim_index_ok(long long i, long long n, unsigned long long *status)
{
    if (i >= 0 && i < n) return true;
    if (status) atomicOr(status, (unsigned long long)SKIM_STATUS_BOUNDS);
    return false;
}
#define SKIM_IDX(i, n, status) skim_index_ok((long long)(i), (long long)(n), (status))
#else
#define SKIM_IDX(i, n, status) true
#endif

// Validated description of a bit set.
struct SkimBits {
    int n_bits;
    int b_min;
    int b_max;
    int sumk;
};

int skim_check_bits(const int *bit_set, int n_bits, SkimBits *out);

#define SKIM_CUDA_OK(expr)                         \
    do {                                           \
        cudaError_t e_ = (expr);                   \
        if (e_ != cudaSuccess) return SKIM_ERR_CUDA; \
    } while (0)

// Launchers implemented in the kernel translation units.  All return SKIM_OK or SKIM_ERR_*.
// exact_scratch == nullptr: Lloyd iterations (Algorithm 3); else the exact optimum of every row (skim_exact.cu)
int skim_launch_cluster(skim_ctx *ctx, const uint16_t *W, const float *importance, int64_t rows,
                        int64_t cols, int64_t ld, const uint8_t *row_bits, const SkimBits &bits,
                        int iters, float *centroids, uint8_t *codes, float *err, void *exact_scratch = nullptr);
size_t skim_exact_slot_bytes(int64_t cols);
int skim_exact_slots(const skim_ctx *ctx, int64_t rows, int64_t cols);
int skim_cluster_max_cols(int max_smem_optin, int64_t *out);
int skim_launch_reciprocal(skim_ctx *ctx, const float *s, int64_t cols);
int skim_launch_allocate(skim_ctx *ctx, const float *err, int64_t rows, const SkimBits &bits, int first_col,
                         int64_t K, uint8_t *out_bits);
size_t skim_allocate_optimal_scratch(int64_t rows, int64_t K);
int skim_launch_allocate_optimal(skim_ctx *ctx, const float *err, int64_t rows, const SkimBits &bits, int64_t K,
                                 void *scratch, uint8_t *out_bits, double *cost);
int skim_launch_quantize(skim_ctx *ctx, const uint16_t *W, int64_t rows, int64_t cols, int64_t ld,
                         const uint8_t *bits, const float *centroids, const SkimBits &bs,
                         uint32_t *packed, int32_t *row_order, int64_t *group_info, uint16_t *lut);
int skim_launch_dequantize(skim_ctx *ctx, const uint32_t *packed, const int32_t *row_order, const int64_t *group_info,
                           const uint16_t *lut, const float *s, int64_t rows, int64_t cols, const SkimBits &bs,
                           uint16_t *out, int64_t ld_out);
int skim_launch_matvec(skim_ctx *ctx, const uint32_t *packed, const int32_t *row_order, const int64_t *group_info,
                       const uint16_t *lut, const float *s, const uint16_t *x, int64_t rows, int64_t cols,
                       const SkimBits &bs, float *y);
int skim_launch_scale_update(skim_ctx *ctx, const uint16_t *W, const float *importance, int64_t rows,
                             int64_t cols, int64_t ld, const uint8_t *labels, float *alpha, int steps,
                             float lr0, float decay, int decay_every, double *loss_trace);

int skim_launch_residual(skim_ctx *ctx, const uint16_t *W, int64_t rows, int64_t cols, int64_t ld, const float *centroids,
                         const uint8_t *row_bits, int width, const SkimBits &bs, const float *s, int exp2, uint16_t *D,
                         int64_t ldd);
size_t skim_lfull_scratch_bytes(int64_t rows, int64_t cols);
// Sums of Y alpha by cluster, R_ik = sum_{j in k} Y_ij alpha_j, formed in the contraction's epilogue for the scale update.
struct SkimLfullClusters {
    const uint8_t *labels;   // [rows][cols]
    const double *alpha;     // [cols]
    double *rpart;           // skim_lfull_cluster_bytes(): per row, column tile and half of it
    const double2 *tconst;   // [rows][16]  (G_k, .)
    double2 *tq;             // [rows][16]  y <- 2 R_k / (2^exp2 G_k)
};
size_t skim_lfull_cluster_bytes(int64_t rows, int64_t cols);
// Y (optional): the product D H itself, [rows][ldy] binary32; err64 (optional): the row errors in binary64
int skim_launch_err_lfull(skim_ctx *ctx, const uint16_t *D, int64_t rows, int64_t cols, int64_t ldd, const uint16_t *H,
                          int64_t ldh, int exp2, void *scratch, float *err, int64_t err_stride, float *Y = nullptr,
                          int64_t ldy = 0, double *err64 = nullptr, const SkimLfullClusters *clusters = nullptr);
size_t skim_scale_lfull_scratch_bytes(int64_t rows, int64_t cols);
int skim_launch_scale_update_lfull(skim_ctx *ctx, const uint16_t *W, const float *importance, int64_t rows, int64_t cols,
                                   int64_t ld, const uint8_t *labels, const uint16_t *H, int64_t ldh, float *alpha,
                                   int steps, float lr0, float decay, int decay_every, int exp2, void *scratch,
                                   double *loss_trace);

__host__ __device__ static inline int64_t skim_row_stride_words(int64_t cols, int b)
{
    int64_t w = (cols * (int64_t)b + 31) / 32;
    return (w + 3) / 4 * 4;
}

// Programmatic dependent launches: the kernel may start while the one before it on the stream drains, and waits itself
// before it reads what that one (or any earlier one) wrote and before it writes anything.
__device__ __forceinline__ void skim_wait_for_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void skim_let_next_kernel_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... Params, typename... Args>
int skim_launch_dependent_on(cudaStream_t stream, void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    SKIM_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, args...));
    return SKIM_OK;
}
template <typename... Params, typename... Args>
int skim_launch_dependent(skim_ctx *ctx, void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, Args... args)
{
    const int rc = skim_launch_dependent_on(ctx->stream, kernel, grid, threads, smem, args...);
    if (rc == SKIM_OK) ctx->launches += 1;
    return rc;
}
