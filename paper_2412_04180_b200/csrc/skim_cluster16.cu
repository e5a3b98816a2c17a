// fp16-key row-sorting kernel, the first half of the row clustering (SKIM Algorithm 3, error pre-recording loop; objective of
// Section 3.2, diagonal form) where no scale vector is installed: rows too long for skim_bucket.cu to be faster, and all
// rows of the exact clustering.  The sort itself is in skim_sort16.cuh.
#include "skim_sort16.cuh"

namespace {

using namespace skimk;

// HALF_RECORD: the compact row record, for the Lloyd kernel; else the full one, for the exact kernel.
template <bool HALF_RECORD, int THREADS, int VEC>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) skim_sort16_kernel(ClusterArgs a)
{
    skim_let_next_kernel_start();
    skim_wait_for_previous_kernel();
    sort16_row<HALF_RECORD, THREADS, VEC, true>(a, (int)blockIdx.x, 0u);
}

// The rows that the bucket kernel has put on a.sort_list (usually none).  The next kernel may start as the blocks leave (see skim_cluster.cu).
template <int THREADS, int VEC>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) skim_sort16_list_kernel(ClusterArgs a)
{
    skim_wait_for_previous_kernel();
    const int listed = min(*a.sort_count, a.chunk_rows);
    if ((int)blockIdx.x >= listed) return;
    extern __shared__ __align__(16) unsigned char smem[];
    if (threadIdx.x == 0) mbar_init(reinterpret_cast<uint64_t *>(smem + layout16(a.m, THREADS).mbar), 1);      // (a barrier follows)
    bool ok = true;
    uint32_t parity = 0u;
    for (int at = blockIdx.x; at < listed; at += gridDim.x, parity ^= 1u) {
        const int local = a.sort_list[at];
        if (ok) ok = sort16_row<true, THREADS, VEC, false>(a, local, parity);
        else if (threadIdx.x == 0) *reinterpret_cast<int *>(a.scratch + (size_t)local * (size_t)a.rec_stride) = -1;      // a copy may still be in flight
        __syncthreads();
    }
}

struct Variant16 {
    int cap;
    int threads;
    void (*kernel[2])(ClusterArgs);      // full record, compact record
};

#define SKIM_V16(T, V) {T * V * 8, T, {skim_sort16_kernel<false, T, V>, skim_sort16_kernel<true, T, V>}}
#define SKIM_V16F(T, V) {T * V * 8, T, {skim_sort16_kernel<false, T, V>, nullptr}}      // short rows with compact records: skim_bucket.cu
#define SKIM_V16L(T, V) {T * V * 8, T, {nullptr, skim_sort16_list_kernel<T, V>}}

// An SM holds 1024 threads; small blocks wait for their own barriers only.
const Variant16 kVariants16[] = {
    SKIM_V16F(128, 1), SKIM_V16F(128, 2), SKIM_V16F(256, 2), SKIM_V16F(256, 3), SKIM_V16F(512, 2), SKIM_V16(512, 3), SKIM_V16(1024, 2),
    SKIM_V16(1024, 3),
};
// The rows that the bucket kernel refuses.  No smaller blocks: short rows are mostly the work on the 4096 counters, and the launch,
// which usually finds the list empty, has fewer blocks (1184 of 128 threads cost 0.7 us, 592 of 256 nothing measurable).
const Variant16 kVariantsList16[] = {SKIM_V16L(256, 1)};

template <int N>
const Variant16 *pick16(const Variant16 (&table)[N], const skim_ctx *ctx, int m)
{
    for (const Variant16 &v : table)
        if (v.cap >= m && layout16(m, v.threads).total <= (size_t)ctx->max_smem_optin) return &v;
    return nullptr;
}

}  // namespace

int skim_launch_sort16(skim_ctx *ctx, const ClusterArgs &args, int64_t rows, bool listed)
{
    const Variant16 *v = listed ? pick16(kVariantsList16, ctx, args.m) : pick16(kVariants16, ctx, args.m);
    void (*kernel)(ClusterArgs) = v ? v->kernel[args.rec_half ? 1 : 0] : nullptr;
    if (!kernel) return SKIM_ERR_SHAPE;
    const size_t smem = layout16(args.m, v->threads).total;
    // set on every launch: a host-side call of microseconds, and no state shared between contexts
    SKIM_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (listed) return skim_launch_dependent(ctx, kernel, dim3(skim_list_blocks(ctx, v->threads, rows)), v->threads, smem, args);
    return skim_launch_dependent(ctx, kernel, dim3((unsigned)rows), v->threads, smem, args);
}
