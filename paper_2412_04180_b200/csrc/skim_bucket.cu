// Row-sorting kernel, the first half of the row clustering (SKIM Algorithm 3, error pre-recording loop; objective of
// Section 3.2, diagonal form).  One block per row: every element's bucket is a monotone function of its value, chosen so that a bucket holds about one
// element of a bell-shaped row; one counting pass orders the row up to the order inside the buckets.
//
// Two kernels, for scaled rows (binary32 products) and for unscaled ones (the binary16 weights themselves), of the same steps:
//   load     values and the sum of |x|, which sets the buckets' scale.
//   count    one shared-memory atomic per element; its return value is the element's slot inside its bucket.
//   scatter  bucket base + slot: value and importance (read from global memory here) go to their bucket's place.
//   order    the buckets that reach from one group of 8 into the next are sorted (groups ascend; inside a group the Lloyd
//            kernel compares every element with its boundary, so its order does not matter; in scaled rows the record pass
//            puts the group in order, for sums that are the same on every run).
//   then     one pass over the row (skim_cluster_phases.cuh) writes the row record -- group records with
//            prefix sums, group index, segment table -- to global memory, from which the Lloyd kernel
//            (skim_lloyd.cu) iterates with one warp per row.  Unscaled rows write the compact record.
//
// Buckets: v = 1 + |x| / s with s half a standard deviation (from the mean of |x|).  The bits of v grow with |x|: the
// first three octaves, v in [1, 8), i.e. |x| up to 3.5 deviations, have N/8 buckets each on either side of zero, the next
// eight share N/8 (N = 32 per thread).  A row whose values this cannot spread (a bucket with BUCKET_LIMIT elements, or 32 in
// three neighbouring ones; unscaled rows: see there) is sorted by 16-bit keys (skim_sort16.cuh), by the block itself or through a list by the kernel
// of skim_cluster16.cu, or, where scaled, goes through the list to the radix kernel of skim_cluster.cu (sort of 4096 x 11008 scaled, us: a few nearby
// values 1281, bell-shaped rows 374).
//
// Zeros (a pruned matrix) are one value and need no bucket: a row that cannot be spread and has zeros is read again and spread with
// its zeros between the negative and the positive buckets in column order, by ballots, the scale taken from the other elements.
// (One pass that always looks for zeros cost rows without any 4-15 %: every register is taken.)  Sort of a matrix with half of its
// weights zero, us, before (all its rows went to the radix kernel) and with its zeros apart: 4096 x 11008 scaled 1313 -> 447, the
// same matrix unpruned 374.
//
// Why not a radix sort: rows of 32-bit keys took four passes, each with ballots or random shared-memory traffic of all
// elements (1.17 ms for 4096 x 11008); 16-bit keys two (0.284 ms).  What bounds this kernel is the same resource,
// shared-memory wavefronts of random accesses, but there is one counting atomic and one scatter per element.
#include "skim_sort16.cuh"

#include <algorithm>

namespace {

using namespace skimk;

constexpr int BUCKET_LIMIT = 48;
constexpr unsigned ZEROS_APART = 16;     // fewer are not what a bucket is refused for

template <int THREADS> struct Buckets {
    static constexpr int N = 32 * THREADS;
    static constexpr int HALF = N / 2;
    static constexpr int LOG = (THREADS == 128 ? 9 : THREADS == 256 ? 10 : THREADS == 512 ? 11 : 12);      // log2(N / 8)
    static_assert((8 << LOG) == N, "eight octave blocks");
    float inv_s;
    // ascends with x (not -0); any bit pattern of x gives an index inside [0, N)
    __device__ __forceinline__ int operator()(float x) const
    {
        const uint32_t b = __float_as_uint(__fmaf_rn(fabsf(x), inv_s, 1.0f)) - 0x3f800000u;
        // below three octaves the second term wraps round to a large number, beyond them it is the smaller one
        const uint32_t i = min(min(b >> (23 - LOG), ((b - (3u << 23)) >> (26 - LOG)) + 3u * (N / 8)), (uint32_t)HALF - 1u);
        return HALF + (int)(i ^ (uint32_t)(__float_as_int(x) >> 31));          // negative: HALF - 1 - i
    }
};

// keys, gs: values and importances in bucket order
// uni:      the bucket counters, four 8-bit ones a word; then, in their place, the positions of the four buckets: the first
//           one's in bits 15.., the elements between it and each of the others in three 5-bit fields
struct BucketLayout {
    size_t keys, gs, uni, phase, total;
};
__host__ __device__ inline BucketLayout bucket_layout(int m, int threads)
{
    BucketLayout L;
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off += (b + 15) & ~(size_t)15; return o; };
    const size_t mpad = ((size_t)m + 7) & ~(size_t)7;
    L.keys = take(mpad * 4);
    L.gs = take(mpad * 4);
    L.uni = take((size_t)threads * 32);
    L.phase = take(sizeof(PhaseSmem));
    L.total = off;
    return L;
}

// Insertion sort of n elements by one thread, equal values by importance.
__device__ __forceinline__ void sort_bucket(float *keys, float *gs, int lo, int n)
{
    for (int i = lo + 1; i < lo + n; ++i) {
        const float k = keys[i], g = gs[i];
        int j = i;
        for (; j > lo; --j) {
            const float y = keys[j - 1];
            if (y < k || (y == k && gs[j - 1] <= g)) break;
            keys[j] = y;
            gs[j] = gs[j - 1];
        }
        if (j != i) {
            keys[j] = k;
            gs[j] = g;
        }
    }
}

// Zeros kept apart: of every warp, and behind them the row's.
__device__ __forceinline__ uint32_t *bucket_zeros(PhaseSmem &ps) { return reinterpret_cast<uint32_t *>(ps.segtot) + 64; }

// First position of bucket b, from the words that the scan leaves in the counters' place.
__device__ __forceinline__ int bucket_base(const uint32_t *cnt, int b)
{
    const uint32_t w = cnt[b >> 2];
    return (int)((w >> 15) + (((w << 5) >> (5 * (b & 3))) & 31u));
}

struct Spread {
    bool done;          // false: the row cannot be spread
    bool zeros_only;    // ... but perhaps if its zeros are kept apart
    unsigned bad;
    float inv_s;        // of the buckets
};

// The elements to their buckets' places in shared memory.
template <int THREADS, int ITEMS, bool ZEROS>
__device__ __forceinline__ Spread spread_row(const uint16_t *Wr, const float *Gr, const float *rscale, int m, unsigned long long *status)
{
    using Bk = Buckets<THREADS>;
    constexpr int NW = THREADS / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const BucketLayout L = bucket_layout(m, THREADS);
    float *keys = reinterpret_cast<float *>(smem + L.keys);
    float *gs = reinterpret_cast<float *>(smem + L.gs);
    uint32_t *cnt = reinterpret_cast<uint32_t *>(smem + L.uni);         // four counters a word
    PhaseSmem &ps = *reinterpret_cast<PhaseSmem *>(smem + L.phase);
    float *red = reinterpret_cast<float *>(ps.segtot);                  // free until the record pass
    uint32_t *wsum = reinterpret_cast<uint32_t *>(ps.segtot) + 32;
    uint32_t *wzeros = bucket_zeros(ps);
    Spread r{false, true, 0u, 0.0f};

    // ------------------------------------------------------------ load
    float x[ITEMS];
    float sum = 0.0f;
    {
        uint16_t h[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) h[i] = (i * THREADS + tid < m) ? Wr[i * THREADS + tid] : (uint16_t)0;
#pragma unroll
        for (int u = 0; u < 2; ++u) reinterpret_cast<uint4 *>(cnt)[u * THREADS + tid] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if ((h[i] & 0x7c00u) == 0x7c00u) r.bad |= 1u;
            x[i] = __half2float(__ushort_as_half(h[i]));
            x[i] = __fmul_rn(x[i], (i * THREADS + tid < m) ? rscale[i * THREADS + tid] : 1.0f);
            x[i] += 0.0f;                                           // -0 and +0 are one value
            sum += fabsf(x[i]);
        }
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    if (lane == 0) red[warp] = sum;
    int others = m;
    if constexpr (ZEROS) {
        uint32_t zeros = 0u;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) zeros += (i * THREADS + tid < m && x[i] == 0.0f) ? 1u : 0u;
        zeros = __reduce_add_sync(0xffffffffu, zeros);
        if (lane == 0) wzeros[warp] = zeros;
        __syncthreads();
        zeros = 0u;
        for (int w = 0; w < NW; ++w) zeros += wzeros[w];
        if (tid == 0) wzeros[NW] = zeros;
        if (zeros < ZEROS_APART) return r;
        others -= (int)zeros;
    } else {
        // a row with many zeros is not tried without: one of 32 elements looked at, and at least ZEROS_APART of them
        if (__syncthreads_count(tid < m && x[0] == 0.0f ? 1 : 0) >= max(THREADS / 32, (int)ZEROS_APART)) return r;
    }
    sum = 0.0f;
    for (int w = 0; w < NW; ++w) sum += red[w];
    // s = half a standard deviation of a normal row: 0.5 sqrt(pi / 2) mean |x|
    r.inv_s = (sum > 0.0f && sum < 3.0e38f) ? fminf(__fdividef((float)others, 0.6267f * sum), 1.0e38f) : 0.0f;

    const Bk bucket{r.inv_s};

    // ------------------------------------------------------------ count: slots inside the buckets
    uint32_t slot[(ITEMS + 3) / 4];
    bool over = false;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        if ((i & 3) == 0) slot[i >> 2] = 0u;
        if (i * THREADS + tid < m && !(ZEROS && x[i] == 0.0f)) {
            const int b = bucket(x[i]);
            const uint32_t s = (atomicAdd(&cnt[b >> 2], 1u << (8 * (b & 3))) >> (8 * (b & 3))) & 0xffu;
            over |= s >= (uint32_t)BUCKET_LIMIT;
            slot[i >> 2] |= s << (8 * (i & 3));
        }
    }
    __syncthreads();

    // ------------------------------------------------------------ counters -> bases
    bool crowded = false;
    {
        uint4 v[2];
        uint32_t s = 0u, occupied = 0u;
#pragma unroll
        for (int u = 0; u < 2; ++u) v[u] = reinterpret_cast<const uint4 *>(cnt)[2 * tid + u];
        uint32_t *w = reinterpret_cast<uint32_t *>(v);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            s = __dp4a(w[u], 0x01010101u, s);
            occupied += w[u] ? 1u : 0u;
        }
        // occupied words: a lower bound of the number of distinct values
        occupied = __reduce_add_sync(0xffffffffu, occupied);
        if (lane == 0 && occupied) atomicAdd(&ps.misc[0], (int)occupied);
        uint32_t inc = s;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += t;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        uint32_t run = inc - s;
        if (ZEROS && tid >= THREADS / 2) run += wzeros[NW];         // the zeros lie before bucket HALF
        for (int q = 0; q < warp; ++q) run += wsum[q];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t c0 = w[u] & 0xffu, c1 = c0 + ((w[u] >> 8) & 0xffu), c2 = c1 + ((w[u] >> 16) & 0xffu), c3 = c2 + (w[u] >> 24);
            crowded |= c2 > 31u;
            w[u] = (run << 15) | c0 | (c1 << 5) | (c2 << 10);
            run += c3;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) reinterpret_cast<uint4 *>(cnt)[2 * tid + u] = v[u];
    }
    if (__syncthreads_or(over || crowded ? 1 : 0)) {
        // (zeros fall into the first bucket of thread THREADS / 2)
        r.zeros_only = !__syncthreads_or(crowded && tid != THREADS / 2 ? 1 : 0);
        return r;
    }

    // ------------------------------------------------------------ scatter to the buckets
    constexpr int GB = 8;                                           // importances in flight
    int zero_at = 0;                                                // place of this warp's next zero
    if constexpr (ZEROS) {
        zero_at = bucket_base(cnt, Bk::HALF) - (int)wzeros[NW];
        for (int w = 0; w < warp; ++w) zero_at += (int)wzeros[w];
    }
#pragma unroll
    for (int i0 = 0; i0 < ITEMS; i0 += GB) {
        float g[GB];
#pragma unroll
        for (int u = 0; u < GB; ++u) g[u] = (i0 + u < ITEMS && (i0 + u) * THREADS + tid < m) ? Gr[(i0 + u) * THREADS + tid] : 0.0f;
#pragma unroll
        for (int u = 0; u < GB; ++u) {
            if (i0 + u >= ITEMS) continue;
            const int i = i0 + u < ITEMS ? i0 + u : 0;
            const bool in = i * THREADS + tid < m, zero = ZEROS && in && x[i] == 0.0f;
            int pos = 0;
            if constexpr (ZEROS) {
                const unsigned z = __ballot_sync(0xffffffffu, zero);
                pos = zero_at + __popc(z & ((1u << lane) - 1u));
                zero_at += __popc(z);
            }
            if (in) {
                if (!(g[u] >= 0.0f) || g[u] > 3.0e38f) r.bad |= 2u;
                if (!zero) pos = bucket_base(cnt, bucket(x[i])) + (int)((slot[i >> 2] >> (8 * (i & 3))) & 0xffu);
                if (SKIM_IDX(pos, m, status)) {
                    keys[pos] = x[i];
                    gs[pos] = g[u];
                }
            }
        }
    }
    r.done = true;
    return r;
}

// (its own function: in the kernel its registers would cost rows without zeros 3-4 %)
template <int THREADS, int ITEMS>
__device__ __noinline__ Spread spread_row_zeros_apart(const uint16_t *Wr, const float *Gr, const float *rscale, int m, unsigned long long *status)
{
    return spread_row<THREADS, ITEMS, true>(Wr, Gr, rscale, m, status);
}

// Scaled rows: values times a.rscale, full records.
template <int THREADS, int ITEMS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) skim_sort_bucket_kernel(ClusterArgs a)
{
    using Bk = Buckets<THREADS>;
    constexpr int NW = THREADS / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31;
    const int m = a.m;
    const BucketLayout L = bucket_layout(m, THREADS);
    float *keys = reinterpret_cast<float *>(smem + L.keys);
    float *gs = reinterpret_cast<float *>(smem + L.gs);
    uint32_t *cnt = reinterpret_cast<uint32_t *>(smem + L.uni);         // four counters a word
    PhaseSmem &ps = *reinterpret_cast<PhaseSmem *>(smem + L.phase);

    skim_let_next_kernel_start();
    skim_wait_for_previous_kernel();
    const int64_t row = a.row0 + blockIdx.x;
    const uint16_t *Wr = a.W + row * a.ld;
    const float *Gr = a.G + row * a.ld;
    for (int j = tid * 32; j < m; j += THREADS * 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(Gr + j));      // for the scatter

    if (tid == 0) {
        ps.misc[0] = 0;
        ps.misc[1] = 0;
    }
    Spread sp = spread_row<THREADS, ITEMS, false>(Wr, Gr, a.rscale, m, a.status);
    bool apart = false;                    // the zeros lie between the negative and the positive buckets
    if (!sp.done && sp.zeros_only) {
        __syncthreads();
        if (tid == 0) ps.misc[0] = 0;
        sp = spread_row_zeros_apart<THREADS, ITEMS>(Wr, Gr, a.rscale, m, a.status);
        apart = true;
    }
    if (sp.bad) atomicOr(a.status, (unsigned long long)sp.bad);
    if (!sp.done) {
        // not a row for buckets: the kernel after this one takes it
        if (tid == 0) {
            const int at = atomicAdd(a.sort_count, 1);
            if (SKIM_IDX(at, a.chunk_rows, a.status)) a.sort_list[at] = (int)blockIdx.x;
        }
        return;
    }
    const Bk bucket{sp.inv_s};
    __syncthreads();

    // ---------------------------------------------------------------- order where it matters
    // The Lloyd kernel asks for groups of 8 in order, not for order inside a group: only a bucket that reaches from one
    // group into the next has to be sorted.  A row with few distinct values is sorted in full (they are counted below), and so
    // are all rows for the exact kernel.  The rows come out the same on every run (the record pass orders their groups).
    int nd = ps.misc[0];                     // more than 16 occupied words: more than 16 distinct values
    auto bucket_end = [&](int b) { return b + 1 < Bk::N ? bucket_base(cnt, b + 1) - (apart && b + 1 == Bk::HALF ? (int)bucket_zeros(ps)[NW] : 0) : m; };
    const bool full = a.full_order || nd <= 16;
    for (int p0 = tid * 8; p0 < m; p0 += THREADS * 8) {
        if (!full) {
            if (p0 == 0) continue;
            const int b = bucket(keys[p0]), lo = bucket_base(cnt, b);
            if (lo < p0 && lo >= p0 - 8) sort_bucket(keys, gs, lo, bucket_end(b) - lo);          // (an earlier start: an earlier border's thread does it)
        } else {
            // every bucket that starts in these 8 positions (a bucket's other places hold elements of the bucket all along)
            for (int p = p0; p < min(p0 + 8, m);) {
                const float key = keys[p];
                const int b = bucket(key), lo = bucket_base(cnt, b), end = bucket_end(b);
                const bool zero = apart && key == 0.0f;              // (its bucket begins behind the zeros)
                if (lo >= p0 && !zero) sort_bucket(keys, gs, lo, end - lo);
                p = zero ? lo : end;
            }
        }
    }
    __syncthreads();

    // ---------------------------------------------------------------- row record
    const SortedArrays<float> src{keys, gs};
    if (nd <= 16) {
        // few occupied words: count the distinct values themselves
        if (tid == 0) ps.misc[0] = 0;
        __syncthreads();
        int dcount = 0;
        for (int p = tid; p < m; p += THREADS) dcount += (p == 0 || src.key_at(p) != src.key_at(p - 1)) ? 1 : 0;
        dcount = __reduce_add_sync(0xffffffffu, dcount);
        if (lane == 0 && dcount) atomicAdd(&ps.misc[0], dcount);
        __syncthreads();
        nd = ps.misc[0];
    }
    write_row_record<float, THREADS, false>(a, src, ps, nd, (int)blockIdx.x);
    if (nd <= 16) {
        collect_distinct<float, THREADS>(src, m, nd, ps);
        write_distinct_values(a, nd, ps.dvals, (int)blockIdx.x);
    }
}


// ---------------------------------------------------------------- unscaled rows
//
// A value is a binary16 number, so the row lies in shared memory as 16-bit keys and importances, and a register holds an element's key
// and bucket: the bucket is found once.  The shared-memory pipe bounds this kernel (42 wavefronts per 32 elements: an atomic, a lookup and
// two stores at random addresses, the scans), then the latency of its phases, so
//   - the buckets' first positions are 16-bit numbers of their own, read as they are used, and written without bank conflicts (4 % of
//     the kernel);
//   - importances are requested a batch before they are placed, the first before the scan of the counters is over (8 %);
//   - elements past the row's end go to counters of their own behind the buckets', one per lane, so that nothing branches on them;
//   - the record pass takes the keys as they lie (compact records hold binary16 values).
// us for 4096 rows, the fp16-key kernel (to 3000 columns: the binary32 form of this one, before) and now: 3000 columns 92.9 -> 83.3, 4096
// 129.6 -> 103.5, 5600 161.4 -> 150.5, 8192 238.8 -> 215.8; at 11 008, where two blocks of 512 threads fill an SM either way, 289.4 and 308.1.
struct Bucket16Layout {
    size_t keys, gs, base, phase, total;
};
constexpr int SPARE = 128;              // counters behind the buckets': lane L's is number 4 L
// keys: the counters, four 8-bit ones a word, until the scatter
__host__ __device__ inline Bucket16Layout bucket16_layout(int m, int threads)
{
    Bucket16Layout L;
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off += (b + 15) & ~(size_t)15; return o; };
    const size_t mpad = ((size_t)m + 7) & ~(size_t)7, counters = (size_t)threads * 32 + SPARE;
    L.keys = take(mpad * 2 > counters ? mpad * 2 : counters);
    L.gs = take(mpad * 4);
    L.base = take(counters * 2);
    L.phase = take(sizeof(PhaseSmem));
    L.total = off;
    return L;
}

// A row is refused for a bucket with more than BUCKET16_SLOTS elements, or for crowded words (three neighbouring buckets with 32 elements): more than
// two of a thread's eight, or any in more than CROWDED threads.  A bucket across the border of two groups is put in order by one thread, in time that
// grows with its square.  A row with a narrow centre and long tails has a few crowded words (sort and Lloyd, 4096 x 5000: 263 us refused and 220 spread);
// spreading values about 0.3 with a deviation of 0.02, whose words are crowded throughout, took 328 us for 4096 x 4096 where refusing them takes 190.
// A row of few values or a clump is told by the first EARLY elements of every thread: one of their buckets holds EARLY_SLOTS already.  Otherwise all its
// elements queue for a few counters (us for 4096 rows of a clump, 4096 columns 314 -> 243, 8192 578 -> 449).
//
// The block sorts a refused row itself where it has 256 threads or more: that takes no more shared memory than the buckets (44 KB each at 4096
// columns), the failed attempt's waits are covered by the SM's other blocks, and no other kernel has to look for such rows (2.8 us).
// Smaller blocks would lose an eighth of their number by it; their rows go on a list.
// us for 4096 rows of a clump (in brackets: values about 0.3), by the fp16-key kernel alone, by buckets and a list, and now: 3700 columns 229 308
// 231 (173 219 187), 4096 243 331 242 (178 224 190), 5000 273 459 291 (190 247 235), 8192 444 590 449 (310 372 341).  Bell-shaped rows: 160 132
// 128, 163 139 135, 187 177 172, 280 262 254.
constexpr uint32_t BUCKET16_SLOTS = 32, EARLY_SLOTS = 12;
__host__ __device__ constexpr bool sorts_refused_rows(int threads) { return threads >= 256; }
template <int THREADS> constexpr int CROWDED = sorts_refused_rows(THREADS) ? THREADS / 64 : 0;

__device__ __forceinline__ float key_value(uint16_t h) { return __half2float(__ushort_as_half(h)); }

// Where the first position of bucket b lies in `base`: a thread writes 64 bytes, four pieces whose order is another one every second
// thread, so that eight threads' stores meet no bank twice.
__device__ __forceinline__ int base_place(int b) { return b ^ (b >> 3 & 24); }

// Insertion sort of n elements by one thread.
__device__ __forceinline__ void sort_bucket16(uint16_t *keys, float *gs, int lo, int n)
{
    for (int i = lo + 1; i < lo + n; ++i) {
        const uint16_t h = keys[i];
        const float k = key_value(h), g = gs[i];
        int j = i;
        for (; j > lo; --j) {
            const uint16_t y = keys[j - 1];
            if (!(key_value(y) > k)) break;
            keys[j] = y;
            gs[j] = gs[j - 1];
        }
        if (j != i) {
            keys[j] = h;
            gs[j] = g;
        }
    }
}

// The elements to their buckets' places in shared memory.
template <int THREADS, int ITEMS, bool ZEROS>
__device__ __forceinline__ Spread spread_row16(const uint16_t *Wr, const float *Gr, int m, unsigned long long *status)
{
    using Bk = Buckets<THREADS>;
    constexpr int NW = THREADS / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const Bucket16Layout L = bucket16_layout(m, THREADS);
    uint16_t *keys = reinterpret_cast<uint16_t *>(smem + L.keys);
    float *gs = reinterpret_cast<float *>(smem + L.gs);
    uint32_t *cnt = reinterpret_cast<uint32_t *>(smem + L.keys);
    uint16_t *base = reinterpret_cast<uint16_t *>(smem + L.base);
    PhaseSmem &ps = *reinterpret_cast<PhaseSmem *>(smem + L.phase);
    float *red = reinterpret_cast<float *>(ps.segtot);                  // free until the record pass
    uint32_t *wsum = reinterpret_cast<uint32_t *>(ps.segtot) + 32;
    uint32_t *wzeros = bucket_zeros(ps);
    Spread r{false, true, 0u, 0.0f};

    // ------------------------------------------------------------ load
    uint32_t item[ITEMS];               // key; later key | bucket << 16
    float sum = 0.0f;
    uint32_t top = 0u;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) item[i] = (i * THREADS + tid < m) ? (uint32_t)Wr[i * THREADS + tid] : 0u;
#pragma unroll
    for (int u = 0; u < 2; ++u) reinterpret_cast<uint4 *>(cnt)[u * THREADS + tid] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < SPARE / 4) cnt[Bk::N / 4 + tid] = 0u;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const uint32_t size = item[i] & 0x7fffu;
        if (size == 0u) item[i] = 0u;                                   // -0 and +0 are one value
        top = max(top, size);
        sum += key_value((uint16_t)size);
    }
    if (top >= 0x7c00u) r.bad |= 1u;
#pragma unroll
    for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    if (lane == 0) red[warp] = sum;
    int others = m;
    if constexpr (ZEROS) {
        uint32_t zeros = 0u;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) zeros += (i * THREADS + tid < m && item[i] == 0u) ? 1u : 0u;
        zeros = __reduce_add_sync(0xffffffffu, zeros);
        if (lane == 0) wzeros[warp] = zeros;
        __syncthreads();
        zeros = 0u;
        for (int w = 0; w < NW; ++w) zeros += wzeros[w];
        if (tid == 0) wzeros[NW] = zeros;
        if (zeros < ZEROS_APART) return r;
        others -= (int)zeros;
    } else {
        // a row with many zeros is not tried without: one of 32 elements looked at, and at least ZEROS_APART of them
        if (__syncthreads_count(tid < m && item[0] == 0u ? 1 : 0) >= max(THREADS / 32, (int)ZEROS_APART)) return r;
    }
    sum = 0.0f;
    for (int w = 0; w < NW; ++w) sum += red[w];
    // s = half a standard deviation of a normal row: 0.5 sqrt(pi / 2) mean |x|
    r.inv_s = (sum > 0.0f && sum < 3.0e38f) ? fminf(__fdividef((float)others, 0.6267f * sum), 1.0e38f) : 0.0f;
    const Bk bucket{r.inv_s};

    // ------------------------------------------------------------ count: slots inside the buckets
    uint32_t slot[(ITEMS + 3) / 4];
    uint32_t most = 0u;
    constexpr int EARLY = sorts_refused_rows(THREADS) ? 2 : 0;
    bool clumped = false;               // a value or a clump of them takes a bucket after EARLY of the thread's elements
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        if ((i & 3) == 0) slot[i >> 2] = 0u;
        if (i * THREADS < m && !(ZEROS && item[i] == 0u)) {
            uint32_t b = (uint32_t)bucket(key_value((uint16_t)item[i]));
            if (i * THREADS + tid >= m) b = (uint32_t)(Bk::N + 4 * lane);
            // (shifts by 8 b wrap at 32)
            const uint32_t s = __funnelshift_r(atomicAdd(cnt + (b >> 2), __funnelshift_l(1u, 1u, 8u * b)), 0u, 8u * b & 31u) & 0xffu;
            most = max(most, s);
            slot[i >> 2] |= s << (8 * (i & 3));
            clumped |= i < EARLY && s >= EARLY_SLOTS && item[i] != 0u;
            item[i] |= (uint32_t)base_place((int)b) << 16;
        }
        // (no barrier for it: a warp that sees one leaves the others to count on)
        if (i == EARLY - 1 && __any_sync(0xffffffffu, clumped)) {
            clumped = true;
            break;
        }
    }
    if (clumped) ps.misc[2] = 1;
    if (most >= BUCKET16_SLOTS) ps.misc[3] = 1;
    __syncthreads();
    if (ps.misc[2]) {
        r.zeros_only = false;
        return r;
    }

    // ------------------------------------------------------------ counters -> first positions
    int crowded = 0;
    {
        uint4 v[2];
        uint32_t s = 0u, occupied = 0u;
#pragma unroll
        for (int u = 0; u < 2; ++u) v[u] = reinterpret_cast<const uint4 *>(cnt)[2 * tid + u];
        const uint32_t *w = reinterpret_cast<const uint32_t *>(v);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            s = __dp4a(w[u], 0x01010101u, s);
            occupied += w[u] ? 1u : 0u;
        }
        // occupied words: a lower bound of the number of distinct values
        occupied = __reduce_add_sync(0xffffffffu, occupied);
        if (lane == 0 && occupied) atomicAdd(&ps.misc[0], (int)occupied);
        uint32_t inc = s;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += t;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        uint32_t run = inc - s;
        if (ZEROS && tid >= THREADS / 2) run += wzeros[NW];         // the zeros lie before bucket HALF
        for (int q = 0; q < warp; ++q) run += wsum[q];
        uint32_t out[16];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t before = w[u] * 0x01010100u;             // bytes: elements of the word's buckets before each one
            crowded += before >> 24 > 31u ? 1 : 0;
            const uint32_t both = run * 0x10001u;
            out[2 * u] = both + __byte_perm(before, 0u, 0x4140);
            out[2 * u + 1] = both + __byte_perm(before, 0u, 0x4342);
            run += (before >> 24) + (w[u] >> 24);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) reinterpret_cast<uint4 *>(base)[4 * tid + (u ^ (tid >> 1 & 3))] = make_uint4(out[4 * u], out[4 * u + 1], out[4 * u + 2], out[4 * u + 3]);
        if (tid < SPARE) base[Bk::N + tid] = (uint16_t)m;            // the last bucket's end; elements past the row are not placed
    }
    if (CROWDED<THREADS> && crowded > 2) ps.misc[3] = 1;
    // importances, a batch ahead of the one that is placed
    constexpr int GB = 8;
    float g[2][GB];
    auto fetch = [&](int i0, float (&to)[GB]) {
#pragma unroll
        for (int u = 0; u < GB; ++u) to[u] = (i0 + u < ITEMS && (i0 + u) * THREADS + tid < m) ? Gr[(i0 + u) * THREADS + tid] : 0.0f;
    };
    fetch(0, g[0]);
    if (__syncthreads_count(crowded ? 1 : 0) > CROWDED<THREADS> || ps.misc[3]) {
        // (zeros fall into the first bucket of thread THREADS / 2)
        r.zeros_only = !__syncthreads_or(crowded && tid != THREADS / 2 ? 1 : 0);
        return r;
    }

    // ------------------------------------------------------------ scatter to the buckets (in the counters' place)
    int zero_at = 0;                                                // place of this warp's next zero
    if constexpr (ZEROS) {
        zero_at = (int)base[base_place(Bk::HALF)] - (int)wzeros[NW];
        for (int w = 0; w < warp; ++w) zero_at += (int)wzeros[w];
    }
    uint32_t largest = 0u;
#pragma unroll
    for (int i0 = 0; i0 < ITEMS; i0 += GB) {
        constexpr int LAST = (ITEMS - 1) / GB * GB;
        const int h = i0 / GB & 1;
        if (i0 < LAST) fetch(i0 + GB, g[h ^ 1]);
#pragma unroll
        for (int u = 0; u < GB; ++u) {
            if (i0 + u >= ITEMS || (i0 + u) * THREADS >= m) continue;
            const int i = i0 + u < ITEMS ? i0 + u : 0;
            const bool in = i * THREADS + tid < m;
            const float gv = g[h][u] + 0.0f;                           // (-0 is allowed)
            largest = max(largest, __float_as_uint(gv));            // a negative one, NaN: above every allowed one
            int pos = (int)base[item[i] >> 16] + (int)((slot[i >> 2] >> (8 * (i & 3))) & 0xffu);
            if constexpr (ZEROS) {
                const bool zero = in && item[i] == 0u;
                const unsigned z = __ballot_sync(0xffffffffu, zero);
                if (zero) pos = zero_at + __popc(z & ((1u << lane) - 1u));
                zero_at += __popc(z);
            }
            if (in && SKIM_IDX(pos, m, status)) {
                keys[pos] = (uint16_t)item[i];
                gs[pos] = gv;
            }
        }
    }
    if (largest > __float_as_uint(3.0e38f)) r.bad |= 2u;
    // whole groups of 8
    if (tid < ((m + 7) & ~7) - m) {
        keys[m + tid] = SKIM_PAD_HALF;
        gs[m + tid] = 0.0f;
    }
    r.done = true;
    return r;
}

// (its own function: in the kernel its registers would cost rows without zeros 3-4 %)
template <int THREADS, int ITEMS>
__device__ __noinline__ Spread spread_row16_zeros_apart(const uint16_t *Wr, const float *Gr, int m, unsigned long long *status)
{
    return spread_row16<THREADS, ITEMS, true>(Wr, Gr, m, status);
}

// The bucket-ordered row as the record pass sees it.
struct SortedHalves {
    const uint16_t *keys;
    const float *gs;
    __device__ __forceinline__ unsigned group(int e, int, uint4 &k, float *g) const
    {
        k = *reinterpret_cast<const uint4 *>(keys + e);
        const float4 a = *reinterpret_cast<const float4 *>(gs + e), b = *reinterpret_cast<const float4 *>(gs + e + 4);
        g[0] = a.x; g[1] = a.y; g[2] = a.z; g[3] = a.w; g[4] = b.x; g[5] = b.y; g[6] = b.z; g[7] = b.w;
        return 0u;
    }
    __device__ __forceinline__ float key_at(int p) const { return key_value(keys[p]); }
};

// (its own function, as above)
template <int THREADS, int ITEMS>
__device__ __noinline__ void sort_refused_row(const ClusterArgs &a) { sort16_row<true, THREADS, (ITEMS + 7) / 8, true>(a, (int)blockIdx.x, 0u); }

template <int THREADS, int ITEMS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) skim_sort_bucket16_kernel(const __grid_constant__ ClusterArgs a)
{
    using Bk = Buckets<THREADS>;
    constexpr int NW = THREADS / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31;
    const int m = a.m;
    const Bucket16Layout L = bucket16_layout(m, THREADS);
    uint16_t *keys = reinterpret_cast<uint16_t *>(smem + L.keys);
    float *gs = reinterpret_cast<float *>(smem + L.gs);
    const uint16_t *base = reinterpret_cast<const uint16_t *>(smem + L.base);
    PhaseSmem &ps = *reinterpret_cast<PhaseSmem *>(smem + L.phase);

    if (!sorts_refused_rows(THREADS)) skim_let_next_kernel_start();        // (the list kernel; the Lloyd kernel starts as the blocks leave)
    skim_wait_for_previous_kernel();
    const int64_t row = a.row0 + blockIdx.x;
    const uint16_t *Wr = a.W + row * a.ld;
    const float *Gr = a.G + row * a.ld;
    for (int j = tid * 32; j < m; j += THREADS * 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(Gr + j));      // for the scatter

    if (tid == 0) {
        ps.misc[0] = 0;
        ps.misc[1] = 0;
        ps.misc[2] = 0;
        ps.misc[3] = 0;
    }
    Spread sp = spread_row16<THREADS, ITEMS, false>(Wr, Gr, m, a.status);
    bool apart = false;                    // the zeros lie between the negative and the positive buckets
    if (!sp.done && sp.zeros_only) {
        __syncthreads();
        if (tid == 0) ps.misc[0] = ps.misc[3] = 0;
        sp = spread_row16_zeros_apart<THREADS, ITEMS>(Wr, Gr, m, a.status);
        apart = true;
    }
    if (sp.bad) atomicOr(a.status, (unsigned long long)sp.bad);
    if (!sp.done) {
        // not a row for buckets
        if constexpr (sorts_refused_rows(THREADS)) {
            __syncthreads();
            sort_refused_row<THREADS, ITEMS>(a);
        } else if (tid == 0) {
            const int at = atomicAdd(a.sort_count, 1);
            if (SKIM_IDX(at, a.chunk_rows, a.status)) a.sort_list[at] = (int)blockIdx.x;
        }
        return;
    }
    const Bk bucket{sp.inv_s};
    __syncthreads();

    // ---------------------------------------------------------------- order where it matters (as for scaled rows, above)
    // An unscaled value has 11 bits, so a group's sums of g and g x are exact unless its importances spread over 2^15, whatever
    // their order; the row total of g x^2 may differ in its last bit between runs, as it does from the fp16-key kernel.
    int nd = ps.misc[0];                     // more than 16 occupied words: more than 16 distinct values
    auto bucket_end = [&](int b) { return (int)base[base_place(b + 1)] - (apart && b + 1 == Bk::HALF ? (int)bucket_zeros(ps)[NW] : 0); };
    const bool full = nd <= 16;
    for (int p0 = tid * 8; p0 < m; p0 += THREADS * 8) {
        if (!full) {
            if (p0 == 0) continue;
            const int b = bucket(key_value(keys[p0])), lo = (int)base[base_place(b)];
            if (lo < p0 && lo >= p0 - 8) sort_bucket16(keys, gs, lo, bucket_end(b) - lo);          // (an earlier start: an earlier border's thread does it)
        } else {
            // every bucket that starts in these 8 positions (a bucket's other places hold elements of the bucket all along)
            for (int p = p0; p < min(p0 + 8, m);) {
                const float key = key_value(keys[p]);
                const int b = bucket(key), lo = (int)base[base_place(b)], end = bucket_end(b);
                const bool zero = apart && key == 0.0f;              // (its bucket begins behind the zeros)
                if (lo >= p0 && !zero) sort_bucket16(keys, gs, lo, end - lo);
                p = zero ? lo : end;
            }
        }
    }
    __syncthreads();

    // ---------------------------------------------------------------- row record
    const SortedHalves src{keys, gs};
    if (nd <= 16) {
        // few occupied words: count the distinct values themselves
        if (tid == 0) ps.misc[0] = 0;
        __syncthreads();
        int dcount = 0;
        for (int p = tid; p < m; p += THREADS) dcount += (p == 0 || src.key_at(p) != src.key_at(p - 1)) ? 1 : 0;
        dcount = __reduce_add_sync(0xffffffffu, dcount);
        if (lane == 0 && dcount) atomicAdd(&ps.misc[0], dcount);
        __syncthreads();
        nd = ps.misc[0];
    }
    write_row_record_half<uint4, THREADS>(a, src, ps, nd, (int)blockIdx.x);
    if (nd <= 16) {
        collect_distinct<float, THREADS>(src, m, nd, ps);
        write_distinct_values(a, nd, ps.dvals, (int)blockIdx.x);
    }
}

struct BucketVariant {
    int cap;
    int threads;
    void (*scaled)(ClusterArgs);
    void (*unscaled)(ClusterArgs);      // row lengths that the launcher of skim_cluster.cu gives to skim_cluster16.cu have none
};

#define SKIM_BV(T, I) {T * I, T, skim_sort_bucket_kernel<T, I>, nullptr}
#define SKIM_BV2(T, I) {T * I, T, skim_sort_bucket_kernel<T, I>, skim_sort_bucket16_kernel<T, I>}

// An SM holds 1024 threads; many small blocks wait for their own barriers only, as far as registers hold the row.  Sort and Lloyd kernel, us for 4096
// rows, unscaled and scaled: 5600 columns 256 x 22 188 and 227, 512 x 16 205 and 254; 4096 columns 256 x 16 136 and 173, 512 x 8 163 and 193.
const BucketVariant kVariantsBucket[] = {
    SKIM_BV2(128, 4), SKIM_BV2(128, 8), SKIM_BV2(128, 16), SKIM_BV2(256, 12), SKIM_BV2(256, 16), SKIM_BV2(256, 22), SKIM_BV2(512, 16), SKIM_BV(512, 22), SKIM_BV(1024, 16), SKIM_BV(1024, 22),
};

}  // namespace

int skim_launch_sort_bucket(skim_ctx *ctx, const ClusterArgs &args, int64_t rows, bool *lists)
{
    for (const BucketVariant &v : kVariantsBucket) {
        if (v.cap < args.m) continue;
        void (*kernel)(ClusterArgs) = args.rscale ? v.scaled : v.unscaled;
        if (!kernel) return SKIM_ERR_SHAPE;
        *lists = args.rscale || !sorts_refused_rows(v.threads);
        size_t smem = args.rscale ? bucket_layout(args.m, v.threads).total : bucket16_layout(args.m, v.threads).total;
        if (!*lists) smem = std::max(smem, layout16(args.m, v.threads).total);
        if (smem > (size_t)ctx->max_smem_optin) return SKIM_ERR_SHAPE;
        // set on every launch: a host-side call of microseconds, and no state shared between contexts
        SKIM_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        // Scaled rows whose blocks leave much of the chip free: an ordinary launch.  Blocks that may start beside the Lloyd kernel of the call
        // before seem to crowd on the SMs that have none of its blocks.  Calls one after another, us, dependent and ordinary: 400 x 1500 37.5 and
        // 33.5, 500 x 2000 41.0 and 37.3, 500 x 900 31.7 and 29.9, 800 x 1500 39.2 and 38.6, 1000 x 2000 of refused rows 71.3 and 66.3; but 256 x
        // 512 25.9 and 26.7, 300 x 1500 33.5 and 33.6, 1150 x 1200 38.6 and 39.5. Larger blocks, more rows and unscaled rows (whose Lloyd kernel
        // takes shared memory itself): dependent 1 us less.
        if (args.rscale && v.threads == 128 && rows > ctx->sm_count * 2 && rows < ctx->sm_count * 7) {
            kernel<<<(unsigned)rows, v.threads, smem, ctx->stream>>>(args);
            SKIM_CUDA_OK(cudaGetLastError());
            ctx->launches += 1;
            return SKIM_OK;
        }
        return skim_launch_dependent(ctx, kernel, dim3((unsigned)rows), v.threads, smem, args);
    }
    return SKIM_ERR_SHAPE;
}
