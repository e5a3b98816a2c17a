// Greedy bit allocation (SKIM Section 4.2, Algorithm 1) as one selection problem.
//
// Algorithm 1 raises, K times, the row whose next bit removes the most error.  Give step t of
// row i the key q(i,t) = min over u <= t of the row's u-th error reduction (a running minimum,
// so keys never increase along a row).  The sequential greedy takes exactly the first K items in
// the order (q descending, row ascending, t ascending): a row's later, larger reduction becomes
// available only once the smaller one before it has been taken, and is then taken at once.
// The kernel finds the K-th key by splitting the range of the live keys (order-preserving 64-bit images of q) into 2048
// equal parts, as often as it takes to leave a few hundred, which are ranked directly; ties at the threshold are
// resolved by row-major rank.  One block: the work is latency, and the fewer passes the better -- an 8-bit radix select,
// whose first digits are the same for all keys, took eight (4096 rows: 20.5 us; 22 016 rows: 108 us).
#include "skim_internal.cuh"
#include "skim_key_range.h"

namespace {

constexpr int AT = 1024;  // threads of the single block
constexpr int BINS = 1 << SkimKeyRange::PART_BITS;
static_assert(BINS == 2 * AT, "a thread has two bins");
constexpr int LIST_CAP = 512;    // live keys that are ranked directly

__device__ __forceinline__ unsigned long long ordered_bits(double v)
{
    if (v == 0.0) v = 0.0;  // -0 and +0 compare equal
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

// keys of one row: q[t] for t = 0 .. nb-2 (entries beyond stay 0); ld floats between rows of the table.  vec: the row is
// one aligned 16-byte load
__device__ __forceinline__ void row_keys(const float *err, int64_t i, int ld, int nb, bool vec, unsigned long long *q)
{
    float e[SKIM_MAX_NBITS];
    if (vec) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(err) + i);
        e[0] = v.x; e[1] = v.y; e[2] = v.z; e[3] = v.w;
    } else {
#pragma unroll
        for (int t = 0; t < SKIM_MAX_NBITS; ++t) e[t] = t < nb ? __ldg(err + i * ld + t) : 0.0f;
    }
    double run = 0.0;
#pragma unroll
    for (int t = 0; t < SKIM_MAX_NBITS - 1; ++t) {
        q[t] = 0ull;
        if (t + 1 < nb) {
            const double gain = (double)e[t] - (double)e[t + 1];
            run = (t == 0 || gain < run) ? gain : run;
            q[t] = ordered_bits(run);
        }
    }
}

// Rows are dealt to threads so that a warp reads consecutive rows: warp w owns the rows
// [w * rounds * 32, (w + 1) * rounds * 32), lane l takes row j * 32 + l of that range in round j.
// CACHE_ROWS > 0: every thread keeps the keys of its (at most CACHE_ROWS) rows in registers for all
// passes; CACHE_ROWS == 0: keys are recomputed from the table in every pass.
template <int CACHE_ROWS>
__global__ void __launch_bounds__(AT) skim_allocate_kernel(const float *__restrict__ err, int64_t n, int ld, int nb,
                                                            int bmin, long long K, uint8_t *__restrict__ bits)
{
    constexpr int STEPS_MAX = SKIM_MAX_NBITS - 1;
    constexpr int NC = CACHE_ROWS > 0 ? CACHE_ROWS : 1;
    __shared__ unsigned int hist[BINS];
    __shared__ SkimKeyRange s_range;             // of the live keys
    __shared__ long long s_need;                 // the wanted key is the s_need-th largest of them
    __shared__ unsigned int s_live;
    __shared__ long long wsum[AT / 32];
    __shared__ unsigned long long list[LIST_CAP];
    __shared__ unsigned int s_count;             // entries of the list
    __shared__ unsigned long long s_thr;
    __shared__ long long s_take;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int steps = nb - 1;
    const bool vec = nb == SKIM_MAX_NBITS && ld == nb && (reinterpret_cast<uintptr_t>(err) & 15u) == 0;
    skim_wait_for_previous_kernel();
    skim_let_next_kernel_start();

    if (K <= 0 || steps <= 0) {
        for (int64_t i = tid; i < n; i += AT) bits[i] = (uint8_t)bmin;
        return;
    }
    const int rounds = (int)((n + AT - 1) / AT);
    const int64_t row_base = (int64_t)warp * rounds * 32 + lane;

    unsigned long long cache[NC][STEPS_MAX];
    if (CACHE_ROWS > 0) {
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            const int64_t i = row_base + (int64_t)j * 32;
            unsigned long long q[SKIM_MAX_NBITS] = {0ull, 0ull, 0ull, 0ull};
            if (j < rounds && i < n) row_keys(err, i, ld, nb, vec, q);
#pragma unroll
            for (int t = 0; t < STEPS_MAX; ++t) cache[j][t] = q[t];
        }
    }
    // keys of this thread's row of round j (valid only when the row exists)
    auto keys_of = [&](int j, int64_t i, unsigned long long *q) {
        if (CACHE_ROWS > 0) {
#pragma unroll
            for (int jj = 0; jj < NC; ++jj)
                if (jj == j) {
#pragma unroll
                    for (int t = 0; t < STEPS_MAX; ++t) q[t] = cache[jj][t];
                }
        } else {
            row_keys(err, i, ld, nb, vec, q);
        }
    };

    // visits every key of the thread's rows
    auto each_key = [&](auto &&f) {
#pragma unroll (CACHE_ROWS > 0 ? NC : 1)
        for (int j = 0; j < (CACHE_ROWS > 0 ? NC : rounds); ++j) {
            if (CACHE_ROWS > 0 && j >= rounds) break;
            const int64_t i = row_base + (int64_t)j * 32;
            if (i < n) {
                unsigned long long q[SKIM_MAX_NBITS];
                keys_of(j, i, q);
#pragma unroll
                for (int t = 0; t < STEPS_MAX; ++t)
                    if (t < steps) f(q[t]);
            }
        }
    };

    // ---- the range of the keys
    unsigned long long lo = ~0ull, hi = 0ull;
    each_key([&](unsigned long long key) { lo = min(lo, key); hi = max(hi, key); });
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, off));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, off));
    }
    if (lane == 0) { list[2 * warp] = lo; list[2 * warp + 1] = hi; }
    for (int d = tid; d < BINS; d += AT) hist[d] = 0u;
    __syncthreads();
    if (warp == 0) {
        lo = list[2 * lane];
        hi = list[2 * lane + 1];
#pragma unroll
        for (int off = 16; off; off >>= 1) {
            lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, off));
            hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, off));
        }
        if (lane == 0) { s_range.lo = lo; s_range.hi = hi; s_need = K; s_live = (unsigned)min((long long)n * steps, 0xffffffffll); s_count = 0u; }
    }
    __syncthreads();

    // ---- narrow the range down to the part that holds the K-th largest key
    while (s_live > (unsigned)LIST_CAP && s_range.lo < s_range.hi) {
        const SkimKeyRange range = s_range;
        const int shift = range.shift();
        each_key([&](unsigned long long key) {
            if (range.holds(key)) atomicAdd(&hist[range.part_of(key, shift)], 1u);
        });
        __syncthreads();
        // suffix counts: thread t has bins 2t and 2t + 1
        const unsigned c0 = hist[2 * tid], c1 = hist[2 * tid + 1];
        hist[2 * tid] = 0u;
        hist[2 * tid + 1] = 0u;
        unsigned inc = c0 + c1;                                 // this thread's and the higher lanes'
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned v = __shfl_down_sync(0xffffffffu, inc, off);
            if (lane + off < 32) inc += v;
        }
        if (lane == 0) wsum[warp] = (long long)inc;
        __syncthreads();
        long long above = (long long)inc - (c0 + c1);           // keys in higher bins
        for (int w = warp + 1; w < AT / 32; ++w) above += wsum[w];
        const long long need = s_need;
        __syncthreads();
        if (above < need && need <= above + c1 + c0) {
            const bool upper = need <= above + c1;
            s_need = upper ? need - above : need - above - c1;
            s_live = upper ? c1 : c0;
            s_range = range.part(2u * tid + (upper ? 1u : 0u), shift);
        }
        __syncthreads();
    }
    if (s_range.lo == s_range.hi) {
        // one value is left: all live keys equal it
        if (tid == 0) { s_thr = s_range.lo; s_take = s_need; }
    } else {
        const SkimKeyRange range = s_range;
        each_key([&](unsigned long long key) {
            if (range.holds(key)) {
                const unsigned at = atomicAdd(&s_count, 1u);
                if (at < (unsigned)LIST_CAP) list[at] = key;      // (there are s_live <= LIST_CAP of them)
            }
        });
        __syncthreads();
        const unsigned cnt = min(s_count, (unsigned)LIST_CAP);
        if ((unsigned)tid < cnt) {
            const unsigned long long key = list[tid];
            unsigned greater = 0u, equal = 0u;
            for (unsigned x = 0; x < cnt; ++x) {
                greater += list[x] > key ? 1u : 0u;
                equal += list[x] == key ? 1u : 0u;
            }
            // (several threads with equal keys write the same)
            if ((long long)greater < s_need && s_need <= (long long)(greater + equal)) { s_thr = key; s_take = s_need - greater; }
        }
    }
    __syncthreads();
    const unsigned long long thr = s_thr;      // the K-th largest key
    const long long take_eq = s_take;          // how many items equal to it are taken, in row-major order

    // items equal to the threshold are taken in row-major order: count them per warp, ...
    unsigned eq_all = 0u;
#pragma unroll (CACHE_ROWS > 0 ? NC : 1)
    for (int j = 0; j < (CACHE_ROWS > 0 ? NC : rounds); ++j) {
        if (CACHE_ROWS > 0 && j >= rounds) break;
        const int64_t i = row_base + (int64_t)j * 32;
        if (i < n) {
            unsigned long long q[SKIM_MAX_NBITS];
            keys_of(j, i, q);
#pragma unroll
            for (int t = 0; t < STEPS_MAX; ++t) eq_all += (t < steps && q[t] == thr) ? 1u : 0u;
        }
    }
    const unsigned warp_eq = __reduce_add_sync(0xffffffffu, eq_all);
    if (lane == 0) wsum[warp] = (long long)warp_eq;
    __syncthreads();
    long long carry = 0;                       // equal items in rows before this warp's current round
    for (int w = 0; w < warp; ++w) carry += wsum[w];

    // ... then rank them round by round with a warp prefix sum (rows of a round ascend with the lane)
#pragma unroll (CACHE_ROWS > 0 ? NC : 1)
    for (int j = 0; j < (CACHE_ROWS > 0 ? NC : rounds); ++j) {
        if (CACHE_ROWS > 0 && j >= rounds) break;
        const int64_t i = row_base + (int64_t)j * 32;
        const bool row_ok = i < n;
        unsigned long long q[SKIM_MAX_NBITS];
        if (row_ok) keys_of(j, i, q);
        unsigned eq = 0u;
#pragma unroll
        for (int t = 0; t < STEPS_MAX; ++t) eq += (row_ok && t < steps && q[t] == thr) ? 1u : 0u;
        unsigned inc = eq;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned v = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += v;
        }
        long long before = carry + (long long)(inc - eq);
        carry += (long long)__shfl_sync(0xffffffffu, inc, 31);
        if (row_ok) {
            int extra = 0;
#pragma unroll
            for (int t = 0; t < STEPS_MAX; ++t) {
                if (t < steps) {
                    if (q[t] > thr) {
                        ++extra;
                    } else if (q[t] == thr) {
                        if (before < take_eq) ++extra;
                        ++before;
                    }
                }
            }
            bits[i] = (uint8_t)(bmin + extra);
        }
    }
}

// Exact allocation (the dynamic programme Section 4.2 mentions as the precise but quadratic solution):
// f_i(s) = min_u f_{i-1}(s - u) + E[i-1][u] over s = bits handed out beyond b_min, smallest u on ties; one
// block walks the rows, its threads share the states; the choices are kept to walk back from s = K.
__global__ void __launch_bounds__(AT) skim_allocate_optimal_kernel(const float *__restrict__ err, int64_t n, int nb,
                                                                    int bmin, long long K, double *fa, double *fb,
                                                                    uint8_t *choice, uint8_t *__restrict__ bits,
                                                                    double *cost)
{
    const int tid = threadIdx.x;
    const double INF = __longlong_as_double(0x7ff0000000000000ll);
    for (long long s = tid; s <= K; s += AT) { fa[s] = INF; fb[s] = INF; }
    __syncthreads();
    if (tid == 0) fa[0] = 0.0;
    __syncthreads();
    double *prev = fa, *cur = fb;
    for (int64_t i = 0; i < n; ++i) {
        double e[SKIM_MAX_NBITS];
#pragma unroll
        for (int u = 0; u < SKIM_MAX_NBITS; ++u) e[u] = u < nb ? (double)__ldg(err + i * nb + u) : 0.0;
        const long long top = min(K, (long long)(i + 1) * (nb - 1));     // states beyond are unreachable (and stay infinite)
        uint8_t *ch = choice + (size_t)i * (size_t)(K + 1);
        for (long long s = tid; s <= top; s += AT) {
            double best = INF;
            int bu = 0;
#pragma unroll
            for (int u = 0; u < SKIM_MAX_NBITS; ++u) {
                if (u < nb && u <= s) {
                    const double v = prev[s - u] + e[u];
                    if (v < best) { best = v; bu = u; }
                }
            }
            cur[s] = best;
            ch[s] = (uint8_t)bu;
        }
        __syncthreads();
        double *t = prev; prev = cur; cur = t;
    }
    if (tid == 0) {
        if (cost) *cost = prev[K];
        long long s = K;
        for (int64_t i = n - 1; i >= 0; --i) {
            // s <= (i + 1)(nb - 1) here, so its choice has been written.  Where every way to s costs infinitely much no choice was
            // better than 0: the rows before take at most i (nb - 1), so that s stays a state that they have
            const long long least = s - i * (nb - 1);
            long long u = choice[(size_t)i * (size_t)(K + 1) + (size_t)s];
            if (u < least) u = least;
            bits[i] = (uint8_t)(bmin + u);
            s -= u;
        }
    }
}

}  // namespace

size_t skim_allocate_optimal_scratch(int64_t rows, int64_t K)
{
    const size_t f = skim_align256((size_t)(K + 1) * sizeof(double));
    return 2 * f + skim_align256((size_t)rows * (size_t)(K + 1));
}

int skim_launch_allocate_optimal(skim_ctx *ctx, const float *err, int64_t rows, const SkimBits &bits, int64_t K,
                                 void *scratch, uint8_t *out_bits, double *cost)
{
    const size_t f = skim_align256((size_t)(K + 1) * sizeof(double));
    unsigned char *p = (unsigned char *)scratch;
    skim_allocate_optimal_kernel<<<1, AT, 0, ctx->stream>>>(err, rows, bits.n_bits, bits.b_min, (long long)K, (double *)p,
                                                           (double *)(p + f), p + 2 * f, out_bits, cost);
    SKIM_CUDA_OK(cudaGetLastError());
    ctx->launches += 1;
    return SKIM_OK;
}

int skim_launch_allocate(skim_ctx *ctx, const float *err, int64_t rows, const SkimBits &bits, int first_col, int64_t K,
                         uint8_t *out_bits)
{
    // the greedy runs on the columns first_col .. n_bits-1 of the table: every row starts at b_min + first_col
    const int ld = bits.n_bits, nb = bits.n_bits - first_col, start = bits.b_min + first_col;
    return skim_launch_dependent(ctx, rows <= 4 * AT ? skim_allocate_kernel<4> : skim_allocate_kernel<0>, dim3(1), AT, 0, err + first_col, rows, ld, nb,
                                 start, (long long)K, out_bits);
}
