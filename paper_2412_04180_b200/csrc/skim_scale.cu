// Scaling-vector training with the labels held fixed (SKIM Section 4.3, Algorithm 2, inner
// repeat; optimiser settings of Section 5.1).
//
//   loss(alpha) = sum_ij g_ij (W_ij - alpha_j c_{i,l_ij})^2,
//   c_ik        = sum_{j in k} g_ij W_ij / alpha_j  /  sum_{j in k} g_ij   (re-fitted each step)
//
// Once per call skim_scale_order_kernel writes every row in label order.  Per Adam step the matrix is then read twice:
//   skim_scale_sums_kernel  one warp per row, on the label-ordered copy.  Per cluster k of the row it forms, in binary64,
//       S_k = sum g w / alpha,  A_k = sum g w alpha,  B_k = sum g alpha^2  (sums over the members).
//       With the per-call constants G_k = sum g and D_k = sum g w^2 (the same kernel, run once in
//       its INIT form) these give the centroid c_k = S_k / G_k, the row's loss
//       sum_k D_k - 2 c_k A_k + c_k^2 B_k, and the factor q_k = 2 (A_k - c_k B_k) / G_k through which the
//       re-fitted centroid enters the gradient -- without a second pass over the row.  No atomics: every sum has a
//       fixed order.
//   skim_scale_grad_kernel  a thread owns four columns and walks a range of rows:
//       d loss / d alpha_j = sum_i  -2 g c (w - alpha_j c) + q g w / alpha_j^2   (c, q of the element's
//       cluster, from the 256-byte table the first kernel left for the row), accumulated in
//       registers; the row ranges leave partial gradients that the Adam kernel adds in a fixed order.
// Every kernel of a step is a programmatic dependent of the one before it: it starts while that one drains and fetches
// what no kernel of the loop writes (the matrix) before it waits.
//   skim_scale_adam_kernel  sums the partials and the rows' losses (deterministic), applies the
//       Adam update to the binary64 master copy of alpha.
#include "skim_internal.cuh"

namespace {

constexpr int KC = 16;      // clusters per row at most (4 bits)
constexpr int GT = 256;     // threads of a gradient block
constexpr int GC = 4;       // columns per thread

struct ScaleArgs {
    const uint16_t *W;
    const float *G;
    const uint8_t *labels;
    const double *alpha;
    int64_t rows, ld;
    int cols;
    int vec;                // rows of W, G and labels allow the vector loads of both kernels
    uint2 *ord;             // [rows][skim_ordered_stride(cols)]  the matrix in label order
    uint16_t *ord_end;      // [rows][KC]  units of the clusters up to and including each
    double2 *tconst;        // [rows][KC]  (G_k, D_k)
    double2 *tq;            // [rows][KC]  (c_k, q_k)
    double *loss_row;       // [rows]
    double *grad_part;      // [row ranges][cols]
    uint16_t *D;            // L-full loss: [rows][cols] binary16 residual * 2^exp2
    int exp2;
    int rows_per_range;
    int grad_warps;         // warps of a gradient block side by side over the columns; its other warps take other rows
};

// 1 / a for a positive, normal binary64 a (the scale vector is checked to be that): the hardware's approximate
// reciprocal (better than 20 bits, error e) and one step of the series 1 + e + e^2, within one unit in the last place.  Four
// instructions where the correctly rounded division-free reciprocal takes about twelve; the sums kernel needs one per element.
__device__ __forceinline__ double rcp_pos(double a)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
    const double e = fma(-a, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// ---------------------------------------------------------------- the label-ordered copy of the matrix
//
// Labels are fixed during a call, so every row is put in label order once: element = (importance, weight, column) in
// 8 bytes, the members of a cluster padded to whole units of 64.  The sums of a unit then belong to one cluster and
// stay in registers (in column order every element costs three binary64 read-modify-writes of an accumulator slot in
// shared memory, 96 wavefronts of the L1 data path per 256 elements, which bound the kernel), and the price is one
// gather of alpha from shared memory per element.  Inside a cluster the elements are dealt by column modulo 16, the
// bank pair of alpha's entry, so that the 16 lanes of a half-warp mostly hit 16 different bank pairs: the i-th
// elements of all 16 classes come first for i = 0, then for i = 1, and so on.
constexpr int OT = 512;                    // threads per block of the ordering kernel
constexpr int OW = OT / 32;
constexpr int OB = 6;                      // chunks of 32 columns whose loads a warp has in flight
constexpr int UNIT = SKIM_ORDER_UNIT;
static_assert(UNIT == 64 && KC == 16 && OW == KC, "a lane takes two elements of a unit; the ordering kernel has a warp per label");

// entries of the ordering kernel's place tables: sum over the labels of the largest class, about cols / 12 when
// columns and labels are unrelated; rows that need more take the slow branch
__host__ __device__ __forceinline__ int order_table_entries(int cols) { return cols / 6 + 256; }

__host__ __device__ __forceinline__ size_t order_smem_bytes(int cols)
{
    return (size_t)skim_ordered_stride(cols) * sizeof(uint2) + (size_t)OW * KC * 32 * sizeof(uint16_t) + KC * 16 * sizeof(uint16_t) +
           (size_t)order_table_entries(cols) * 4 + (3 * KC + 1) * sizeof(int);
}

// Of the 16 classes' counts (packed in tw): how many elements come before element i of class `cls`, i.e. the first
// min(count, i) of every class and the i-th of the classes before it.
__device__ __forceinline__ int order_place(const uint16_t *tot, uint32_t i, int cls)
{
    int before = 0;
    for (int c = 0; c < 16; ++c) before += min((int)tot[c], (int)i) + ((c < cls && tot[c] > i) ? 1 : 0);
    return before;
}

__global__ void __launch_bounds__(OT) skim_scale_order_kernel(ScaleArgs a)
{
    extern __shared__ __align__(16) unsigned char osmem[];
    uint2 *row_out = reinterpret_cast<uint2 *>(osmem);                                              // the ordered row
    uint16_t *cnt = reinterpret_cast<uint16_t *>(row_out + skim_ordered_stride(a.cols));           // [OW][KC][32] per lane and label
    uint16_t *tot = cnt + OW * KC * 32;                                                              // [KC][16] per label and class
    uint32_t *table = reinterpret_cast<uint32_t *>(tot + KC * 16);                                   // per label and i: elements before | classes with an i-th
    int *base = reinterpret_cast<int *>(table + order_table_entries(a.cols));                        // [KC] first element of a label
    int *members = base + KC;                                                                        // [KC]
    int *tbase = members + KC;                                                                       // [KC] its table; [KC] all units
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t row = blockIdx.x;
    const uint16_t *Wr = a.W + row * a.ld;
    const float *Gr = a.G + row * a.ld;
    const uint8_t *Lr = a.labels + row * (int64_t)a.cols;
    uint16_t *mine = cnt + warp * KC * 32 + lane;                                                    // entry l at mine[l * 32]
#pragma unroll
    for (int l = 0; l < KC; ++l) mine[l * 32] = 0;
    __syncwarp();
    // a warp takes 32 consecutive columns at a time, so a lane's columns are all of class lane % 16
    const int chunks = (a.cols + 31) / 32;
    for (int c0 = warp; c0 < chunks; c0 += OW * OB) {
        int l[OB];
#pragma unroll
        for (int u = 0; u < OB; ++u) l[u] = Lr[min((c0 + u * OW) * 32 + lane, a.cols - 1)] & (KC - 1);
#pragma unroll
        for (int u = 0; u < OB; ++u)
            if ((c0 + u * OW) * 32 + lane < a.cols) mine[l[u] * 32] += 1;
    }
    __syncthreads();
    // thread (label, class): the counts of the class's 2 OW lanes become exclusive prefixes
    if (tid < KC * 16) {
        const int l = tid >> 4, cls = tid & 15;
        int run = 0;
        for (int w = 0; w < OW; ++w)
            for (int h = 0; h < 2; ++h) {
                uint16_t *p = cnt + (w * KC + l) * 32 + h * 16 + cls;
                const int v = *p;
                *p = (uint16_t)run;
                run += v;
            }
        tot[tid] = (uint16_t)run;
    }
    __syncthreads();
    if (warp == 0) {
        // units of every label, where its elements start, and where its place table does
        int n = 0, most = 0;
        if (lane < KC)
            for (int c = 0; c < 16; ++c) {
                n += tot[lane * 16 + c];
                most = max(most, (int)tot[lane * 16 + c]);
            }
        const int units = (n + UNIT - 1) / UNIT;
        int inc = units, tinc = most;
#pragma unroll
        for (int off = 1; off < KC; off <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, off), tt = __shfl_up_sync(0xffffffffu, tinc, off);
            if (lane >= off) { inc += t; tinc += tt; }
        }
        if (lane < KC) {
            base[lane] = (inc - units) * UNIT;
            members[lane] = n;
            tbase[lane] = tinc <= order_table_entries(a.cols) ? tinc - most : -1;      // -1: no room, the slow branch
            a.ord_end[row * KC + lane] = (uint16_t)inc;
        }
        if (lane == KC - 1) tbase[KC] = inc;
    }
    __syncthreads();
    const int total = tbase[KC] * UNIT;
    // slot of position p: the two 32-element halves of a unit are interleaved, so that a lane's two elements are one
    // 16-byte load and the warp's first (second) elements are 32 consecutive positions
    auto slot = [](int p) { return (p & ~(UNIT - 1)) + 2 * (p & 31) + ((p >> 5) & 1); };
    {
        // warp l: the padding behind label l's elements, and its place table
        const int l = warp, n = members[l];
        for (int q = n + lane; q < (n + UNIT - 1) / UNIT * UNIT; q += 32) row_out[slot(base[l] + q)] = make_uint2(0u, 0u);
        if (tbase[l] >= 0) {
            int most = lane < 16 ? (int)tot[l * 16 + lane] : 0;
            const int own = most;
            most = __reduce_max_sync(0xffffffffu, most);
            int run = 0;
            for (int i0 = 0; i0 < most; i0 += 32) {
                uint32_t have = 0u;
#pragma unroll
                for (int c = 0; c < 16; ++c) have |= (__shfl_sync(0xffffffffu, own, c) > i0 + lane ? 1u : 0u) << c;
                const int pc = __popc(have);
                int inc = pc;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, inc, off);
                    if (lane >= off) inc += t;
                }
                if (i0 + lane < most) table[tbase[l] + i0 + lane] = ((uint32_t)(run + inc - pc) << 16) | have;
                run += __shfl_sync(0xffffffffu, inc, 31);
            }
        }
    }
    __syncthreads();
    const uint32_t below = (1u << (lane & 15)) - 1u;           // classes before mine
    for (int c0 = warp; c0 < chunks; c0 += OW * OB) {
        int l[OB];
        uint32_t w[OB];
        float g[OB];
#pragma unroll
        for (int u = 0; u < OB; ++u) {
            const int j = min((c0 + u * OW) * 32 + lane, a.cols - 1);
            l[u] = Lr[j] & (KC - 1);
            w[u] = Wr[j];
            g[u] = Gr[j];
        }
#pragma unroll
        for (int u = 0; u < OB; ++u) {
            const int j = (c0 + u * OW) * 32 + lane;
            if (j < a.cols) {
                const uint32_t i = mine[l[u] * 32];
                mine[l[u] * 32] = (uint16_t)(i + 1);
                const int tb = tbase[l[u]];
                int place;
                if (tb >= 0) {
                    const uint32_t e = table[tb + i];
                    place = (int)(e >> 16) + __popc(e & below);
                } else {
                    place = order_place(tot + l[u] * 16, i, lane & 15);
                }
                const int pos = slot(base[l[u]] + place);
                if (SKIM_IDX(pos, total, nullptr)) row_out[pos] = make_uint2(__float_as_uint(g[u]), (w[u] << 16) | (uint32_t)j);
            }
        }
    }
    __syncthreads();
    uint4 *dst = reinterpret_cast<uint4 *>(a.ord + row * skim_ordered_stride(a.cols));
    const uint4 *src = reinterpret_cast<const uint4 *>(row_out);
    for (int q = tid; q < total / 2; q += OT) dst[q] = src[q];
}

// Short rows: padding to whole units and the reductions at every cluster's end would cost more than the elements do (22016 x 128:
// 8 clusters of 16 elements padded to 64 each).  Such rows are written without padding, by one warp each, in column order inside a
// cluster; ord_end counts elements.  Whole step, before and after: 22016 x 128 85 -> 49 us, 9000 x 300 43 -> 28.5 us; at 4096 x 1500 36.6 -> 43.6 us,
// since the longest cluster decides.  Up to 1024 columns it pays where every warp of the sums kernel has a row of its own (4096 x 700 28.4 ->
// 26.1 us, ordering 9000 x 1000 170 -> 100 us; 1000 x 1001 16.9 -> 19.0 us).
constexpr int SHORT_COLS = SKIM_ORDER_SHORT_COLS, SHORT_COLS_MANY_ROWS = 1024;
constexpr int OST = 256;

__global__ void __launch_bounds__(OST) skim_scale_order_short_kernel(ScaleArgs a)
{
    __shared__ int count_all[OST / 32][2 * KC];
    const int lane = threadIdx.x & 31;
    int *count = count_all[threadIdx.x >> 5];                  // entry KC: columns past the end
    const int64_t row = (int64_t)blockIdx.x * (OST / 32) + (threadIdx.x >> 5);
    if (row >= a.rows) return;                                 // (whole warps; no block-wide barrier follows)
    const uint16_t *Wr = a.W + row * a.ld;
    const float *Gr = a.G + row * a.ld;
    const uint8_t *Lr = a.labels + row * (int64_t)a.cols;
    uint2 *dst = a.ord + row * skim_ordered_stride(a.cols);
    count[lane] = 0;
    __syncwarp();
    for (int j0 = 0; j0 < a.cols; j0 += 32) {
        const int l = j0 + lane < a.cols ? (int)(Lr[j0 + lane] & (KC - 1)) : KC;
        const uint32_t same = __match_any_sync(0xffffffffu, l);
        if ((same & ((1u << lane) - 1u)) == 0u) count[l] += __popc(same);
        __syncwarp();
    }
    const int n = count[lane & (KC - 1)];
    int inc = n;
#pragma unroll
    for (int off = 1; off < KC; off <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, off, KC);
        if ((lane & (KC - 1)) >= off) inc += t;
    }
    __syncwarp();
    if (lane < KC) {
        a.ord_end[row * KC + lane] = (uint16_t)inc;
        count[lane] = inc - n;
    }
    __syncwarp();
    for (int j0 = 0; j0 < a.cols; j0 += 32) {
        const int j = j0 + lane;
        const bool in = j < a.cols;
        const int l = in ? (int)(Lr[j] & (KC - 1)) : KC;
        const uint32_t w = in ? (uint32_t)Wr[j] : 0u;
        const float g = in ? Gr[j] : 0.0f;
        const uint32_t same = __match_any_sync(0xffffffffu, l), below = same & ((1u << lane) - 1u);
        const int pos = count[l] + __popc(below);
        __syncwarp();
        if (below == 0u) count[l] += __popc(same);
        if (in && SKIM_IDX(pos, a.cols, nullptr)) dst[pos] = make_uint2(__float_as_uint(g), (w << 16) | (uint32_t)j);
        __syncwarp();
    }
}

// ---------------------------------------------------------------- the sums of a step

constexpr int SUM_T = 768;                 // threads per block of the sums kernel, one block per SM (80 registers)
constexpr int SUM_W = SUM_T / 32;
constexpr int AHEAD = 4;                   // units fetched together; two such batches take turns
static_assert(AHEAD * 3 * UNIT * 8 <= SKIM_ORDER_SLACK, "a warp fetches up to three batches past its last unit");

enum SumsMode { SUMS_INIT, SUMS_STEP, SUMS_CENTROIDS };

// shared memory: alpha (not for INIT), then the warps' partial sums
__host__ __device__ __forceinline__ size_t sums_smem_bytes(int cols, bool init)
{
    return (init ? 0 : ((size_t)cols + 1) / 2 * 16) + (size_t)SUM_W * 2 * 32 * sizeof(double);
}

__device__ __forceinline__ double weight_of(const uint2 &w, int u)
{
    const uint32_t x = u < 2 ? w.x : w.y;
    return (double)__half2float(__ushort_as_half((uint16_t)((u & 1) ? (x >> 16) : (x & 0xffffu))));
}

// The tables of two rows in one register pair: lane L holds entry L % 16 of row `row` + L / 16.
__device__ __forceinline__ double2 table_load(const ScaleArgs &a, int64_t row, int64_t last)
{
    const int lane = threadIdx.x & 31;
    return a.tq[min(row + (lane >> 4), last) * KC + (lane & 15)];
}
// A warp's copy of the tables of a batch of rows in shared memory, c and q apart: 16 entries of 8 bytes lie in 16 different
// bank pairs, so a lookup of either is two wavefronts (16-byte entries took about nine together, four 32-bit shuffles eight).
template <int RB>
struct WarpTables {
    double c[RB * KC], q[RB * KC];
    __device__ __forceinline__ void put(int pair, const double2 &t)
    {
        const int lane = threadIdx.x & 31;
        c[pair * 32 + lane] = t.x;
        q[pair * 32 + lane] = t.y;
    }
};

// The two elements a lane has of a unit, added to its accumulators.
template <int MODE>
__device__ __forceinline__ void add_element(uint32_t gbits, uint32_t wcol, const double *alpha, double (&acc)[3])
{
    const double g = (double)__uint_as_float(gbits);
    const double w = (double)__half2float(__ushort_as_half((uint16_t)(wcol >> 16)));
    const double gw = g * w;
    if (MODE == SUMS_INIT) {
        acc[0] += g;
        acc[1] = fma(gw, w, acc[1]);
    } else {
        const double al = alpha[wcol & 0xffffu];
        acc[0] = fma(gw, rcp_pos(al), acc[0]);
        if (MODE == SUMS_STEP) {
            const double ga = g * al;
            acc[1] = fma(ga, w, acc[1]);
            acc[2] = fma(ga, al, acc[2]);
        }
    }
}

// One row's share of one warp: units [t0, t1) of its label-ordered elements.  The sums of cluster k come back in
// lanes k (sum 0) and 16 + k (sum 1) of vx, and in lane k of vb (sum 2).
template <int MODE>
__device__ __forceinline__ void sum_units(const uint4 *src, int end, int t0, int t1, const double *alpha, double &vx, double &vb)
{
    const int lane = threadIdx.x & 31;
    double acc[3] = {0.0, 0.0, 0.0};
    vx = 0.0;
    vb = 0.0;
    int k = 0;
    while (k < KC - 1 && __shfl_sync(0xffffffffu, end, k) <= t0) ++k;
    int stop = min(__shfl_sync(0xffffffffu, end, k), t1);
    src += (int64_t)t0 * (UNIT / 2) + lane;
    uint4 buf[2][AHEAD];
#pragma unroll
    for (int u = 0; u < AHEAD; ++u) buf[0][u] = __ldcs(src + u * (UNIT / 2));
    // Batches of AHEAD units take turns in two register buffers; the reads past the last unit stay inside the
    // ordered matrix and its slack, and are not used.
    for (int t = t0; t < t1; t += 2 * AHEAD) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int u = 0; u < AHEAD; ++u) buf[h ^ 1][u] = __ldcs(src + ((h + 1) * AHEAD + u) * (UNIT / 2));
#pragma unroll
            for (int u = 0; u < AHEAD; ++u) {
                if (t + h * AHEAD + u < t1) {
                    add_element<MODE>(buf[h][u].x, buf[h][u].y, alpha, acc);
                    add_element<MODE>(buf[h][u].z, buf[h][u].w, alpha, acc);
                    if (t + h * AHEAD + u + 1 == stop) {
                        // the cluster (or the share) ends here: sum 0 goes to the lower half-warp, sum 1 to the upper
                        double x = lane < 16 ? acc[0] : acc[1];
                        if (MODE != SUMS_CENTROIDS) x += __shfl_xor_sync(0xffffffffu, lane < 16 ? acc[1] : acc[0], 16);
                        else x = acc[0] + __shfl_xor_sync(0xffffffffu, acc[0], 16);
                        double b = acc[2];
                        if (MODE == SUMS_STEP) b += __shfl_xor_sync(0xffffffffu, b, 16);
#pragma unroll
                        for (int off = 8; off; off >>= 1) {
                            x += __shfl_xor_sync(0xffffffffu, x, off);
                            if (MODE == SUMS_STEP) b += __shfl_xor_sync(0xffffffffu, b, off);
                        }
                        if ((lane & 15) == k) { vx = x; vb = b; }
                        acc[0] = acc[1] = acc[2] = 0.0;
                        const int done = stop;
                        while (k < KC - 1 && __shfl_sync(0xffffffffu, end, k) <= done) ++k;
                        stop = min(__shfl_sync(0xffffffffu, end, k), t1);
                    }
                }
            }
        }
        src += 2 * AHEAD * (UNIT / 2);
    }
}

// The same sums of a short row, all of it: the lanes are dealt to the clusters in equal groups (a power of two of clusters, so
// 2 to 32 lanes each), a lane takes every so-manieth element of its cluster.
template <int MODE>
__device__ __forceinline__ void sum_short(const uint2 *src, int end, const double *alpha, double &vx, double &vb)
{
    constexpr int AT_ONCE = 4;
    const int lane = threadIdx.x & 31;
    const int before = __shfl_up_sync(0xffffffffu, end, 1, KC);
    const uint32_t full = __ballot_sync(0xffffffffu, end > ((lane & (KC - 1)) ? before : 0)) & 0xffffu;
    const int lg = full > 1u ? 32 - __clz(31 - __clz(full)) : 0;       // clusters up to the last one with members: at most 2^lg
    const int sh = 5 - lg, per = 1 << sh, k = lane >> sh;
    const int stop = __shfl_sync(0xffffffffu, end, k);
    const int start = __shfl_sync(0xffffffffu, end, max(k - 1, 0));
    double acc[3] = {0.0, 0.0, 0.0};
    for (int i = (k ? start : 0) + (lane & (per - 1)); i < stop; i += AT_ONCE * per) {
        uint2 v[AT_ONCE];
#pragma unroll
        for (int u = 0; u < AT_ONCE; ++u) v[u] = i + u * per < stop ? src[i + u * per] : make_uint2(0u, 0u);
#pragma unroll
        for (int u = 0; u < AT_ONCE; ++u) add_element<MODE>(v[u].x, v[u].y, alpha, acc);
    }
    __syncwarp();
    for (int off = per >> 1; off; off >>= 1) {
        acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], off);
        if (MODE != SUMS_CENTROIDS) acc[1] += __shfl_xor_sync(0xffffffffu, acc[1], off);
        if (MODE == SUMS_STEP) acc[2] += __shfl_xor_sync(0xffffffffu, acc[2], off);
    }
    const int from = (lane & (KC - 1)) << sh;                          // beyond the last lane: an empty cluster
    const double s0 = __shfl_sync(0xffffffffu, acc[0], from & 31), s1 = __shfl_sync(0xffffffffu, acc[1], from & 31);
    const double s2 = __shfl_sync(0xffffffffu, acc[2], from & 31);
    vx = from < 32 ? (lane < KC ? s0 : s1) : 0.0;
    vb = from < 32 ? s2 : 0.0;
}

// What the sums of a row are turned into (lanes as sum_units leaves them).
//   SUMS_INIT       the per-call constants (G_k, D_k)
//   SUMS_STEP       (c_k, q_k) and the row's loss
//   SUMS_CENTROIDS  (c_k, 0); the kernel then writes the row's residual
template <int MODE>
__device__ __forceinline__ double finish_row(const ScaleArgs &a, int64_t row, double vx, double vb)
{
    const int lane = threadIdx.x & 31;
    const double s1 = __shfl_down_sync(0xffffffffu, vx, 16);
    double loss_k = 0.0, c = 0.0;
    if (lane < KC) {
        if (MODE == SUMS_INIT) {
            a.tconst[row * KC + lane] = make_double2(vx, s1);
        } else {
            const double2 gdk = a.tconst[row * KC + lane];
            double q = 0.0;
            if (gdk.x > 0.0) {
                c = vx / gdk.x;
                if (MODE == SUMS_STEP) {
                    q = 2.0 * (s1 - c * vb) / gdk.x;
                    loss_k = gdk.y - 2.0 * c * s1 + c * c * vb;
                }
            }
            a.tq[row * KC + lane] = make_double2(c, q);
        }
    }
    if (MODE == SUMS_STEP) {
#pragma unroll
        for (int off = 8; off; off >>= 1) loss_k += __shfl_down_sync(0xffffffffu, loss_k, off);
        if (lane == 0) a.loss_row[row] = loss_k;
    }
    return c;
}

// L-full loss: the residual of columns [j0, j1) of a row as the binary16 operand of the contraction; c: the centroid of
// cluster lane % 16.  Four consecutive columns per lane and step.
__device__ __forceinline__ void residual_columns(const ScaleArgs &a, int64_t row, int j0, int j1, const double *alpha, double c)
{
    constexpr int RU = 4;                                     // steps whose loads are in flight
    const int lane = threadIdx.x & 31;
    const float scale = __int_as_float((127 + a.exp2) << 23);
    const uint16_t *Wr = a.W + row * a.ld;
    const uint8_t *Lr = a.labels + row * (int64_t)a.cols;
    uint16_t *Dr = a.D + row * (int64_t)a.cols;
    for (int jb = j0; jb < j1; jb += RU * 128) {
        uint2 w[RU];
        uint32_t l[RU];
#pragma unroll
        for (int u = 0; u < RU; ++u) {
            const int j = min(jb + u * 128 + lane * 4, j1 - 4);
            w[u] = __ldcs(reinterpret_cast<const uint2 *>(Wr + j));
            l[u] = __ldcs(reinterpret_cast<const uint32_t *>(Lr + j));
        }
#pragma unroll
        for (int u = 0; u < RU; ++u) {
            const int j = min(jb + u * 128 + lane * 4, j1 - 4);      // lanes past the end repeat the last columns
            const double2 a0 = *reinterpret_cast<const double2 *>(alpha + j), a1 = *reinterpret_cast<const double2 *>(alpha + j + 2);
            const double al[4] = {a0.x, a0.y, a1.x, a1.y};
            uint32_t h[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const double d = weight_of(w[u], v) - al[v] * __shfl_sync(0xffffffffu, c, (int)((l[u] >> (8 * v)) & (KC - 1)));
                h[v] = __half_as_ushort(__float2half_rn(__fmul_rn((float)d, scale)));
            }
            *reinterpret_cast<uint2 *>(Dr + j) = make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
        }
    }
}

// One block per SM, rows dealt round-robin to the blocks.  A warp takes whole rows while there are rows for all of the
// block's warps; the rows that are left are shared by the warps in equal stretches, whose sums meet in shared memory in a
// fixed order.  Bound by HBM: 8 B an element.
template <int MODE, bool SHORT>
__global__ void __launch_bounds__(SUM_T, 1) skim_scale_sums_kernel(ScaleArgs a)
{
    extern __shared__ __align__(16) double ssmem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double *alpha = ssmem;
    double2 *part = reinterpret_cast<double2 *>(ssmem + (MODE == SUMS_INIT ? 0 : (a.cols + 1) / 2 * 2));     // [SUM_W][32]
    skim_let_next_kernel_start();
    const int64_t stride = skim_ordered_stride(a.cols) / 2;
    const int mine = (int)((a.rows - blockIdx.x + gridDim.x - 1) / gridDim.x);       // rows of this block (at least one)
    const int whole = mine / SUM_W * SUM_W, rest = mine - whole;
    if (MODE != SUMS_INIT && !SHORT) {
        // the start of this warp's first row, while the previous kernel ends
        const int r = whole ? warp : warp / (SUM_W / rest);
        if (r < mine) {
            const uint4 *p = reinterpret_cast<const uint4 *>(a.ord) + (blockIdx.x + (int64_t)gridDim.x * r) * stride;
#pragma unroll
            for (int u = 0; u < 2 * AHEAD; ++u) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + u * (UNIT / 2) + lane));
        }
    }
    skim_wait_for_previous_kernel();
    if (MODE != SUMS_INIT) {
        for (int q = threadIdx.x; q < a.cols / 2; q += SUM_T)
            reinterpret_cast<double2 *>(alpha)[q] = __ldg(reinterpret_cast<const double2 *>(a.alpha) + q);
        if ((a.cols & 1) && threadIdx.x == 0) alpha[a.cols - 1] = a.alpha[a.cols - 1];
        __syncthreads();
    }
    double vx, vb;
    if constexpr (SHORT) {
        int end = warp < mine ? (int)a.ord_end[(blockIdx.x + (int64_t)gridDim.x * warp) * KC + (lane & 15)] : 0;
        for (int r = warp; r < mine; r += SUM_W) {
            const int64_t row = blockIdx.x + (int64_t)gridDim.x * r, next = row + (int64_t)gridDim.x * SUM_W;
            const int ahead = r + SUM_W < mine ? (int)a.ord_end[next * KC + (lane & 15)] : 0;
            sum_short<MODE>(a.ord + row * stride * 2, end, alpha, vx, vb);
            const double c = finish_row<MODE>(a, row, vx, vb);
            if (MODE == SUMS_CENTROIDS) residual_columns(a, row, 0, a.cols, alpha, c);
            end = ahead;
        }
    } else {
        for (int r = warp; r < whole; r += SUM_W) {
            const int64_t row = blockIdx.x + (int64_t)gridDim.x * r;
            const int end = a.ord_end[row * KC + (lane & 15)];
            sum_units<MODE>(reinterpret_cast<const uint4 *>(a.ord) + row * stride, end, 0, __shfl_sync(0xffffffffu, end, KC - 1), alpha, vx, vb);
            const double c = finish_row<MODE>(a, row, vx, vb);
            if (MODE == SUMS_CENTROIDS) residual_columns(a, row, 0, a.cols, alpha, c);
        }
        if (rest == 0) return;
        const int per_row = SUM_W / rest, idx = warp / per_row, sub = warp - idx * per_row;
        const int64_t row = blockIdx.x + (int64_t)gridDim.x * (whole + idx);
        if (idx < rest) {
            const int end = a.ord_end[row * KC + (lane & 15)];
            const int total = __shfl_sync(0xffffffffu, end, KC - 1);
            const int t0 = total * sub / per_row, t1 = total * (sub + 1) / per_row;
            sum_units<MODE>(reinterpret_cast<const uint4 *>(a.ord) + row * stride, end, t0, t1, alpha, vx, vb);
            part[threadIdx.x] = make_double2(vx, vb);
        }
        __syncthreads();
        if (idx < rest && sub == 0) {
            for (int q = 1; q < per_row; ++q) {
                const double2 o = part[threadIdx.x + 32 * q];
                vx += o.x;
                vb += o.y;
            }
            const double c = finish_row<MODE>(a, row, vx, vb);
            if (MODE == SUMS_CENTROIDS) part[threadIdx.x].x = c;
        }
        if (MODE == SUMS_CENTROIDS) {
            // the row's columns are shared by the same warps (in fours: cols is a multiple of 8 on this path)
            __syncthreads();
            const int quads = a.cols / 4, q0 = quads * sub / per_row, q1 = quads * (sub + 1) / per_row;
            if (idx < rest && q0 < q1) residual_columns(a, row, q0 * 4, q1 * 4, alpha, part[idx * per_row * 32 + lane].x);
        }
    }
}

// ---------------------------------------------------------------- the gradient of a step
//
// A thread owns four columns and walks a range of rows.  The (c_k, q_k) entry of an element comes from the warp's own copy
// of the rows' tables in shared memory; warps do not wait for one another.  Two blocks are resident
// per SM and the grid is one wave of them.  HBM traffic: 7 B an element.
template <bool VEC>
struct GradCols {
    int j[VEC ? 1 : GC];          // columns as loaded: clamped to the matrix, so that no load needs a guard
    bool in[VEC ? 1 : GC];
    // VEC: four consecutive columns (cols % 4 == 0: all inside or all outside).  Otherwise four columns a block width
    // apart, so that scalar loads are contiguous across a warp.
    // thread t of the `width` threads that share a tile
    __device__ __forceinline__ GradCols(int tile, int cols, int t, int width)
    {
        if constexpr (VEC) {
            const int c = (tile * width + t) * GC;
            in[0] = c < cols;
            j[0] = min(c, cols - GC);
        } else {
#pragma unroll
            for (int u = 0; u < GC; ++u) {
                const int c = (tile * GC + u) * width + t;
                in[u] = c < cols;
                j[u] = min(c, cols - 1);
            }
        }
    }
    __device__ __forceinline__ int col(int u) const { return VEC ? j[0] + u : j[VEC ? 0 : u]; }
    __device__ __forceinline__ bool inside(int u) const { return in[VEC ? 0 : u]; }
};

// One row's entries at a thread's columns.
struct GradRow {
    uint2 w;
    float4 g;
    uint32_t l;
};

template <bool VEC>
__device__ __forceinline__ void grad_load(const ScaleArgs &a, int64_t row, const GradCols<VEC> &c, GradRow &r)
{
    const uint16_t *Wr = a.W + row * a.ld;
    const float *Gr = a.G + row * a.ld;
    const uint8_t *Lr = a.labels + row * (int64_t)a.cols;
    if constexpr (VEC) {
        r.w = __ldcs(reinterpret_cast<const uint2 *>(Wr + c.j[0]));
        r.g = __ldcs(reinterpret_cast<const float4 *>(Gr + c.j[0]));
        r.l = __ldcs(reinterpret_cast<const uint32_t *>(Lr + c.j[0]));
    } else {
        r.w = make_uint2((uint32_t)__ldcs(Wr + c.j[0]) | ((uint32_t)__ldcs(Wr + c.j[1]) << 16),
                         (uint32_t)__ldcs(Wr + c.j[2]) | ((uint32_t)__ldcs(Wr + c.j[3]) << 16));
        r.g = make_float4(__ldcs(Gr + c.j[0]), __ldcs(Gr + c.j[1]), __ldcs(Gr + c.j[2]), __ldcs(Gr + c.j[3]));
        r.l = (uint32_t)__ldcs(Lr + c.j[0]) | ((uint32_t)__ldcs(Lr + c.j[1]) << 8) | ((uint32_t)__ldcs(Lr + c.j[2]) << 16) |
              ((uint32_t)__ldcs(Lr + c.j[3]) << 24);
    }
}

// NARROW: the block's warps share the rows as well (its own instance: the wide form has no register to spare)
template <bool VEC, bool NARROW>
__global__ void __launch_bounds__(GT, 2) skim_scale_grad_kernel(ScaleArgs a)
{
    __shared__ WarpTables<4> tables[GT / 32];
    WarpTables<4> &tw = tables[threadIdx.x >> 5];
    constexpr int RB = VEC ? 4 : 2;   // rows of a batch (four column addresses leave fewer registers); two batches take turns in registers, one of them in flight
    const int side = NARROW ? a.grad_warps : GT / 32, subs = (GT / 32) / side, sub = NARROW ? (int)(threadIdx.x >> 5) / side : 0;
    const GradCols<VEC> c(blockIdx.x, a.cols, (int)threadIdx.x - sub * side * 32, side * 32);
    const int64_t b0 = (int64_t)blockIdx.y * a.rows_per_range, b1 = min(a.rows, b0 + a.rows_per_range), last = b1 - 1;
    // this warp's share of the block's rows (none for the warps left over)
    const int64_t share = NARROW ? (b1 - b0 + subs - 1) / subs : 0, r0 = NARROW ? min(b1, b0 + sub * share) : b0;
    const int64_t r1 = NARROW ? (sub < subs ? min(b1, r0 + share) : r0) : b1;
    GradRow row[2][RB];
    double2 tab[2][RB / 2];
    auto fetch_rows = [&](int h, int64_t rb) {
#pragma unroll
        for (int q = 0; q < RB; ++q) grad_load<VEC>(a, min(rb + q, last), c, row[h][q]);
    };
    auto fetch_tables = [&](int h, int64_t rb) {
#pragma unroll
        for (int q = 0; q < RB / 2; ++q) tab[h][q] = table_load(a, rb + 2 * q, last);
    };
    skim_let_next_kernel_start();
    fetch_rows(0, r0);
    skim_wait_for_previous_kernel();
    fetch_tables(0, r0);
    double ah[GC], rr[GC], acc[GC];   // alpha / 2, alpha^-2
#pragma unroll
    for (int u = 0; u < GC; ++u) {
        const double al = a.alpha[c.col(u)], r = __drcp_rn(al);
        ah[u] = 0.5 * al;
        rr[u] = r * r;
        acc[u] = 0.0;
    }
    for (int64_t rb = r0; rb < r1; rb += 2 * RB) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            __syncwarp();
#pragma unroll
            for (int q = 0; q < RB / 2; ++q) tw.put(q, tab[h][q]);
            __syncwarp();
            fetch_rows(h ^ 1, rb + (h + 1) * RB);
            fetch_tables(h ^ 1, rb + (h + 1) * RB);
#pragma unroll
            for (int q = 0; q < RB; ++q) {
                if (rb + h * RB + q < r1) {
                    const float g[GC] = {row[h][q].g.x, row[h][q].g.y, row[h][q].g.z, row[h][q].g.w};
#pragma unroll
                    for (int u = 0; u < GC; ++u) {
                        // g (q w / alpha^2 - 2 c (w - alpha c)) with d = 2 c:  g (w (q / alpha^2 - d) + d (d alpha / 2))
                        const int l = q * KC + (int)((row[h][q].l >> (8 * u)) & (KC - 1));
                        const double c = tw.c[l], d = c + c;
                        const double t = fma(weight_of(row[h][q].w, u), fma(tw.q[l], rr[u], -d), d * (d * ah[u]));
                        acc[u] = fma((double)g[u], t, acc[u]);
                    }
                }
            }
        }
    }
    if constexpr (NARROW) {
        // the shares' sums, in the order of the rows
        __shared__ double red[GC][GT];
#pragma unroll
        for (int u = 0; u < GC; ++u) red[u][threadIdx.x] = acc[u];
        __syncthreads();
        if (sub != 0) return;
        for (int q = 1; q < subs; ++q)
#pragma unroll
            for (int u = 0; u < GC; ++u) acc[u] += red[u][threadIdx.x + q * side * 32];
    }
#pragma unroll
    for (int u = 0; u < GC; ++u)
        if (c.inside(u)) a.grad_part[(int64_t)blockIdx.y * a.cols + c.col(u)] = acc[u];
}

__global__ void __launch_bounds__(256) skim_scale_adam_kernel(const double *__restrict__ grad_part,
                                                               const double *__restrict__ loss_row, int nranges,
                                                               int64_t rows, int cols, double *alpha,
                                                               double *m1, double *m2, double lr, double beta1, double beta2,
                                                               double bc1, double bc2, double eps, double *loss_out)
{
    __shared__ double red[256];
    skim_let_next_kernel_start();
    skim_wait_for_previous_kernel();
    if (blockIdx.x == gridDim.x - 1) {
        // the last block adds the rows' losses: strided partial sums, then a fixed tree
        double s = 0.0;
#pragma unroll 8
        for (int64_t i = threadIdx.x; i < rows; i += 256) s += loss_row[i];
        red[threadIdx.x] = s;
        __syncthreads();
        for (int off = 128; off; off >>= 1) {
            if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
            __syncthreads();
        }
        if (threadIdx.x == 0 && loss_out) *loss_out = red[0];
        return;
    }
    // 32 columns a block; the row ranges' partial gradients are dealt to 8 groups of threads, and the groups' sums
    // are added in a fixed order
    const int c = threadIdx.x & 31, sgrp = threadIdx.x >> 5;
    const int j = blockIdx.x * 32 + c;
    double gs = 0.0;
    if (j < cols)
        for (int b = sgrp; b < nranges; b += 8) gs += grad_part[(int64_t)b * cols + j];
    red[threadIdx.x] = gs;
    __syncthreads();
    if (sgrp != 0 || j >= cols) return;
    double g = 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) g += red[q * 32 + c];
    const double a1 = beta1 * m1[j] + (1.0 - beta1) * g;
    const double a2 = beta2 * m2[j] + (1.0 - beta2) * g * g;
    m1[j] = a1;
    m2[j] = a2;
    const double an = alpha[j] - lr * (a1 / bc1) / (sqrt(a2 / bc2) + eps);
    alpha[j] = an;
}

__global__ void skim_scale_init_kernel(const float *__restrict__ alpha32, int cols, double *alpha,
                                       double *m1, double *m2, unsigned long long *status)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= cols) return;
    const float v = alpha32[j];
    if (!(v > 0.0f) || v > 3.0e38f) atomicOr(status, (unsigned long long)SKIM_STATUS_BAD_SCALE);
    alpha[j] = (double)v;
    m1[j] = 0.0;
    m2[j] = 0.0;
}

__global__ void skim_scale_finish_kernel(const double *__restrict__ alpha, int cols, float *__restrict__ alpha32)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < cols) alpha32[j] = (float)alpha[j];
}

// ---------------------------------------------------------------- the same update on the L-full loss
//
//   loss(alpha) = sum_i d_i H d_i^T,  d_ij = W_ij - alpha_j c_{i,l_ij},  H = X X^T   (Section 4.3 with the L-full form of
//   Section 3.4).  With Y = D H:  d loss / d alpha_j = sum_i -2 Y_ij c_{i,l} + q_{i,l} g_ij W_ij / alpha_j^2,
//   q_ik = 2 R_ik / G_ik,  R_ik = sum_{j in k} Y_ij alpha_j.
// Per Adam step: skim_scale_sums_kernel (centroids of the step, and the residual as the binary16 operand of the
// contraction), the tcgen05 GEMM of skim_lfull.cu (Y = D H stored, row-wise dot = the loss, R_ik summed in its epilogue
// and q_ik in its reduction), skim_scale_lf_grad_kernel (column sums), and the Adam kernel above.

// A thread owns four columns and walks a range of rows: sum_i -2 Y_ij c + q g w / alpha_j^2; as skim_scale_grad_kernel
// (cols is a multiple of 8 and the rows are aligned: vector loads always).
__global__ void __launch_bounds__(GT, 2) skim_scale_lf_grad_kernel(ScaleArgs a, const float *Y)
{
    __shared__ WarpTables<2> tables[GT / 32];
    WarpTables<2> &tw = tables[threadIdx.x >> 5];
    constexpr int RB = 2;
    const GradCols<true> c(blockIdx.x, a.cols, (int)threadIdx.x, GT);
    const int64_t r0 = (int64_t)blockIdx.y * a.rows_per_range;
    const int64_t r1 = min(a.rows, r0 + a.rows_per_range), last = r1 - 1;
    const double ys = ldexp(-2.0, -a.exp2);
    skim_let_next_kernel_start();
    skim_wait_for_previous_kernel();
    double rr[GC], acc[GC];
#pragma unroll
    for (int u = 0; u < GC; ++u) {
        const double r = __drcp_rn(a.alpha[c.col(u)]);
        rr[u] = r * r;
        acc[u] = 0.0;
    }
    GradRow row[2][RB];
    float4 yv[2][RB];
    double2 tab[2];
    auto fetch = [&](int h, int64_t rb) {
#pragma unroll
        for (int q = 0; q < RB; ++q) {
            const int64_t i = min(rb + q, last);
            grad_load<true>(a, i, c, row[h][q]);
            yv[h][q] = __ldcs(reinterpret_cast<const float4 *>(Y + i * (int64_t)a.cols + c.j[0]));
        }
        tab[h] = table_load(a, rb, last);
        tab[h].x *= ys;                 // -2 c / 2^exp2
    };
    fetch(0, r0);
    for (int64_t rb = r0; rb < r1; rb += 2 * RB) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            __syncwarp();
            tw.put(0, tab[h]);
            __syncwarp();
            fetch(h ^ 1, rb + (h + 1) * RB);
#pragma unroll
            for (int q = 0; q < RB; ++q) {
                if (rb + h * RB + q < r1) {
                    const float g[GC] = {row[h][q].g.x, row[h][q].g.y, row[h][q].g.z, row[h][q].g.w};
                    const float y[GC] = {yv[h][q].x, yv[h][q].y, yv[h][q].z, yv[h][q].w};
#pragma unroll
                    for (int u = 0; u < GC; ++u) {
                        const int l = q * KC + (int)((row[h][q].l >> (8 * u)) & (KC - 1));
                        acc[u] = fma((double)y[u], tw.c[l], acc[u]);
                        acc[u] = fma((tw.q[l] * rr[u]) * (double)g[u], weight_of(row[h][q].w, u), acc[u]);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int u = 0; u < GC; ++u)
        if (c.inside(u)) a.grad_part[(int64_t)blockIdx.y * a.cols + c.col(u)] = acc[u];
}

}  // namespace

size_t skim_scale_lfull_scratch_bytes(int64_t rows, int64_t cols)
{
    return skim_align256((size_t)rows * cols * 2) + skim_align256((size_t)rows * cols * 4) + skim_lfull_cluster_bytes(rows, cols) +
           skim_lfull_scratch_bytes(rows, cols);
}

namespace {

// What both updates do first: alpha's master copies, the label-ordered matrix, the per-call constants (G_k, D_k).
struct ScalePlan {
    void (*step)(ScaleArgs), (*centroids)(ScaleArgs);      // the sums kernel by row length
    ScaleArgs a;
    unsigned cb, ab;                 // blocks over the columns; Adam: 32 columns a block
    dim3 grad_grid;
    int ranges;
    unsigned sum_blocks;
};

int scale_begin(skim_ctx *ctx, const SkimWorkspace &ws, const uint16_t *W, const float *importance, int64_t rows, int64_t cols,
                int64_t ld, const uint8_t *labels, const float *alpha, ScalePlan *p)
{
    p->cb = (unsigned)((cols + 255) / 256);
    p->ab = (unsigned)((cols + 31) / 32);
    ScaleArgs &a = p->a;
    a.W = W;
    a.G = importance;
    a.labels = labels;
    a.alpha = ws.alpha64;
    a.rows = rows;
    a.ld = ld;
    a.cols = (int)cols;
    a.vec = ((reinterpret_cast<uintptr_t>(W) & 7u) == 0 && (reinterpret_cast<uintptr_t>(importance) & 15u) == 0 &&
             (reinterpret_cast<uintptr_t>(labels) & 3u) == 0 && ld % 4 == 0 && cols % 4 == 0) ? 1 : 0;
    a.ord = reinterpret_cast<uint2 *>(ws.cluster_scratch);
    a.ord_end = ws.scale_ord_end;
    a.tconst = reinterpret_cast<double2 *>(ws.scale_const);
    a.tq = reinterpret_cast<double2 *>(ws.scale_cq);
    a.loss_row = ws.loss_part;
    a.grad_part = ws.grad_part;
    a.D = nullptr;
    a.exp2 = 0;
    // gradient kernels: column tiles x row ranges, one wave of two blocks per SM
    const int tiles = (int)((cols + GT * GC - 1) / (GT * GC));
    int ranges = 2 * ctx->sm_count / tiles;
    if (ranges > SKIM_SCALE_MAX_CTAS) ranges = SKIM_SCALE_MAX_CTAS;
    if (ranges > rows) ranges = (int)rows;
    if (ranges < 1) ranges = 1;
    // warps side by side over the columns: narrow matrices would leave most of a block idle (22016 x 128: 7 warps of 8;
    // a step 49 -> 30 us)
    a.grad_warps = tiles > 1 || cols > GT / 2 * GC ? GT / 32 : (int)((cols + 32 * GC - 1) / (32 * GC));
    a.rows_per_range = (int)((rows + ranges - 1) / ranges);
    p->ranges = (int)((rows + a.rows_per_range - 1) / a.rows_per_range);
    p->grad_grid = dim3((unsigned)tiles, (unsigned)p->ranges);
    // sums kernel: one block per SM
    p->sum_blocks = (unsigned)(rows < ctx->sm_count ? rows : ctx->sm_count);
    // set on every launch: host-side calls of microseconds, and no state shared between contexts
    const int sm_order = (int)order_smem_bytes((int)cols), sm_init = (int)sums_smem_bytes((int)cols, true), sm_sums = (int)sums_smem_bytes((int)cols, false);
    const bool is_short = cols <= SHORT_COLS || (cols <= SHORT_COLS_MANY_ROWS && rows >= (int64_t)SUM_W * ctx->sm_count);
    void (*init)(ScaleArgs) = is_short ? skim_scale_sums_kernel<SUMS_INIT, true> : skim_scale_sums_kernel<SUMS_INIT, false>;
    p->step = is_short ? skim_scale_sums_kernel<SUMS_STEP, true> : skim_scale_sums_kernel<SUMS_STEP, false>;
    p->centroids = is_short ? skim_scale_sums_kernel<SUMS_CENTROIDS, true> : skim_scale_sums_kernel<SUMS_CENTROIDS, false>;
    SKIM_CUDA_OK(cudaFuncSetAttribute(skim_scale_order_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_order));
    SKIM_CUDA_OK(cudaFuncSetAttribute(init, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_init));
    SKIM_CUDA_OK(cudaFuncSetAttribute(p->step, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_sums));
    SKIM_CUDA_OK(cudaFuncSetAttribute(p->centroids, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_sums));
    skim_scale_init_kernel<<<p->cb, 256, 0, ctx->stream>>>(alpha, (int)cols, ws.alpha64, ws.adam_m, ws.adam_v, ws.status);
    SKIM_CUDA_OK(cudaGetLastError());
    if (is_short) skim_scale_order_short_kernel<<<(unsigned)((rows + OST / 32 - 1) / (OST / 32)), OST, 0, ctx->stream>>>(a);
    else skim_scale_order_kernel<<<(unsigned)rows, OT, sm_order, ctx->stream>>>(a);
    SKIM_CUDA_OK(cudaGetLastError());
    init<<<p->sum_blocks, SUM_T, sm_init, ctx->stream>>>(a);
    SKIM_CUDA_OK(cudaGetLastError());
    ctx->launches += 3;
    return SKIM_OK;
}

// The learning rate and bias corrections of the Adam steps (Section 5.1: betas 0.9 / 0.999, eps 1e-8).
struct AdamSchedule {
    double lr, p1 = 1.0, p2 = 1.0, decay;
    int every, t = 0;
    AdamSchedule(float lr0, float d, int e) : lr((double)lr0), decay((double)d), every(e) {}
    void next()
    {
        if (t > 0 && t % every == 0) lr *= decay;
        p1 *= 0.9;
        p2 *= 0.999;
        ++t;
    }
};

int scale_adam(skim_ctx *ctx, const SkimWorkspace &ws, const ScalePlan &p, const AdamSchedule &s, double *loss_trace)
{
    return skim_launch_dependent(ctx, skim_scale_adam_kernel, dim3(p.ab + 1), 256, 0, (const double *)ws.grad_part, (const double *)ws.loss_part, p.ranges,
                            p.a.rows, p.a.cols, ws.alpha64, ws.adam_m, ws.adam_v, s.lr, 0.9, 0.999, 1.0 - s.p1, 1.0 - s.p2,
                            1e-8, loss_trace ? loss_trace + (s.t - 1) : nullptr);
}

int scale_finish(skim_ctx *ctx, const SkimWorkspace &ws, const ScalePlan &p, float *alpha)
{
    skim_scale_finish_kernel<<<p.cb, 256, 0, ctx->stream>>>(ws.alpha64, p.a.cols, alpha);
    SKIM_CUDA_OK(cudaGetLastError());
    ctx->launches += 1;
    return SKIM_OK;
}

}  // namespace

int skim_launch_scale_update_lfull(skim_ctx *ctx, const uint16_t *W, const float *importance, int64_t rows, int64_t cols,
                                   int64_t ld, const uint8_t *labels, const uint16_t *H, int64_t ldh, float *alpha,
                                   int steps, float lr0, float decay, int decay_every, int exp2, void *scratch,
                                   double *loss_trace)
{
    SkimWorkspace ws = skim_carve(ctx->ws, rows, cols);
    ScalePlan p;
    int rc = scale_begin(ctx, ws, W, importance, rows, cols, ld, labels, alpha, &p);
    if (rc) return rc;
    unsigned char *sp = (unsigned char *)scratch;
    p.a.D = (uint16_t *)sp;
    sp += skim_align256((size_t)rows * cols * 2);
    float *Y = (float *)sp;
    sp += skim_align256((size_t)rows * cols * 4);
    SkimLfullClusters cl;
    cl.labels = labels;
    cl.alpha = ws.alpha64;
    cl.rpart = (double *)sp;
    cl.tconst = p.a.tconst;
    cl.tq = p.a.tq;
    sp += skim_lfull_cluster_bytes(rows, cols);
    p.a.exp2 = exp2;
    AdamSchedule sched(lr0, decay, decay_every);
    for (int t = 0; t < steps; ++t) {
        sched.next();
        rc = skim_launch_dependent(ctx, p.centroids, dim3(p.sum_blocks), SUM_T, sums_smem_bytes((int)cols, false), p.a);
        if (rc) return rc;
        rc = skim_launch_err_lfull(ctx, p.a.D, rows, cols, cols, H, ldh, exp2, sp, nullptr, 1, Y, cols, ws.loss_part, &cl);
        if (rc) return rc;
        rc = skim_launch_dependent(ctx, skim_scale_lf_grad_kernel, p.grad_grid, GT, 0, p.a, (const float *)Y);
        if (rc) return rc;
        rc = scale_adam(ctx, ws, p, sched, loss_trace);
        if (rc) return rc;
    }
    return scale_finish(ctx, ws, p, alpha);
}

int skim_launch_scale_update(skim_ctx *ctx, const uint16_t *W, const float *importance, int64_t rows, int64_t cols,
                             int64_t ld, const uint8_t *labels, float *alpha, int steps, float lr0, float decay,
                             int decay_every, double *loss_trace)
{
    SkimWorkspace ws = skim_carve(ctx->ws, rows, cols);
    ScalePlan p;
    int rc = scale_begin(ctx, ws, W, importance, rows, cols, ld, labels, alpha, &p);
    if (rc) return rc;
    const bool narrow = p.a.grad_warps < GT / 32;
    auto grad = p.a.vec ? (narrow ? skim_scale_grad_kernel<true, true> : skim_scale_grad_kernel<true, false>)
                        : (narrow ? skim_scale_grad_kernel<false, true> : skim_scale_grad_kernel<false, false>);
    AdamSchedule sched(lr0, decay, decay_every);
    for (int t = 0; t < steps; ++t) {
        sched.next();
        rc = skim_launch_dependent(ctx, p.step, dim3(p.sum_blocks), SUM_T, sums_smem_bytes((int)cols, false), p.a);
        if (rc) return rc;
        rc = skim_launch_dependent(ctx, grad, p.grad_grid, GT, 0, p.a);
        if (rc) return rc;
        rc = scale_adam(ctx, ws, p, sched, loss_trace);
        if (rc) return rc;
    }
    return scale_finish(ctx, ws, p, alpha);
}
