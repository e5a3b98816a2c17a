// Exact 1-D weighted K-means of every row: the optimum of the clustering objective of SKIM Section 3.2
// (diagonal form), sum_j g_j (x_j - c_{l_j})^2, which the Lloyd iterations of Algorithm 3 only approach.
// In one dimension the optimal clusters are intervals of the sorted row, so the optimum is a dynamic programme
// over split points,
//     F_1(i) = cost(0, i),    F_j(i) = min_{j-1 <= t < i} F_{j-1}(t) + cost(t, i),
//     cost(t, i) = S2 - S1^2 / S0 over the sorted elements t .. i-1 (0 for an interval without weight),
// and the minimising t never decreases with i, which turns the quadratic search of a layer into m log m
// evaluations.  One block owns a row and reads the row record the sort kernels leave (sorted values and
// importances by groups of 8 with their binary64 prefix sums).
//
//   prefix   the record's two-level prefix sums become flat arrays P0, P1, P2 (sums of g, g x, g x^2) with a position per distinct
//            value -- no optimum splits equal values, and a row of 11 008 binary16 weights has some 6600 values (512 x 11008
//            3972 -> 2632 us, 256 x 4096 with 3280 values a row 648 -> 597) -- and
//            A = F_{j-1} - P2: the cost of a candidate is A(t) - S1^2 / S0 up to a term of i alone, so a candidate needs
//            (P0, P1, A)(t), 24 bytes.  They sit in shared memory where the row fits, else in global memory.
//   layer    positions are visited like the in-order nodes of a perfect binary tree, level by level: a node's
//            search range is bounded by the minimisers of its two nearest finished neighbours.  The ranges of
//            a level tile the span of split points, sharing their end points, so candidate number x of node q in
//            the level's list of all candidates is known without a scan: P(q) = tlo(q) - tlo(0) + q come before it.  The list is
//            dealt to the threads in equal stretches -- by candidates, not by nodes or by split points: one range can be a
//            thousand times another (the minimiser jumps where an outlier enters the prefix), and a thousand nodes
//            can share one split point (it stays put while the elements behind it weigh nothing).  Nodes that end inside a
//            thread's stretch are written at once; the rest meet in a segmented minimum over the lanes, then over the warps.
//            Not every position is needed: only F_K(m), K the largest width, is asked of the last layer, so layer K - 1 is needed at the split
//            points of that alone, and so on down.  The minimisers of a layer lie at or above the ones of the layer before it,
//            t_{j-1}(i) <= t_j(i) (the cost is Monge), so when layer j - 1 is known, layer j needs no position below
//            L_j = t_{j-1}(t_{j-1}(... (m))), K - j times, and no split point below t_{j-1}(L_j).  With 16 clusters that leaves about 60 %
//            of all candidates: 256 x 4096 952 -> 726 us a call.
//   result   for every width the split points are walked back from the row's end; centroid = weighted mean of
//            its interval (an interval without weight: mean of its first and last value), error = F_k(m).
// All widths share the layers: F_2, F_4, F_8, F_16 are read off on the way.
#include "skim_cluster_phases.cuh"

namespace {

using namespace skimk;

constexpr int X_MAX_K = 1 << SKIM_MAX_BIT;    // 16 layers at most

struct ExactSlot {
    size_t q, t, total;                       // byte offsets inside a block's scratch slot
};

__host__ __device__ inline ExactSlot exact_slot(int m)
{
    ExactSlot S;
    const size_t mpad = ((size_t)m + 7) & ~(size_t)7;
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off += (b + 255) & ~(size_t)255; return o; };
    S.q = take((mpad + 8) * 32);                                  // (P0, P1, P2, A) of position 0 .. mpad; only P2 where the rest is in shared memory
    S.t = take((size_t)(X_MAX_K + 1) * ((size_t)m + 1) * 2);      // minimisers of every layer, 16-bit
    S.total = off;
    return S;
}

// A candidate: the node it belongs to, its cost, its split point.
struct Cand {
    double v;
    int q, t;
};
__device__ __forceinline__ bool better(const Cand &x, const Cand &y) { return x.v < y.v || (x.v == y.v && x.t < y.t); }
__device__ __forceinline__ Cand shfl_up(const Cand &c, int off)
{
    Cand r;
    r.v = __shfl_up_sync(0xffffffffu, c.v, off);
    r.q = __shfl_up_sync(0xffffffffu, c.q, off);
    r.t = __shfl_up_sync(0xffffffffu, c.t, off);
    return r;
}
// Every lane's candidate becomes the best of its node's candidates in this and the lower lanes (nodes ascend, so the doubling stops
// as soon as no node reaches that far).
__device__ __forceinline__ void segmented_min(Cand &c)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int q = __shfl_up_sync(0xffffffffu, c.q, off);
        const bool same = lane >= off && q == c.q;
        if (!__any_sync(0xffffffffu, same)) break;
        const double v = __shfl_up_sync(0xffffffffu, c.v, off);
        const int t = __shfl_up_sync(0xffffffffu, c.t, off);
        if (same && (v < c.v || (v == c.v && t < c.t))) {
            c.v = v;
            c.t = t;
        }
    }
}

constexpr int X_NONE = 0x7fffffff;            // node of an idle lane (above every node)

struct ExactShared {
    Cand head[32], tail[32];                  // per warp: its first node, if that ends inside the warp, and its last
    int first[32];                            // per warp: its first node
    float dvals[16];
};

// Where P0, P1 and A of a row live: all in shared memory, P0 and P1 there and A in global memory, or all in global memory.
enum SumsPlace { SUMS_SHARED, SUMS_MIXED, SUMS_GLOBAL };

// shared memory: the minimisers by tree position, ExactShared, and the sums
__host__ __device__ inline size_t exact_optarr_bytes(int m)
{
    return (((size_t)m + 8) * sizeof(uint16_t) + 15) & ~(size_t)15;
}
__host__ __device__ inline size_t exact_smem_bytes(int m, int place)
{
    const size_t mpad = ((size_t)m + 7) & ~(size_t)7;
    return exact_optarr_bytes(m) + ((sizeof(ExactShared) + 15) & ~(size_t)15) + (mpad + 8) * (place == SUMS_SHARED ? 24 : place == SUMS_MIXED ? 16 : 0);
}

// The per-position sums, either way.
template <int PLACE> struct Sums {
    double *p0, *p1, *a, *p2;                 // p2 in global memory
    __device__ __forceinline__ void init(unsigned char *smem, unsigned char *slot, int m)
    {
        const int n = ((m + 7) & ~7) + 8;
        p0 = reinterpret_cast<double *>(smem);
        p1 = p0 + n;
        p2 = reinterpret_cast<double *>(slot);
        a = PLACE == SUMS_SHARED ? p1 + n : p2 + n;
    }
    __device__ __forceinline__ void set(int t, double s0, double s1, double s2) { p0[t] = s0; p1[t] = s1; p2[t] = s2; }
    __device__ __forceinline__ void load(int t, double &s0, double &s1, double &av) const { s0 = p0[t]; s1 = p1[t]; av = a[t]; }
    __device__ __forceinline__ void load_i(int t, double &s0, double &s1) const { s0 = p0[t]; s1 = p1[t]; }
    __device__ __forceinline__ double get_p2(int t) const { return p2[t]; }
    __device__ __forceinline__ void set_a(int t, double v) { a[t] = v; }
};
template <> struct Sums<SUMS_GLOBAL> {
    double4 *q;
    __device__ __forceinline__ void init(unsigned char *, unsigned char *slot, int) { q = reinterpret_cast<double4 *>(slot); }
    __device__ __forceinline__ void set(int t, double s0, double s1, double s2) { q[t] = make_double4(s0, s1, s2, 0.0); }
    __device__ __forceinline__ void load(int t, double &s0, double &s1, double &av) const
    {
        [[maybe_unused]] double unused;
        asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(s0), "=d"(s1), "=d"(unused), "=d"(av) : "l"(q + t));
    }
    __device__ __forceinline__ void load_i(int t, double &s0, double &s1) const { const double2 v = *reinterpret_cast<const double2 *>(q + t); s0 = v.x; s1 = v.y; }
    __device__ __forceinline__ double get_p2(int t) const { return q[t].z; }
    __device__ __forceinline__ void set_a(int t, double v) { reinterpret_cast<double *>(q + t)[3] = v; }
};

// S1^2 / S0 of the candidates: the hardware's approximate reciprocal (better than 20 bits) and one step of the series
// 1 + e + e^2, within one unit in the last place.  What is kept (the layer's F, the result) uses the division.
__device__ __forceinline__ double square_over(double s1, double s0)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(s0));
    const double e = fma(-s0, r, 1.0);
    return s1 * s1 * fma(r, fma(e, e, e), r);
}

template <int PLACE, int XT>
__global__ void __launch_bounds__(XT, 1024 / XT) skim_exact_kernel(ClusterArgs a, int rows_in_chunk, unsigned char *scratch, size_t slot_bytes)
{
    extern __shared__ __align__(16) unsigned char xsmem[];
    constexpr int NW = XT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cols = a.m;
    const RowRecord R = row_record(cols);
    const ExactSlot S = exact_slot(cols);
    unsigned char *slot = scratch + (size_t)blockIdx.x * slot_bytes;
    uint16_t *T = reinterpret_cast<uint16_t *>(slot + S.t);
    uint16_t *optarr = reinterpret_cast<uint16_t *>(xsmem);           // minimisers of the current layer by node position
    ExactShared &sh = *reinterpret_cast<ExactShared *>(xsmem + exact_optarr_bytes(cols));
    Sums<PLACE> Q;
    Q.init(xsmem + exact_optarr_bytes(cols) + ((sizeof(ExactShared) + 15) & ~(size_t)15), slot + S.q, cols);
    const int kmax = 1 << (a.bmin + a.nb - 1);
    if (blockIdx.x == 0 && tid == 0) *a.sort_count = 0;

    for (int local = blockIdx.x; local < rows_in_chunk; local += gridDim.x) {
        const int64_t row = a.row0 + local;
        const unsigned char *rec = a.scratch + (size_t)local * (size_t)a.rec_stride;
        const int nd_rec = *reinterpret_cast<const int *>(rec);
        if (nd_rec < 0) continue;                                   // the sort kernel gave the row up
        const int nd = max(nd_rec, 1);
        if (tid < 16) sh.dvals[tid] = reinterpret_cast<const float *>(rec + 64)[tid];
        const unsigned char *groups = rec + R.groups;
        const double4 *seg = reinterpret_cast<const double4 *>(rec + R.seg);

        // ------------------------------------------------------------ flat prefix sums, a position per distinct value
        float *xv = reinterpret_cast<float *>(T);                   // the values: rows 0 and 1 of T hold no minimisers
        int m;                                                       // distinct values
        {
            const float *gi = reinterpret_cast<const float *>(rec + R.gi);
            const int per = (R.ngrp + XT - 1) / XT, q0 = min(tid * per, R.ngrp), q1 = min(q0 + per, R.ngrp);
            // bit u: element u of group q is the last one of its value
            auto last_of_value = [&](int q, const float (&xs)[8]) {
                const float next = q + 1 < R.ngrp ? gi[q + 1] : SKIM_PAD_VALUE;
                uint32_t r = 0u;
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (q * 8 + u < cols && (q * 8 + u == cols - 1 || xs[u] != (u < 7 ? xs[u < 7 ? u + 1 : 7] : next))) r |= 1u << u;
                return r;
            };
            auto load_values = [&](int q, float (&xs)[8]) {
                const float4 xa = *reinterpret_cast<const float4 *>(groups + (size_t)q * SKIM_GROUP_BYTES), xb = *reinterpret_cast<const float4 *>(groups + (size_t)q * SKIM_GROUP_BYTES + 16);
                xs[0] = xa.x; xs[1] = xa.y; xs[2] = xa.z; xs[3] = xa.w; xs[4] = xb.x; xs[5] = xb.y; xs[6] = xb.z; xs[7] = xb.w;
            };
            int own = 0;
            for (int q = q0; q < q1; ++q) {
                float xs[8];
                load_values(q, xs);
                own += __popc(last_of_value(q, xs));
            }
            int inc = own;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, inc, off);
                if (lane >= off) inc += t;
            }
            if (lane == 31) sh.first[warp] = inc;
            __syncthreads();
            int at = inc - own;
            m = 0;
            for (int w = 0; w < NW; ++w) {
                if (w < warp) at += sh.first[w];
                m += sh.first[w];
            }
            for (int q = q0; q < q1; ++q) {
                float xs[8];
                load_values(q, xs);
                const unsigned char *gr = groups + (size_t)q * SKIM_GROUP_BYTES;
                const float4 ga = *reinterpret_cast<const float4 *>(gr + 32), gb = *reinterpret_cast<const float4 *>(gr + 48);
                const double4 gp = *reinterpret_cast<const double4 *>(gr + 64);
                const double4 sb = seg[q >> SKIM_SEG_SHIFT];
                double p0 = sb.x + gp.x, p1 = sb.y + gp.y, p2 = sb.z + gp.z;
                const float gs[8] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w};
                const uint32_t ends = last_of_value(q, xs);
                if (q == 0) Q.set(0, p0, p1, p2);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const double g = (double)gs[u], x = (double)xs[u];      // padding: g = 0
                    p0 += g;
                    p1 += g * x;
                    p2 += g * x * x;
                    if (ends >> u & 1u) {
                        xv[at] = xs[u];
                        Q.set(++at, p0, p1, p2);
                    }
                }
            }
        }
        __syncthreads();

        // ------------------------------------------------------------ layer 1: F_1(i) - P2(i) = -S1^2 / S0 over [0, i)
        double z0, z1, za;
        Q.load(0, z0, z1, za);
        for (int i = 1 + tid; i <= m; i += XT) {
            double p0, p1, pa;
            Q.load(i, p0, p1, pa);
            const double s0 = p0 - z0, s1 = p1 - z1;
            Q.set_a(i, s0 > 0.0 ? -(s1 * s1 / s0) : -Q.get_p2(i));
        }
        __syncthreads();

        // ------------------------------------------------------------ layers 2 .. kmax
        // up to the largest width with k < nd (the others take the distinct values instead)
        int layers = kmax;
        while (layers >= nd) layers >>= 1;
        // Positions below lowest = L_j are not needed in layer j, and split points below tmin not tried (see the top of the file); L_1 = 1.
        int lowest = layers > 2 ? 2 : m, tmin = 1;
        for (int j = 2; j <= layers; ++j) {
            const int n = m - lowest + 1;                      // positions p = 1 .. n  <->  i = lowest + p - 1
            int L = 1;
            while ((1 << L) - 1 < n) ++L;
            if (tid == 0) optarr[0] = (uint16_t)tmin;
            __syncthreads();
            for (int lev = 0; lev < L; ++lev) {
                const int sh_h = L - 1 - lev, h = 1 << sh_h;
                const int nvalid = ((n >> sh_h) + 1) >> 1;                 // nodes (2q + 1) h <= n of this level
                // a node's position, and the range of split points its two finished neighbours leave it
                auto node_i = [&](int q) { return lowest + ((2 * q + 1) << sh_h) - 1; };
                auto node_tlo = [&](int q) { return (int)optarr[(2 * q) << sh_h]; };
                auto node_thi = [&](int q) {
                    const int thi = node_i(q) - 1, right = (2 * q + 2) << sh_h;
                    return right <= n ? min(thi, (int)optarr[right]) : thi;
                };
                // the list of candidates: node q has P(q) = tlo(q) - tlo(0) + q before its own tlo(q) .. thi(q) (where the limit
                // t < i cuts a range short of its right neighbour's minimiser, the missing split points are skipped)
                const int total = node_thi(nvalid - 1) - tmin + nvalid;
                const int chunk = ((total + XT - 1) / XT) | 1;       // odd: neighbouring lanes' reads fall into different banks
                const int xa = min(tid * chunk, total), xb = min(xa + chunk, total);
                Cand head{__longlong_as_double(0x7ff0000000000000ll), -1, 0}, cur{head.v, X_NONE, 0};
                int first = X_NONE;
                if (xa < xb) {
                    int lo = 0, hi = nvalid - 1;                     // the last node with P(q) <= xa
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (node_tlo(mid) - tmin + mid <= xa) lo = mid; else hi = mid - 1;
                    }
                    int i = node_i(lo), t = xa - lo + tmin, o = (2 * lo + 1) << sh_h;       // o: the node's place in the tree
                    first = lo;
                    // `end`: the last split point that is counted as the node's (a split point past its limit i - 1 is replaced by that)
                    int end = (lo + 1 < nvalid) ? node_tlo(lo + 1) : node_thi(lo);
                    double i0, i1;
                    Q.load_i(i, i0, i1);
                    const double none = __longlong_as_double(0x7ff0000000000000ll);
                    double best = none, head_v = none;
                    int bt = min(t, i - 1), head_t = -1;
                    // a node that ends inside the stretch is written at once; where it began in an earlier one (the first), its
                    // minimiser is written again below
                    for (int left = xb - xa; left > 0; --left) {
                        const int te = min(t, i - 1);
                        double t0, t1, av;
                        Q.load(te, t0, t1, av);
                        const double s0 = i0 - t0, s1 = i1 - t1;
                        const double v = s0 > 0.0 ? av - square_over(s1, s0) : av;
                        const bool less = v < best;
                        best = less ? v : best;
                        bt = less ? te : bt;
                        if (t == end && left > 1) {
                            optarr[o] = (uint16_t)bt;
                            head_v = head_t < 0 ? best : head_v;
                            head_t = head_t < 0 ? bt : head_t;
                            o += 2 << sh_h;
                            i += 2 << sh_h;
                            best = none;
                            bt = min(end, i - 1);
                            const int right = o + h;
                            end = right <= n ? (int)optarr[right] : i - 1;
                            Q.load_i(i, i0, i1);
                        } else {
                            ++t;
                        }
                    }
                    if (head_t >= 0) head = Cand{head_v, first, head_t};
                    cur = Cand{best, o >> (sh_h + 1), bt};
                }
                // ---- over the lanes
                segmented_min(cur);
                const Cand below = shfl_up(cur, 1);
                if (lane > 0 && head.q >= 0 && below.q == head.q && better(below, head)) head = below;
                const int wfirst = __shfl_sync(0xffffffffu, first, 0), nfirst = __shfl_down_sync(0xffffffffu, first, 1);
                if (lane == 0) {
                    sh.first[warp] = wfirst;
                    sh.head[warp].q = -1;
                }
                __syncwarp();
                if (head.q >= 0) {
                    if (head.q == wfirst) sh.head[warp] = head; else optarr[(2 * head.q + 1) << sh_h] = (uint16_t)head.t;
                }
                const bool last = lane == 31 || nfirst == X_NONE;     // no lane behind this one has candidates
                if (lane == 0) sh.tail[warp].q = X_NONE;
                __syncwarp();
                if (first == X_NONE) {
                    // idle
                } else if (last) {
                    sh.tail[warp] = cur;
                } else if (nfirst != cur.q) {
                    // the node ends exactly where the stretch does
                    if (cur.q == wfirst) sh.head[warp] = cur; else optarr[(2 * cur.q + 1) << sh_h] = (uint16_t)cur.t;
                }
                __syncthreads();
                // ---- over the warps
                if (warp == 0) {
                    Cand tl{0.0, X_NONE, 0}, hd{0.0, -1, 0};
                    int nf = X_NONE;
                    if (lane < NW) {
                        tl = sh.tail[lane];
                        hd = sh.head[lane];
                        if (lane + 1 < NW) nf = sh.first[lane + 1];
                    }
                    segmented_min(tl);
                    const Cand bl = shfl_up(tl, 1);
                    if (hd.q >= 0) {
                        if (lane > 0 && bl.q == hd.q && better(bl, hd)) hd = bl;
                        optarr[(2 * hd.q + 1) << sh_h] = (uint16_t)hd.t;
                    }
                    if (tl.q != X_NONE && nf != tl.q) optarr[(2 * tl.q + 1) << sh_h] = (uint16_t)tl.t;
                }
                __syncthreads();
            }
            // F_j - P2 becomes the previous layer.  A position needs the old values of lower ones only: stretches of positions
            // go by from the top, each read in full before it is written.
            uint16_t *Tj = T + (size_t)j * (cols + 1);
            constexpr int PER = 4;
            for (int base = lowest + (n - 1) / (PER * XT) * (PER * XT); base >= lowest; base -= PER * XT) {
                double an[PER];
#pragma unroll
                for (int u = 0; u < PER; ++u) {
                    const int i = base + tid + u * XT;
                    if (i <= m) {
                        const int t = optarr[i - lowest + 1];
                        Tj[i] = (uint16_t)t;
                        double t0, t1, av, i0, i1, ia;
                        Q.load(t, t0, t1, av);
                        Q.load(i, i0, i1, ia);
                        const double s0 = i0 - t0, s1 = i1 - t1;
                        an[u] = s0 > 0.0 ? av - s1 * s1 / s0 : av;
                    }
                }
                __syncthreads();
#pragma unroll
                for (int u = 0; u < PER; ++u) {
                    const int i = base + tid + u * XT;
                    if (i <= m) Q.set_a(i, an[u]);
                }
            }
            // the next layer's limits, from this one's minimisers
            int x = m;
            for (int u = layers - j - 1; u > 0; --u) x = max((int)optarr[x - lowest + 1], lowest);
            x = max(x, lowest + 1);
            if (j < layers) tmin = max((int)optarr[x - lowest + 1], lowest);
            lowest = x;
            __syncthreads();
        }

        // ------------------------------------------------------------ results, one thread per width
        if (tid < a.nb) {
            const int width = a.bmin + tid;
            const int k = 1 << width;
            int off = 0;
            for (int u = 0; u < tid; ++u) off += 1 << (a.bmin + u);
            float *cout = a.centroids + row * a.sumk + off;
            if (nd <= k) {
                for (int u = 0; u < k; ++u) cout[u] = sh.dvals[min(u, nd - 1)];
                a.err[row * a.nb + tid] = 0.0f;
            } else {
                // walk the minimisers back and add the interval costs up
                int i = m;
                double total = 0.0, i0, i1, ia;
                Q.load(m, i0, i1, ia);
                for (int jj = k; jj >= 1; --jj) {
                    const int t = (jj == 1) ? 0 : (int)T[(size_t)jj * (cols + 1) + i];
                    double t0, t1, ta;
                    Q.load(t, t0, t1, ta);
                    const double s0 = i0 - t0, s1 = i1 - t1;
                    float c;
                    if (s0 > 0.0) {
                        c = (float)(s1 / s0);
                        total += (Q.get_p2(i) - Q.get_p2(t)) - s1 * s1 / s0;
                    } else {
                        c = (float)(0.5 * ((double)xv[t] + (double)xv[i - 1]));
                    }
                    cout[jj - 1] = c;
                    i = t;
                    i0 = t0;
                    i1 = t1;
                }
                a.err[row * a.nb + tid] = (float)fmax(total, 0.0);
            }
        }
        __syncthreads();
    }
}
}  // namespace

namespace {
struct ExactVariant {
    void (*kernel)(ClusterArgs, int, unsigned char *, size_t);
    int threads;
    int place;
    int cap;                 // columns up to which it is taken
};
#define SKIM_XV(P, T, CAP) {skim_exact_kernel<P, T>, T, P, CAP}
// Few threads for short rows: a level then has some ten candidates per thread, and its search and reductions (about
// half of the instructions) are not paid by threads with nothing to do; 64 to 512 threads at 512 columns take 1.00, 0.98, 1.54
// and 2.57 ms for 2048 rows.  With no more rows than SMs nothing else fills the SM: twice the threads (32 x 1000: 473 ->
// 416 us).  The largest cap of a place is what one of its blocks (two of those of 512 threads) finds in an SM's shared memory.
const ExactVariant kVariantsExact[] = {
    SKIM_XV(SUMS_SHARED, 64, 384),   SKIM_XV(SUMS_SHARED, 128, 1024),  SKIM_XV(SUMS_SHARED, 256, 2304), SKIM_XV(SUMS_SHARED, 512, 4300),
    SKIM_XV(SUMS_SHARED, 1024, 8700), SKIM_XV(SUMS_MIXED, 1024, 12500), SKIM_XV(SUMS_GLOBAL, 512, 1 << 30),
};
const ExactVariant *exact_variant(const skim_ctx *ctx, int64_t rows, int64_t cols)
{
    for (const ExactVariant &v : kVariantsExact)
        if (cols * (v.threads < 512 && rows <= ctx->sm_count ? 2 : 1) <= v.cap && exact_smem_bytes((int)cols, v.place) <= (size_t)ctx->max_smem_optin) return &v;
    return nullptr;
}
}  // namespace

size_t skim_exact_slot_bytes(int64_t cols) { return exact_slot((int)cols).total; }

// Blocks in flight, each with a scratch slot: what 1024 threads of an SM hold, at most eight per SM.
int skim_exact_slots(const skim_ctx *ctx, int64_t rows, int64_t cols)
{
    const ExactVariant *v = exact_variant(ctx, rows, cols);
    int per_sm = v ? 1024 / v->threads : 1;
    if (per_sm > 8) per_sm = 8;
    const int64_t want = (int64_t)ctx->sm_count * per_sm;
    return (int)(rows < want ? rows : want);
}

int skim_launch_exact(skim_ctx *ctx, const ClusterArgs &args, int64_t rows, void *scratch, int slots)
{
    const ExactVariant *v = exact_variant(ctx, rows, args.m);
    if (!v) return SKIM_ERR_SHAPE;
    const size_t smem = exact_smem_bytes(args.m, v->place);
    SKIM_CUDA_OK(cudaFuncSetAttribute(v->kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    // as many blocks as are resident at once (each owns a scratch slot), at most `slots`
    int per_sm = 1;
    SKIM_CUDA_OK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, v->kernel, v->threads, smem));
    int64_t resident = (int64_t)(per_sm > 0 ? per_sm : 1) * ctx->sm_count;
    if (resident > slots) resident = slots;
    const unsigned blocks = (unsigned)(rows < resident ? rows : resident);
    v->kernel<<<blocks, v->threads, smem, ctx->stream>>>(args, (int)rows, (unsigned char *)scratch, exact_slot(args.m).total);
    SKIM_CUDA_OK(cudaGetLastError());
    ctx->launches += 1;
    return SKIM_OK;
}
