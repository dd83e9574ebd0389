// coarse_dev.cuh -- FP64 block-level pieces of the coarse propagator and the
// serial update (Sections 2.2.2, 3.2.3, 4): deterministic scans, the coarse
// step on one state, the iterators, and the serial sweep over the slices;
// shared by the single-problem and the batched kernels.
#pragma once

#include <cooperative_groups.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include "pr_common.cuh"

namespace pr {

namespace cg = cooperative_groups;

// Work split over the CL CTAs of a thread-block cluster (CL = 1: one CTA).
// Each CTA computes its share [lo(n), hi(n)) of an index range into an
// array in its shared memory; share() copies that part into the same array
// of every other CTA of the cluster (the arrays sit at the same offsets in
// every CTA, distributed shared memory) and synchronises the cluster, so
// that every CTA then holds the whole array.  Each element is computed by
// one CTA with the arithmetic of the single-CTA code, so the results do not
// depend on CL.
template <int CL>
struct Dist {
    int rank;
    __device__ static Dist make()
    {
        Dist d;
        d.rank = CL > 1 ? (int)cg::this_cluster().block_rank() : 0;
        return d;
    }
    __device__ int lo(int n) const { return (int)(((long long)n * rank) / CL); }
    __device__ int hi(int n) const { return (int)(((long long)n * (rank + 1)) / CL); }
    template <typename T>
    __device__ void share(T* arr, int b, int e) const
    {
        __syncthreads();
        if constexpr (CL > 1) {
            cg::cluster_group cl = cg::this_cluster();
            for (int q = 1; q < CL; ++q) {
                T* dst = cl.map_shared_rank(arr, (unsigned)((rank + q) % CL));
                for (int i = b + (int)threadIdx.x; i < e; i += (int)blockDim.x) dst[i] = arr[i];
            }
            cl.sync();
        }
    }
    __device__ void sync() const
    {
        if constexpr (CL > 1) cg::this_cluster().sync();
        else __syncthreads();
    }
};

constexpr int kCoarseThreads = 512;   // every coarse apply uses this block size
constexpr int kUpdateMaxBins = 1024;
// Bin masses of a coarse result at or below this are dropped: below it the
// entries of P @ m are rounding noise of the matrix exponential (absolute
// error ~1e-15), which would otherwise decide where the support of the
// result ends, and with it the quantile iterator's q(0) and q(1).
constexpr double kTailMass = 1e-10;

// ---------------------------------------------------------------------------
// Block-level FP64 helpers (deterministic order for a fixed blockDim)
// ---------------------------------------------------------------------------

// Ordered 64-bit key of a double: signed comparison of keys is numeric
// comparison, and -0 and +0 both map to 0.  The keys of NaNs lie beyond those
// of the infinities, on the side of their sign bit.
__device__ __forceinline__ long long okey(double v)
{
    const long long b = __double_as_longlong(v);
    return b >= 0 ? b : (b ^ 0x7FFFFFFFFFFFFFFFll) + 1;
}

// A binary64 number cut to binary32 (within 2^-23 of it), on the integer units;
// numbers outside the normal binary32 range take the conversion instruction.
__device__ __forceinline__ float narrow(double v)
{
    const uint32_t hi = (uint32_t)__double2hiint(v);
    const uint32_t e = (hi & 0x7FFFFFFFu) - 0x38000000u;   // exponent rebased by 1023 - 127
    if (e - 0x00100000u < 0x0FD00000u)
        return __uint_as_float((hi & 0x80000000u) | __funnelshift_l((uint32_t)__double2loint(v), e, 3));
    return (float)v;
}

// a > b on the integer units, false where either is a NaN (a binary64 comparison
// takes the FP64 pipe, 64 cycles of a sub-partition).
constexpr long long kKeyInf = 0x7FF0000000000000ll;
__device__ __forceinline__ bool greater_f64(double a, double b)
{
    const long long x = okey(a), y = okey(b);
    return x > y && x <= kKeyInf && y >= -kKeyInf;
}

// The larger of a (not a NaN) and b; a NaN in b is passed over.
__device__ __forceinline__ double max_f64(double a, double b)
{
    const long long y = okey(b);
    return y > okey(a) && y <= kKeyInf ? b : a;
}

// min(v, 1) for v >= 0; 1 for a NaN.
__device__ __forceinline__ double at_most_one(double v)
{
    return (unsigned long long)__double_as_longlong(v) < 0x3FF0000000000000ull ? v : 1.0;
}

constexpr int kWsum = 56;   // doubles of the scratch `wsum` of the block-level helpers

// Inclusive scan of v[0..n) into out[0..n) (out may equal v); at most 16
// warps; wsum: kWsum doubles.  The warps beyond the data add exact zeros and
// are passed over.
__device__ inline void block_scan_f64(const double* v, double* out, int n, double* wsum)
{
    const int T = blockDim.x;
    const int chunk = (n + T - 1) / T;
    const int b = min(n, (int)threadIdx.x * chunk), e = min(n, b + chunk);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int warps = (n + 32 * chunk - 1) / (32 * chunk);   // with data
    double incl = 0.0;
    if (warp < warps) {
        for (int i = b; i < e; ++i) incl = __dadd_rn(incl, v[i]);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl = __dadd_rn(t, incl);
        }
        if (lane == 31) wsum[warp] = incl;
    }
    __syncthreads();
    double imax = -INFINITY;
    if (warp < warps) {
        // exclusive prefix of this thread: the warp's offset (the totals before it
        // in order) plus the inclusive prefix of the previous lane
        double off = 0.0;
        for (int w = 0; w < warp; ++w) off = __dadd_rn(off, wsum[w]);
        const double prev = __shfl_up_sync(0xffffffffu, incl, 1);
        double run = lane > 0 ? __dadd_rn(off, prev) : off;
        for (int i = b; i < e; ++i) {
            run = __dadd_rn(run, v[i]);
            imax = max_f64(imax, run);
            out[i] = imax;
        }
    }
    // The prefix of a thread's first element and the last prefix of the thread
    // before it are rounded in different orders, so for non-negative inputs they
    // can step back by an ulp.  Where any does, a prefix maximum (exact in any
    // order) makes the scan non-decreasing again.
    __syncthreads();
    const bool back = b < e && b > 0 && okey(out[b]) < okey(out[b - 1]);
    if (!__syncthreads_or(back)) return;
    if (warp < warps) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_up_sync(0xffffffffu, imax, o);
            if (lane >= o) imax = max_f64(imax, t);
        }
        if (lane == 31) wsum[16 + warp] = imax;
    }
    __syncthreads();
    if (warp < warps) {
        double before = __shfl_up_sync(0xffffffffu, imax, 1);
        if (lane == 0) before = -INFINITY;
        for (int w = 0; w < warp; ++w) before = max_f64(before, wsum[16 + w]);
        for (int i = b; i < e; ++i) out[i] = max_f64(out[i], before);
    }
    __syncthreads();
}

// Block sum of one value per thread (deterministic); wsum >= 33 doubles.
__device__ inline double block_sum_f64(double v, double* wsum)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_down_sync(0xffffffffu, v, o));
    if (lane == 0) wsum[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s = __dadd_rn(s, wsum[w]);
        wsum[32] = s;
    }
    __syncthreads();
    const double r = wsum[32];
    __syncthreads();
    return r;
}

// mp[r] = P[r] . mass for r0 <= r < r1 (0 up to kTailMass), R rows per warp at a
// time; the blocks of 32 columns without mass (any[k] = 0) add exact zeros
// and are passed over.  A row's sums over the lanes are added by a butterfly;
// the rows of a group share its instructions, each in its own lanes and with
// the operands of a butterfly of its own (bound by the binary64 pipe: 64
// cycles per warp instruction and sub-partition).
template <int R>
__device__ __forceinline__ void coarse_rows(const double* __restrict__ P, int I, int r0, int r1, const double* mass,
                                            const unsigned char* any, double* mp)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int nb = (I + 31) >> 5;
    for (int r = r0 + R * warp; r < r1; r += R * nw) {
        const double* row[R];
        double acc[R], p[R];
#pragma unroll
        for (int h = 0; h < R; ++h) {
            row[h] = P + (size_t)min(r + h, r1 - 1) * I;
            acc[h] = 0.0;
            p[h] = lane < I ? row[h][lane] : 0.0;
        }
        for (int k = 0; k < nb; ++k) {   // the next block's entries are loaded ahead
            const int c = 32 * k + lane, cn = c + 32;
            double q[R];
#pragma unroll
            for (int h = 0; h < R; ++h) q[h] = cn < I ? row[h][cn] : 0.0;
            if (any[k] && c < I) {
                const double m = mass[c];
#pragma unroll
                for (int h = 0; h < R; ++h) acc[h] = fma(p[h], m, acc[h]);
            }
#pragma unroll
            for (int h = 0; h < R; ++h) p[h] = q[h];
        }
        const bool b4 = lane & 16, b3 = lane & 8;
        double v;
        if (R == 1) {
            v = __dadd_rn(acc[0], __shfl_xor_sync(0xffffffffu, acc[0], 16));
        } else {
            v = __dadd_rn(b4 ? acc[R > 1] : acc[0], __shfl_xor_sync(0xffffffffu, b4 ? acc[0] : acc[R > 1], 16));
        }
        if (R <= 2) {
            v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 8));
        } else {
            const double a2 = acc[R > 2 ? 2 : 0], a3 = acc[R > 3 ? 3 : 0];
            const double w = __dadd_rn(b4 ? a3 : a2, __shfl_xor_sync(0xffffffffu, b4 ? a2 : a3, 16));
            v = __dadd_rn(b3 ? w : v, __shfl_xor_sync(0xffffffffu, b3 ? v : w, 8));
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
        const int h = (b4 ? 1 : 0) + (b3 ? 2 : 0);   // the row of this lane's sum
        if ((lane & 7) == 0 && h < R && r + h < r1) mp[r + h] = greater_f64(v, kTailMass) ? v : 0.0;
    }
}

// ---------------------------------------------------------------------------
// C_dT on one state: masses, P @ masses (masses <= kTailMass dropped), CDF of
// the result normalised to unit mass.  cdf_in, out: [I+1]; mass, mp: [I].
// All in shared memory; every thread of a kCoarseThreads block calls it.
// ---------------------------------------------------------------------------

constexpr int kShareBins = 256;   // beyond, the division of the CDF is split over the cluster

// The cluster's CTAs meet once in it, or twice above kShareBins.  After one
// meeting a CTA may return while others still scan and divide their `mp`: until
// they have met again it stores nothing into `mp` of theirs, nor into memory
// that overlaps it.
template <int CL = 1>
__device__ inline void coarse_apply_block(const double* __restrict__ P, int I, const double* cdf_in,
                                          double* out, double* mass, double* mp, double* wsum,
                                          const Dist<CL> d = Dist<CL>{0})
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    // masses, and which blocks of 32 hold any: a zero mass adds an exact zero to
    // every row, so the empty blocks (the tails) are passed over
    unsigned char* any = reinterpret_cast<unsigned char*>(wsum + 40);
    const int nb = (I + 31) >> 5;
    for (int k = warp; k < nb; k += nw) {
        const int c = 32 * k + lane;
        const double m = c < I ? __dsub_rn(cdf_in[c + 1], cdf_in[c]) : 0.0;
        if (c < I) mass[c] = m;
        const unsigned full = __ballot_sync(0xffffffffu, (__double_as_longlong(m) << 1) != 0);
        if (lane == 0) any[k] = full != 0u;
    }
    __syncthreads();
    const int r0 = d.lo(I), r1 = d.hi(I);
    // the rows in groups of one to four per warp, as many as give every warp one
    switch (min(4, (r1 - r0 + nw - 1) / nw)) {
    case 0: break;
    case 1: coarse_rows<1>(P, I, r0, r1, mass, any, mp); break;
    case 2: coarse_rows<2>(P, I, r0, r1, mass, any, mp); break;
    case 3: coarse_rows<3>(P, I, r0, r1, mass, any, mp); break;
    default: coarse_rows<4>(P, I, r0, r1, mass, any, mp);
    }
    d.share(mp, r0, r1);
    block_scan_f64(mp, mp, I, wsum);
    const double total = mp[I - 1];
    // every CTA divides all of them where that takes less than the exchange
    // (I / 32 divisions of 9 binary64 instructions on four sub-partitions, about
    // 1000 cycles for the exchange)
    const bool split = CL > 1 && I > kShareBins;
    const int q0 = split ? d.lo(I - 1) : 0, q1 = split ? d.hi(I - 1) : I - 1;
    for (int r = q0 + threadIdx.x; r < q1; r += blockDim.x) {
        const double v = total > 0.0 ? __ddiv_rn(mp[r], total) : 0.0;
        out[r + 1] = at_most_one(v);
    }
    if (threadIdx.x == 0) {
        out[0] = 0.0;
        out[I] = 1.0;
    }
    if (split) d.share(out, 1 + q0, 1 + q1);
    else __syncthreads();
}

// ---------------------------------------------------------------------------
// Quantile iterator J_q (Section 4.4) on CDFs in shared memory.
// ---------------------------------------------------------------------------

// #F < v (le = false) or #F <= v (le = true) of two sorted arrays of n values
// in [0, 1] at once, for two values: four searches of equal length, their
// loads in flight together.
struct Count2 {
    int x, y;
};

template <int H>   // how many of the two values
__device__ __forceinline__ void count_pairs(const double* const (&X)[2], const double* const (&Y)[2],
                                            const bool (&lx)[2], const bool (&ly)[2], const double (&v)[2], int n,
                                            Count2 (&out)[2])
{
    int x[H] = {}, y[H] = {};
    long long key_x[H], key_y[H];   // F < key: "<= v" as "< v + 1" on the encodings
#pragma unroll
    for (int h = 0; h < H; ++h) {
        key_x[h] = dkey(v[h]) + lx[h];
        key_y[h] = dkey(v[h]) + ly[h];
    }
    for (int step = 1 << (31 - __clz(n)); step > 0; step >>= 1) {
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int mx = x[h] + step, my = y[h] + step;
            if (mx <= n && dkey(X[h][mx - 1]) < key_x[h]) x[h] = mx;
            if (my <= n && dkey(Y[h][my - 1]) < key_y[h]) y[h] = my;
        }
    }
#pragma unroll
    for (int h = 0; h < H; ++h) out[h] = Count2{x[h], y[h]};
}

// Both one-sided quantiles of a CDF F at a level p,
//   q^-(p) = min{x : F(x) >= p},  q^+(p) = max{x : F(x) <= p},
// given lt = #F < p and le = #F <= p: they differ only where F is flat at p;
// otherwise one interpolation serves both, kept strictly inside its bin (never
// rounded onto an edge).
__device__ __forceinline__ void quantiles(const GridDev& g, const double* edges, const double* F, double p, int lt,
                                          int le, double& qm, double& qp)
{
    if (lt == 0 || le > lt) {
        qm = edges[lt];
        qp = edges[max(le - 1, 0)];
        return;
    }
    const double t = __ddiv_rn(__dsub_rn(p, F[lt - 1]), __dsub_rn(F[lt], F[lt - 1]));
    const double e0 = edges[lt - 1], e1 = edges[lt];
    double q = __dadd_rn(e0, __dmul_rn(t, g.h));
    const long long k = okey(q), k0 = okey(e0), k1 = okey(e1);
    if (k <= k0 || k >= k1) {   // (a NaN stays one)
        if (k <= k0 && k >= -kKeyInf) q = nextafter(e0, e1);
        if (k >= k1 && k <= kKeyInf) q = nextafter(e1, e0);
    }
    qm = qp = q;
}

// Remote stores (Dist::share) go into mp, counted, kq and the CDFs `out` only.
// Between an exchange's barrier and the next exchange the CTAs of a cluster run
// apart, so what the next one stores over must not be in use in between (its own
// part apart).  Per target: the cluster barrier before the stores, and the last
// use by another CTA that it follows:
//   mp                  the read-back's exchange, or the barrier at the end of a
//                       slice: the levels in the read-back, the division of mp
//   out of the coarse   share(mp): the slice before (its CDF is copied or read
//   step (above 256)    before the coarse step)
//   counted             share(mp), and `out` above 256 bins: the repair of the slice
//                       before; a CTA behind may still scan and divide mp
//   kq                  share(counted): the read-back of the slice before; a CTA
//                       behind may still merge into below, compact or take quantiles
//   out of the          share(kq): its copy at the end of the slice before
//   read-back
struct JqSmem {
    double* levels;   // [3(I+1)]; before the iterator the coarse step's mass | mp [I] each
    double *mass, *mp;
    unsigned long long* counted;   // [3(I+1)]  counts per value, in ibuf (the repair comes later)
    unsigned long long* below;     // [3(I+1)]  counts of the merged levels, in bpos (likewise)
    int* per;                      // [3(I+1) / 32 rounded up]  distinct levels per group of 32, in wsum
    double* kq;       // [6(I+1)]  knots
    double* bsum;     // [6(I+1)]  merged levels | counts of the distinct ones, then scratch of the repair
    int* ibuf;        // [6(I+1)]  counts per value, then segment starts, then sizes of pooled blocks
    int* bpos;        // [6(I+1)]  counts of the merged levels, then segments to pool | pooled blocks
    int* flag;        // [0]: level count, [1]: input not a CDF, [2]: segments to pool, [3]: pooled blocks
    double* wsum;     // [kWsum]
    double* edges;    // [I+1]  edge(g, i) (fill_edges)
};

__host__ __device__ inline size_t jq_smem_bytes(int bins)
{
    const size_t M = 3 * (size_t)(bins + 1);
    return (M + 2 * M + 2 * M + kWsum + (size_t)(bins + 1)) * sizeof(double) + (4 * M + 4) * sizeof(int);
}

__host__ __device__ inline JqSmem carve_jq(unsigned char* base, int bins)
{
    const int M = 3 * (bins + 1);
    JqSmem j;
    j.levels = reinterpret_cast<double*>(base);
    j.mass = j.levels;
    j.mp = j.levels + bins;
    j.kq = j.levels + M;
    j.bsum = j.kq + 2 * M;
    j.wsum = j.bsum + 2 * M;
    j.edges = j.wsum + kWsum;
    j.ibuf = reinterpret_cast<int*>(j.edges + bins + 1);
    j.counted = reinterpret_cast<unsigned long long*>(j.ibuf);
    j.bpos = j.ibuf + 2 * M;
    j.below = reinterpret_cast<unsigned long long*>(j.bpos);
    j.per = reinterpret_cast<int*>(j.wsum);
    j.flag = j.bpos + 2 * M;
    return j;
}

// The edges, once per kernel (each costs two binary64 instructions); the
// caller synchronises the block before the iterator reads them.
__device__ inline void fill_edges(const GridDev& g, JqSmem& s)
{
    for (int i = threadIdx.x; i <= g.bins; i += blockDim.x) s.edges[i] = edge(g, i);
}

// Sum of per[0..g) by the calling warp.
__device__ __forceinline__ int warp_prefix_int(const int* per, int g)
{
    int s = 0;
    for (int k = threadIdx.x & 31; k < g; k += 32) s += per[k];
    return (int)__reduce_add_sync(0xffffffffu, (unsigned)s);
}

// Pool adjacent violators (equal weights) on the knots of one segment, from
// `a` to the next start, by one thread: the left-to-right stack algorithm.  The
// stack of pooled blocks lives in bsum[a..] (sums) and ibuf[a..] (sizes, behind
// the starts still to be read), the two topmost blocks in registers.  A new
// knot q joins the top block (sum R, n knots) where R / n > q, taken as
// R > q n, and blocks merge while mean(left) > mean(right), as
// sum_l n_r > sum_r n_l.  The blocks of two knots or more go to the list
// `blocks` (first knot | size << 16, their sum at their first knot).
//
// A serial chain, so what counts is its length: binary64 instructions take 64
// cycles each, so the comparisons are first made in binary32, which decides
// them exactly wherever the products differ by more than their rounding (sums
// cut to 2^-23, 2^-24 per product: far below the 2^-19 asked for, as long as
// the larger product is 2^-100 at least, where what binary32 loses of smaller
// numbers, up to 2^-149 per knot, does not matter either), and one addition per
// merge is left.  (Not inlined: the sweep around it leaves it no registers.)
static __device__ __noinline__ void pool_segment(double* kq, double* bsum, int* ibuf, int* n_blocks, int* blocks, int a,
                                          int nk)
{
    double R = kq[a], Ls = 0.0;
    float Rf = narrow(R), Lf = 0.0f, n = 1.0f, nl = 1.0f;
    int nb = 0;                  // blocks below the top
    double q = kq[a + 1];
    int k = a + 1, more = 1;
    // mean(left) > mean(right)
    auto above = [](double l, float lf, float l_n, double r, float rf, float r_n) {
        const float x = lf * r_n, y = rf * l_n, diff = x - y;
        const float top = fmaxf(fabsf(x), fabsf(y));
        if (top >= 0x1p-100f && fabsf(diff) > 0x1p-19f * top) return diff > 0.0f;
        return greater_f64(__dmul_rn(l, (double)r_n), __dmul_rn(r, (double)l_n));
    };
    do {
        const float qf = narrow(q);
        const double next = kq[min(k + 1, nk - 1)];
        more = ibuf[k + 1];
        if (above(R, Rf, n, q, qf, 1.0f)) {
            R = __dadd_rn(R, q);
            n += 1.0f;
            Rf = narrow(R);
            while (nb > 0 && above(Ls, Lf, nl, R, Rf, n)) {
                R = __dadd_rn(Ls, R);
                n += nl;
                Rf = narrow(R);
                if (--nb > 0) {
                    Ls = bsum[a + nb - 1];
                    nl = __int_as_float(ibuf[a + nb - 1]);
                    Lf = narrow(Ls);
                }
            }
        } else {
            if (nb > 0) {
                bsum[a + nb - 1] = Ls;
                ibuf[a + nb - 1] = __float_as_int(nl);
            }
            Ls = R;
            Lf = Rf;
            nl = n;
            ++nb;
            R = q;
            Rf = qf;
            n = 1.0f;
        }
        q = next;
        ++k;
    } while (more == 0);
    // the last block first: a block starts at or behind its place on the stack
    for (int t = nb; t >= 0; --t) {
        const double sum = t == nb ? R : t == nb - 1 ? Ls : bsum[a + t];
        const int c = (int)(t == nb ? n : t == nb - 1 ? nl : __int_as_float(ibuf[a + t]));
        k -= c;
        if (c >= 2) {   // a knot that pooled with nothing keeps its bits
            kq[k] = sum;
            blocks[atomicAdd(n_blocks, 1)] = k | c << 16;
        }
    }
}

// out = J_q(A, B, C).  A, B, C, out: [I+1] in shared memory (out distinct).
// Returns through flag[1] a non-zero value if an input was not a CDF.  With a
// cluster (CL > 1) the quantiles at the levels and the read-back at the edges
// are split over its CTAs; the rest runs in every CTA on identical data.
template <int CL = 1>
__device__ inline void quantile_iterate_block(const GridDev& g, int qmode, const double* A, const double* B,
                                              const double* C, double* out, JqSmem& s,
                                              const Dist<CL> d = Dist<CL>{0})
{
    const int I = g.bins;
    const int n1 = I + 1;
    const int M = 3 * n1;
    const int T = blockDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = T >> 5;
    int* per = s.per;
    if (threadIdx.x == 0) s.flag[2] = s.flag[3] = 0;
    // validity: in [0, 1] (NaN fails) and non-decreasing, by ordered keys
    const long long k0 = okey(0.0), k1 = okey(1.0);
    for (int i = threadIdx.x; i < n1; i += T) {
        const double* Fs[3] = {A, B, C};
        for (int f = 0; f < 3; ++f) {
            const long long kv = okey(Fs[f][i]);
            bool bad = kv < k0 || kv > k1;
            if (i > 0 && okey(Fs[f][i - 1]) > kv) bad = true;
            if (bad) s.flag[1] = 1;
        }
    }
    // 1. sorted union of the 3(I+1) levels (stable merge by rank) into bsum, and
    //    with each element how many values of A, B and C lie below it (exact
    //    for the first of equal elements) into below
    unsigned long long* below = s.below;
    unsigned long long* counted = s.counted;
    {
        const int m0 = d.lo(M), m1 = d.hi(M);   // this CTA's share
        for (int k = m0 + threadIdx.x; k < m1; k += 2 * T) {
            const double *X[2], *Y[2];
            bool lx[2], ly[2];
            double v[2];
            int f[2], i[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int kk = min(k + h * T, M - 1);
                f[h] = kk / n1;
                i[h] = kk - f[h] * n1;
                // ties keep the order A, B, C
                X[h] = f[h] == 0 ? B : A;
                Y[h] = f[h] == 2 ? B : C;
                lx[h] = f[h] != 0;
                ly[h] = f[h] == 2;
                v[h] = (f[h] == 0 ? A : f[h] == 1 ? B : C)[i[h]];
            }
            Count2 c[2];
            if (k + T < m1) count_pairs<2>(X, Y, lx, ly, v, n1, c);
            else count_pairs<1>(X, Y, lx, ly, v, n1, c);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (k + h * T >= m1) break;
                const int na = f[h] == 0 ? i[h] : c[h].x;
                const int nb = f[h] == 0 ? c[h].x : f[h] == 1 ? i[h] : c[h].y;
                const int nc = f[h] == 2 ? i[h] : c[h].y;
                counted[k + h * T] = (unsigned long long)na | (unsigned long long)nb << 16 | (unsigned long long)nc << 32;
            }
        }
        d.share(counted, m0, m1);
    }
    for (int k = threadIdx.x; k < M; k += T) {
        const unsigned long long c = counted[k];
        const int r = min((int)(c & 0xFFFF) + (int)(c >> 16 & 0xFFFF) + (int)(c >> 32), M - 1);   // (clamped: inputs
        s.bsum[r] = k < n1 ? A[k] : k < 2 * n1 ? B[k - n1] : C[k - 2 * n1];                       // that are no CDFs)
        below[r] = c;
    }
    __syncthreads();
    // the distinct levels and their counts, in order
    unsigned long long* lt = reinterpret_cast<unsigned long long*>(s.bsum + M);
    const int groups = (M + 31) >> 5;
    for (int q = warp; q < groups; q += nw) {
        const int k = 32 * q + lane;
        const unsigned first =
            __ballot_sync(0xffffffffu, k < M && (k == 0 || !deq(s.bsum[k], s.bsum[k - 1])));
        if (lane == 0) per[q] = __popc(first);
    }
    __syncthreads();
    for (int q = warp; q < groups; q += nw) {
        const int k = 32 * q + lane;
        const bool is = k < M && (k == 0 || !deq(s.bsum[k], s.bsum[k - 1]));
        const unsigned first = __ballot_sync(0xffffffffu, is);
        const int before = warp_prefix_int(per, q);
        if (is) {
            const int l = before + __popc(first & ((1u << lane) - 1u));
            s.levels[l] = s.bsum[k];
            lt[l] = below[k];
        }
        if (q == groups - 1 && lane == 0) s.flag[0] = before + __popc(first);   // number of levels L
    }
    __syncthreads();
    const int L = s.flag[0];
    // 2-3. quantiles of A, B, C at every level and the combined knots.  #F <= p
    //    at a level is #F < p at the next one.
    const bool two = qmode == PR_QMODE_TWO_SIDED;
    const int nk = two ? 2 * L - 2 : L;
    const int l0 = d.lo(L), l1 = d.hi(L);
    const unsigned long long all = (unsigned long long)n1 | (unsigned long long)n1 << 16 | (unsigned long long)n1 << 32;
    auto counts = [&](int l, int f, int& a, int& b) {
        const unsigned long long now = lt[l], next = l + 1 < L ? lt[l + 1] : all;
        a = min((int)(now >> (16 * f)) & 0xFFFF, I);
        b = min((int)(next >> (16 * f)) & 0xFFFF, n1);
    };
    auto knots = [&](int l, double am, double ap, double bm, double bp, double cm, double cp) {
        const bool first = l == 0, last = l == L - 1;
        if (two) {
            if (!first) s.kq[2 * l - 1] = __dadd_rn(__dadd_rn(bm, __dsub_rn(am, cm)), 0.0);
            if (!last) s.kq[2 * l] = __dadd_rn(__dadd_rn(bp, __dsub_rn(ap, cp)), 0.0);
        } else {
            double qa, qb, qc;
            if (first) { qa = ap; qb = bp; qc = cp; }
            else if (last) { qa = am; qb = bm; qc = cm; }
            else {
                qa = __dmul_rn(0.5, __dadd_rn(am, ap));
                qb = __dmul_rn(0.5, __dadd_rn(bm, bp));
                qc = __dmul_rn(0.5, __dadd_rn(cm, cp));
            }
            s.kq[l] = __dadd_rn(__dadd_rn(qb, __dsub_rn(qa, qc)), 0.0);
        }
    };
    if (CL >= 8) {
        // few levels per CTA: a thread per level and function (whole warps of one
        // function), the quantiles through shared memory (the merged levels'
        // place: 6 (l1 - l0) <= M)
        const int nl = l1 - l0, pad = (nl + 31) & ~31;
        double* qv = s.bsum;
        for (int t = threadIdx.x; t < 3 * pad; t += T) {
            const int f = t / pad, j = t - f * pad;
            if (j < nl) {
                int a, b;
                counts(l0 + j, f, a, b);
                double qm, qp;
                quantiles(g, s.edges, f == 0 ? A : f == 1 ? B : C, s.levels[l0 + j], a, b, qm, qp);
                qv[2 * f * nl + j] = qm;
                qv[(2 * f + 1) * nl + j] = qp;
            }
        }
        __syncthreads();
        for (int j = threadIdx.x; j < nl; j += T)
            knots(l0 + j, qv[j], qv[nl + j], qv[2 * nl + j], qv[3 * nl + j], qv[4 * nl + j], qv[5 * nl + j]);
    } else {
        for (int l = l0 + threadIdx.x; l < l1; l += T) {
            const double p = s.levels[l];
            double qm[3], qp[3];
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                int a, b;
                counts(l, f, a, b);
                quantiles(g, s.edges, f == 0 ? A : f == 1 ? B : C, p, a, b, qm[f], qp[f]);
            }
            knots(l, qm[0], qp[0], qm[1], qp[1], qm[2], qp[2]);
        }
    }
    // knots of levels [l0, l1): 2l - 1 and 2l (two-sided), l (midpoint)
    if (two) d.share(s.kq, max(2 * l0 - 1, 0), min(2 * l1 - 1, nk));
    else d.share(s.kq, l0, l1);
    // 4. monotone repair: pool adjacent violators (PAV) with equal weights.
    //    A boundary between knots k-1 and k where max(q[0..k-1]) <= min(q[k..])
    //    is never crossed by a pooled block, and the left-to-right stack
    //    algorithm does the same merges, with the same additions in the same
    //    order, on each side of it as it does on the whole.  So the knots are
    //    cut at every such boundary (exact integer max/min scans on ordered
    //    keys) and each segment is pooled by its own thread with that
    //    algorithm; the bits are those of the single sequential pass.  Knots
    //    that are in order already have nothing to pool.
    bool out_of_order = false;
    for (int k = 1 + threadIdx.x; k < nk; k += T) out_of_order |= okey(s.kq[k]) < okey(s.kq[k - 1]);
    if (__syncthreads_or(out_of_order)) {
        long long* pm = reinterpret_cast<long long*>(s.bsum);   // max of the keys before each knot
        long long* wmax = reinterpret_cast<long long*>(s.wsum);
        long long* wmin = wmax + 16;
        const int chunk = (nk + T - 1) / T;
        const int b0 = min(nk, (int)threadIdx.x * chunk), e0 = min(nk, b0 + chunk);
        // prefix maximum and suffix minimum, both over the threads' chunks
        long long hi = LLONG_MIN, lo = LLONG_MAX;
        for (int i = b0; i < e0; ++i) {
            const long long k = okey(s.kq[i]);
            pm[i] = hi;      // within the chunk, for now
            hi = max(hi, k);
            lo = min(lo, k);
        }
        long long ih = hi, il = lo;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long th = __shfl_up_sync(0xffffffffu, ih, o), tl = __shfl_down_sync(0xffffffffu, il, o);
            if (lane >= o) ih = max(ih, th);
            if (lane + o < 32) il = min(il, tl);
        }
        if (lane == 31) wmax[warp] = ih;
        if (lane == 0) wmin[warp] = il;
        long long before = __shfl_up_sync(0xffffffffu, ih, 1), after = __shfl_down_sync(0xffffffffu, il, 1);
        if (lane == 0) before = LLONG_MIN;
        if (lane == 31) after = LLONG_MAX;
        __syncthreads();
        for (int w = 0; w < warp; ++w) before = max(before, wmax[w]);
        for (int w = warp + 1; w < nw; ++w) after = min(after, wmin[w]);
        for (int k = e0 - 1; k >= b0; --k) {
            after = min(after, okey(s.kq[k]));
            s.ibuf[k] = (k == 0 || max(before, pm[k]) <= after) ? 1 : 0;   // a segment starts here
        }
        if (threadIdx.x == 0) s.ibuf[nk] = 1;
        __syncthreads();
        // the segments of two knots or more, packed into as few warps as they
        // take (a warp's binary64 instruction costs the same for one lane as for 32)
        for (int k = threadIdx.x; k < nk; k += T) {
            const bool is = s.ibuf[k] == 1 && s.ibuf[k + 1] == 0;
            const unsigned some = __ballot_sync(__activemask(), is);
            if (is) {
                const int leader = __ffs(some) - 1;
                int base = 0;
                if (lane == leader) base = atomicAdd(&s.flag[2], __popc(some));
                base = __shfl_sync(some, base, leader);
                s.bpos[base + __popc(some & ((1u << lane) - 1u))] = k;
            }
        }
        __syncthreads();
        const int nseg = s.flag[2];
        int* blocks = s.bpos + ((nk >> 1) + 1);   // pooled blocks: start | size << 16
        for (int j = threadIdx.x; j < nseg; j += T)
            pool_segment(s.kq, s.bsum, s.ibuf, &s.flag[3], blocks, s.bpos[j], nk);
        __syncthreads();
        // their means, by a thread per block
        const int npool = s.flag[3];
        for (int j = threadIdx.x; j < npool; j += T) {
            const int k = blocks[j] & 0xFFFF, c = blocks[j] >> 16;
            const double mean = __dadd_rn(__ddiv_rn(s.kq[k], (double)c), 0.0);
            for (int u = 0; u < c; ++u) s.kq[k + u] = mean;
        }
    }
    __syncthreads();
    // 5. PL CDF through the knots, right-continuous, read at the interior edges
    const int e0 = 1 + d.lo(I - 1), e1 = 1 + d.hi(I - 1);
    for (int i = e0 + threadIdx.x; i < e1; i += T) {
        const double x = s.edges[i];
        const long long kx = okey(x);
        int lo = 0, hi = nk;   // first knot with kq > x
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (okey(s.kq[mid]) <= kx) lo = mid + 1; else hi = mid;
        }
        const int j = lo - 1;
        double v;
        if (j < 0) v = 0.0;
        else {
            const double pj = s.levels[two ? (j + 1) >> 1 : j];
            if (j == nk - 1) v = pj;
            else {
                const double pn = s.levels[two ? (j + 2) >> 1 : j + 1];
                const double t = __ddiv_rn(__dsub_rn(x, s.kq[j]), __dsub_rn(s.kq[j + 1], s.kq[j]));
                v = __dadd_rn(pj, __dmul_rn(t, __dsub_rn(pn, pj)));
            }
        }
        if ((unsigned long long)__double_as_longlong(v) > 0x3FF0000000000000ull) {
            if (greater_f64(0.0, v)) v = 0.0;   // (a NaN stays: the caller reports it)
            if (greater_f64(v, 1.0)) v = 1.0;
        }
        out[i] = v;
    }
    if (threadIdx.x == 0) {
        out[0] = 0.0;
        out[I] = 1.0;
    }
    d.share(out, e0, e1);
}

// Additive (4.1), multiplicative (4.2) and rotation (4.3) iterators on masses.
__device__ inline void mass_iterate_block(int kind, int I, const double* A, const double* B, const double* C,
                                   double* out, double* r, double* wsum)
{
    double pu = 0.0, pv = 0.0, pw = 0.0;
    for (int i = threadIdx.x; i < I; i += blockDim.x) {
        const double a = __dsub_rn(A[i + 1], A[i]), b = __dsub_rn(B[i + 1], B[i]), c = __dsub_rn(C[i + 1], C[i]);
        if (kind == PR_ITER_ADD) {
            const double v = __dsub_rn(__dadd_rn(a, b), c);
            r[i] = v < 0.0 ? 0.0 : v;
        } else if (kind == PR_ITER_MULT) {
            r[i] = c > 0.0 ? __dmul_rn(a, __ddiv_rn(b, c)) : 0.0;
        } else {
            pu = __dadd_rn(pu, sqrt(__dmul_rn(b, c)));
            pv = __dadd_rn(pv, sqrt(__dmul_rn(b, a)));
            pw = __dadd_rn(pw, sqrt(__dmul_rn(c, a)));
        }
    }
    if (kind == PR_ITER_ROT) {
        const double u = block_sum_f64(pu, wsum);
        const double v = block_sum_f64(pv, wsum);
        const double w = block_sum_f64(pw, wsum);
        const double ca = __ddiv_rn(__dsub_rn(__dadd_rn(u, __dmul_rn(__dmul_rn(2.0, u), w)), v), __dadd_rn(1.0, w));
        const double cc = __ddiv_rn(__dadd_rn(u, v), __dadd_rn(1.0, w));
        for (int i = threadIdx.x; i < I; i += blockDim.x) {
            const double a = __dsub_rn(A[i + 1], A[i]), b = __dsub_rn(B[i + 1], B[i]), c = __dsub_rn(C[i + 1], C[i]);
            const double sv = __dsub_rn(__dadd_rn(__dmul_rn(ca, sqrt(a)), sqrt(b)), __dmul_rn(cc, sqrt(c)));
            r[i] = __dmul_rn(sv, sv);
        }
    }
    __syncthreads();
    block_scan_f64(r, r, I, wsum);
    const double total = r[I - 1];
    if (!(total > 0.0)) {   // no mass to normalise (the multiplicative iterator
        // when the supports of a b and c do not meet): the correction is
        // dropped and the update keeps the fine result b
        for (int i = threadIdx.x; i <= I; i += blockDim.x) out[i] = B[i];
        __syncthreads();
        return;
    }
    for (int i = threadIdx.x; i < I - 1; i += blockDim.x) {
        const double v = __ddiv_rn(r[i], total);
        out[i + 1] = v < 1.0 ? v : 1.0;
    }
    if (threadIdx.x == 0) {
        out[0] = 0.0;
        out[I] = 1.0;
    }
    __syncthreads();
}

__host__ __device__ inline size_t coarse_apply_smem(int bins)
{
    return ((size_t)2 * (bins + 1) + 2 * (size_t)bins + kWsum) * sizeof(double);
}

__host__ __device__ inline size_t update_smem(int bins)
{
    return (size_t)5 * (bins + 1) * sizeof(double) + jq_smem_bytes(bins);
}

// The serial update of Section 3.2.3 (Eq. mm_sequential) for one problem on
// the calling CTA, or on the CL CTAs of a cluster (kCoarseThreads threads,
// update_smem(bins) bytes at usm in each):
//   rho^0 = cdf0, rho^{n+1} = J(C(rho^n), fstar[n], cstar[n]), n < K.
// Every CTA of the cluster holds the whole state; the matrix-vector product,
// the normalisation, the quantiles and the read-back are split between them
// (Dist), so the FP64 work per slice spreads over CL SMs.  Results do not
// depend on CL.
template <int CL = 1>
__device__ inline void serial_sweep(unsigned char* usm, const double* __restrict__ P, const GridDev& g,
                                    int iterator, int qmode, int K, const double* __restrict__ cdf0,
                                    const double* __restrict__ fstar, const double* __restrict__ cstar,
                                    double* __restrict__ next, int32_t* status)
{
    const Dist<CL> d = Dist<CL>::make();
    const bool writer = d.rank == 0;
    const int I = g.bins;
    double* cur = reinterpret_cast<double*>(usm);
    double* Ab = cur + (I + 1);
    double* Bb = Ab + (I + 1);
    double* Cb = Bb + (I + 1);
    double* Ob = Cb + (I + 1);
    JqSmem js = carve_jq(reinterpret_cast<unsigned char*>(Ob + (I + 1)), I);
    if (threadIdx.x == 0) js.flag[1] = 0;
    fill_edges(g, js);
    for (int i = threadIdx.x; i <= I; i += blockDim.x) {
        cur[i] = cdf0[i];
        if (writer) next[i] = cdf0[i];
    }
    d.sync();   // every CTA of the cluster runs before any writes into its shared memory
    for (int n = 0; n < K; ++n) {
        coarse_apply_block<CL>(P, I, cur, Ab, js.mass, js.mp, js.wsum, d);
        double* res = Ab;
        if (iterator != PR_ITER_NONE) {
            for (int i = threadIdx.x; i <= I; i += blockDim.x) {
                Bb[i] = fstar[(size_t)n * (I + 1) + i];
                Cb[i] = cstar[(size_t)n * (I + 1) + i];
            }
            __syncthreads();
            if (iterator == PR_ITER_QUANTILE) quantile_iterate_block<CL>(g, qmode, Ab, Bb, Cb, Ob, js, d);
            else mass_iterate_block(iterator, I, Ab, Bb, Cb, Ob, js.kq, js.wsum);
            res = Ob;
        }
        for (int i = threadIdx.x; i <= I; i += blockDim.x) {
            const double v = res[i];
            if (!isfinite(v)) js.flag[1] = 1;
            cur[i] = v;
            if (writer) next[(size_t)(n + 1) * (I + 1) + i] = v;
        }
        // the next slice stores into mp of CTAs that may still divide it, unless an
        // exchange has followed the coarse step's first one (the quantile
        // iterator's, or that of `out` on larger grids)
        if (iterator != PR_ITER_QUANTILE && I <= kShareBins) d.sync();
        else __syncthreads();
    }
    if (threadIdx.x == 0 && status && writer) *status = js.flag[1] ? PR_ERR_NUMERIC : PR_OK;
    d.sync();   // no CTA leaves while another may still write into its shared memory
}

}  // namespace pr
