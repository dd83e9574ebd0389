// estimator.cu -- the Monte Carlo estimator of Section 2.1.3 (Eq. MCestimator),
// M_hat = sum_p M(X^p, Y^p) W^p, for the power observables M = v^q of one
// coordinate v of the ensemble (the slow variable x, or one fast component),
// q = 1..max_order, with the weights W^p given or uniform (1/n).
//
// A CTA reduces its threads' binary64 sums in a fixed tree (warp shuffles, then
// the warps in order) to one partial per order, and a second kernel adds a
// slice's partials in a fixed order.  The grid depends only on n and the slice
// count, so a call returns the same bits every time on any device.
//
// Binary32 particles without weights (moments_f32_kernel): binary64 arithmetic
// takes 64 cycles of a sub-partition per warp instruction, so the terms are
// summed on the binary32 units in four words per order, with every rounding
// error kept (29 operations per particle for the first two orders); the words
// enter the binary64 sum once per 128 particles.
//
// Weighted sums and binary64 particles (moments_kernel): each order's term
// enters its sum through one binary64 fused multiply-add.  Binary64 particles:
// W v^(q-1) times v, the running power takes one multiply, 2 max_order - 1
// binary64 operations per particle with weights, 2 max_order - 2 without (the
// first order adds v itself).  Binary32 particles with weights: the exact v^2
// comes from the integer units, 1, 2, 4, 5 operations for the orders up to 1..4.
// On GB300's narrow FP64 pipe that, not HBM, bounds the pass.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "pr_common.cuh"

namespace pr {

constexpr int kMomThreads = 256;
constexpr int kMomMaxOrder = 4;
constexpr int kMomUnroll = 8;              // loads in flight per thread
constexpr int64_t kMomPerBlock = 4096;     // particles per CTA at least (then fewer CTAs)
// CTAs over all slices at most: 12 per SM of 152, two waves of the binary32
// kernel's 6 (orders 1, 2), three of its 4 (orders 3, 4); a constant, so that a
// call's bits do not depend on the device.  Against 16 per SM, 49 x 2^20 values:
// binary32 45.5..154 us instead of 51..161 (orders 1..4), weighted 105..449 instead
// of 110..454, binary64 115..565 instead of 118..566; the largest loss measured
// 4 % (49.5 us instead of 47.5, 16 x 600,000 binary32 values, four orders).
constexpr int64_t kMomMaxBlocks = 1824;

static int64_t moments_blocks(int64_t n, int32_t n_slices)
{
    const int64_t cap = std::max<int64_t>(1, kMomMaxBlocks / n_slices);
    return std::min<int64_t>(cap, std::max<int64_t>(1, (n + kMomPerBlock - 1) / kMomPerBlock));
}

// The CTA's sums of acc, in a fixed order, to its place in `partial`.  Binary64
// additions cost a warp 64 cycles each, so the lanes first share the orders out
// between them: 5 additions for one and two orders, 6 for three and four, instead
// of 5 per order.
template <int Q>
__device__ __forceinline__ void reduce_partials(const double (&acc)[Q], double* __restrict__ partial)
{
    __shared__ double red[Q][kMomThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double a = acc[0];
    int own = 0, o = 16;   // this lane's order; the next distance
    if (Q >= 2) {
        double keep[2], give[2];
        const bool up = lane & 16;
#pragma unroll
        for (int q = 0; q < 2; ++q) {   // orders {0, 1} below lane 16, {2, 3} (or order 1) from it on
            constexpr int H = Q > 2 ? 2 : 1;
            const double lo = q < H ? acc[q < Q ? q : 0] : 0.0, hi = q < H && H + q < Q ? acc[H + q < Q ? H + q : 0] : 0.0;
            keep[q] = up ? hi : lo;
            give[q] = up ? lo : hi;
        }
        a = keep[0] + __shfl_xor_sync(0xffffffffu, give[0], 16);
        own = up ? (Q > 2 ? 2 : 1) : 0;
        o = 8;
        if (Q > 2) {
            const double b = keep[1] + __shfl_xor_sync(0xffffffffu, give[1], 16);
            const bool odd = lane & 8;
            a = (odd ? b : a) + __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
            own += odd ? 1 : 0;
            o = 4;
        }
    }
    const int group = 2 * o;   // lanes that hold one order's sums
#pragma unroll
    for (int k = 16; k > 0; k >>= 1)
        if (k <= o) a += __shfl_down_sync(0xffffffffu, a, k);
    if (lane % group == 0 && own < Q) red[own][warp] = a;
    __syncthreads();
    if (threadIdx.x < Q) {
        double t = 0.0;
        for (int k = 0; k < kMomThreads / 32; ++k) t += red[threadIdx.x][k];
        partial[((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * Q + threadIdx.x] = t;
    }
}

// A sum of binary32 terms in four words.  `hi` starts at 1.5 2^k and stays in
// the binade of 2^k while the terms' sum is below 2^(k-1), so that the rounding
// error of each addition comes exactly from two more (Dekker 1971, |hi| >= |x|);
// `mid`, at 1.5 2^(k-15), takes the errors the same way (below 2^(k-24) each),
// `low`, at 1.5 2^(k-28), those of `mid` (2^(k-39)), and `rest` what is left
// (2^(k-52)).  For up to kRun terms of at most 2^(k-8), each with up to two
// terms for add_small.  The sum is kept to about 2^(k-66), the binary64 sum of
// as many terms to 2^(k-8-53) at best.
constexpr int kRun = 128;

struct Sum4 {
    float hi, mid, low, rest;

    __device__ __forceinline__ static float base(int k) { return __int_as_float(((k + 127) << 23) | 0x400000); }

    __device__ __forceinline__ void reset(int k)
    {
        hi = base(k);
        mid = base(k - 15);
        low = base(k - 28);
        rest = 0.0f;
    }
    // w + x with the error of the addition
    __device__ __forceinline__ static float into(float& w, float x)
    {
        const float s = __fadd_rn(w, x);
        const float e = __fsub_rn(x, __fsub_rn(s, w));
        w = s;
        return e;
    }
    __device__ __forceinline__ void add_small(float e) { rest = __fadd_rn(rest, into(low, into(mid, e))); }
    __device__ __forceinline__ void add(float x) { add_small(into(hi, x)); }
    __device__ __forceinline__ double value(int k) const
    {
        return widen(__fsub_rn(hi, base(k))) + (widen(__fsub_rn(mid, base(k - 15))) +
                                                (widen(__fsub_rn(low, base(k - 28))) + widen(rest)));
    }
};

// the largest of three magnitudes (NaNs are passed over)
__device__ __forceinline__ float max3_abs(float a, float b, float c)
{
    float r;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Exponents e of a bound |v| <= 2^e for which every word and every product's
// error term of the orders up to Q is a normal binary32 number (or too small
// to matter: below 2^-57 of one term at the bound).
template <int Q>
__device__ __forceinline__ bool run_exponent_ok(int e)
{
    return Q * e <= 100 && Q * e >= -40;
}

// Bound by issue: 40 instructions per particle for the first two orders, 31 of
// them binary32 additions and products.  49 x 2^20 particles, mean and second
// moment: 67.0 us with the finishing kernel (211 us with binary64 terms), and
// closer to the exact sum (1.1e-16 instead of 3.6e-16).
template <int Q>
__global__ void __launch_bounds__(kMomThreads, Q <= 2 ? 6 : 4)
moments_f32_kernel(const float* __restrict__ v, int64_t stride, int64_t n, int64_t per_block,
                   double* __restrict__ partial)
{
    const float* vs = v + (int64_t)blockIdx.y * stride;
    const int64_t b = (int64_t)blockIdx.x * per_block, e = min(n, b + per_block);
    double acc[Q];
    Sum4 sum[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) acc[q] = 0.0;
    int ex = -1000;          // the run's bound |v| <= 2^ex; -1000: no run open
    float bound = -1.0f;
    int taken = 0;
    auto close_run = [&]() {
        if (ex > -1000)
#pragma unroll
            for (int q = 0; q < Q; ++q) acc[q] += sum[q].value((q + 1) * ex + 8);
        ex = -1000;
        bound = -1.0f;
        taken = 0;
    };
    auto open_run = [&](int at) {
        if (!run_exponent_ok<Q>(at)) return;
        ex = at;
        bound = __int_as_float((at + 127) << 23);
#pragma unroll
        for (int q = 0; q < Q; ++q) sum[q].reset((q + 1) * ex + 8);
    };
    // least e with |v| <= 2^e for the encoding of |v| (not 0)
    auto exponent_of = [](uint32_t bits) { return (int)(bits >> 23) - 126; };
    // every thread walks the whole range, so that a warp decides together
    for (int64_t b0 = b; b0 < e; b0 += kMomUnroll * kMomThreads) {
        float x[kMomUnroll];
        float top = 0.0f;
        if (b0 + kMomUnroll * kMomThreads <= e) {
            const float* at = vs + b0 + threadIdx.x;
#pragma unroll
            for (int k = 0; k < kMomUnroll; ++k) x[k] = __ldcs(at + k * kMomThreads);
        } else {
#pragma unroll
            for (int k = 0; k < kMomUnroll; ++k) {
                const int64_t p = b0 + (int64_t)k * kMomThreads + threadIdx.x;
                x[k] = p < e ? vs[p] : 0.0f;
            }
        }
#pragma unroll
        for (int k = 0; k < kMomUnroll; k += 2) top = max3_abs(top, x[k], x[k + 1]);
        if (taken == kRun || __any_sync(0xffffffffu, !(top <= bound))) {
            // a new run, its bound four times the warp's largest value here, so
            // that the values to come stay within it
            close_run();
            open_run(exponent_of(__reduce_max_sync(0xffffffffu, __float_as_uint(top))) + 2);
        }
        if (top <= bound) {   // the whole warp (a NaN takes either way into the sum)
            taken += kMomUnroll;
#pragma unroll
            for (int k = 0; k < kMomUnroll; ++k) {
                sum[0].add(x[k]);
                if (Q >= 2) {
                    // x^2 = p + pe exactly
                    const float p = __fmul_rn(x[k], x[k]), pe = __fmaf_rn(x[k], x[k], -p);
                    sum[1].add(p);
                    sum[1].add_small(pe);
                    if (Q >= 3) {
                        const float h = __fmul_rn(p, x[k]);
                        sum[2].add(h);
                        sum[2].add_small(__fmaf_rn(p, x[k], -h));
                        sum[2].add_small(__fmul_rn(pe, x[k]));
                    }
                    if (Q >= 4) {
                        const float h = __fmul_rn(p, p);
                        sum[3].add(h);
                        sum[3].add_small(__fmaf_rn(p, p, -h));
                        // (p + pe)^2: without pe^2 every term would lack 2^-50.6 of itself on average
                        sum[3].add_small(__fmaf_rn(2.0f * p, pe, __fmul_rn(pe, pe)));
                    }
                }
            }
        } else {   // values beyond the runs' range: binary64 terms
#pragma unroll
            for (int k = 0; k < kMomUnroll; ++k) {
                const double d = widen(x[k]);
                double t = d;
                acc[0] += d;
#pragma unroll
                for (int q = 1; q < Q; ++q) {
                    acc[q] = fma(t, d, acc[q]);
                    t *= d;
                }
            }
        }
    }
    close_run();
    reduce_partials<Q>(acc, partial);
}

// The square of a binary32 number, exact in binary64, on the integer units: the
// 48-bit product of the significands moved to the top of the fraction.
// Subnormals, infinities and NaNs take the binary64 product.
__device__ __forceinline__ double square_wide(float f)
{
    const uint32_t u = __float_as_uint(f), e = (u >> 23) & 0xFFu;
    if (e - 1u < 254u) {
        const uint32_t m = (u & 0x7FFFFFu) | 0x800000u;
        const uint64_t P = (uint64_t)m * m;              // f^2 = P 2^(2 (e - 150)), 2^46 <= P < 2^48
        const uint32_t top = (uint32_t)(P >> 47);        // 1: from 2^47 on
        return __longlong_as_double((long long)((P << (6 - top)) + ((uint64_t)(768 + 2 * e + top) << 52)));
    }
    if (u << 1 == 0u) return 0.0;
    const double d = widen(f);
    return d * d;
}
__device__ __forceinline__ double square_wide(double d) { return d * d; }

// Bound by the binary64 pipe, 64 cycles per warp instruction.  Weighted binary32
// values take Q of its instructions per particle for the first two orders (the
// exact square comes from the integer units) and Q + 1 above, 2 Q - 1 with a
// multiply per power, and round less often.  31 x 2,164,802 values, 3 orders: 476 us
// instead of 603; 16 x 607,350, 4 orders: 100 us instead of 136.
template <typename T, int Q, bool W>
__global__ void __launch_bounds__(kMomThreads)
moments_kernel(const T* __restrict__ v, int64_t stride, const double* __restrict__ w, int64_t n, int64_t per_block,
               double* __restrict__ partial)
{
    const int s = blockIdx.y;
    const T* vs = v + (int64_t)s * stride;
    const double* ws = W ? w + (int64_t)s * n : nullptr;
    const int64_t b = (int64_t)blockIdx.x * per_block, e = min(n, b + per_block);
    double acc[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) acc[q] = 0.0;
    // kMomUnroll particles per thread and round, their loads issued first
    for (int64_t p0 = b + threadIdx.x; p0 < e; p0 += kMomUnroll * kMomThreads) {
        T xv[kMomUnroll];
        double wv[kMomUnroll];
#pragma unroll
        for (int k = 0; k < kMomUnroll; ++k) {
            const int64_t p = p0 + (int64_t)k * kMomThreads;
            xv[k] = p < e ? vs[p] : T(0);
            wv[k] = W ? (p < e ? ws[p] : 0.0) : 0.0;
        }
#pragma unroll
        for (int k = 0; k < kMomUnroll; ++k) {
            if (p0 + (int64_t)k * kMomThreads >= e) break;
            const double x = widen(xv[k]);
            if constexpr (W && Q >= 2 && sizeof(T) == 4) {
                const double xx = square_wide(xv[k]);
                acc[0] = fma(wv[k], x, acc[0]);
                acc[1] = fma(wv[k], xx, acc[1]);
                if constexpr (Q >= 3) {
                    const double wxx = wv[k] * xx;
                    acc[2] = fma(wxx, x, acc[2]);
                    if constexpr (Q >= 4) acc[3] = fma(wxx, xx, acc[3]);
                }
                continue;
            }
            double t;                     // W x^q before order q + 1
            int q0;
            if (W) {
                t = wv[k];
                q0 = 0;
            } else {
                acc[0] += x;
                t = x;
                q0 = 1;
            }
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                if (q < q0) continue;
                acc[q] = fma(t, x, acc[q]);
                if (q + 1 < Q) t *= x;
            }
        }
    }
    reduce_partials<Q>(acc, partial);
}

// out[s][q] = sum of slice s's partials (divided by n without weights), one
// warp per sum: the partials of each lane in block order, then a fixed tree
__global__ void __launch_bounds__(128)
moments_finish_kernel(const double* __restrict__ partial, int64_t nblk, int32_t n_slices, int Q, int64_t n,
                      int weighted, double* __restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i >= (int64_t)n_slices * Q) return;
    const int lane = threadIdx.x & 31;
    const int64_t s = i / Q, q = i - s * Q;
    double t = 0.0;
    for (int64_t b = lane; b < nblk; b += 32) t += partial[(s * nblk + b) * Q + q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) out[i] = weighted ? t : t / (double)n;
}

template <typename T, int Q>
static void launch_moments(const void* v, int64_t stride, const double* w, int64_t n, int32_t n_slices, int64_t nblk,
                           double* partial, cudaStream_t st)
{
    const int64_t per = (n + nblk - 1) / nblk;
    const dim3 grid((unsigned)nblk, (unsigned)n_slices);
    if (w)
        moments_kernel<T, Q, true><<<grid, kMomThreads, 0, st>>>(static_cast<const T*>(v), stride, w, n, per, partial);
    else if constexpr (sizeof(T) == 4)
        moments_f32_kernel<Q><<<grid, kMomThreads, 0, st>>>(static_cast<const float*>(v), stride, n, per, partial);
    else
        moments_kernel<T, Q, false><<<grid, kMomThreads, 0, st>>>(static_cast<const T*>(v), stride, w, n, per, partial);
}

template <typename T>
static void launch_moments_q(int Q, const void* v, int64_t stride, const double* w, int64_t n, int32_t n_slices,
                             int64_t nblk, double* partial, cudaStream_t st)
{
    switch (Q) {
    case 1: launch_moments<T, 1>(v, stride, w, n, n_slices, nblk, partial, st); break;
    case 2: launch_moments<T, 2>(v, stride, w, n, n_slices, nblk, partial, st); break;
    case 3: launch_moments<T, 3>(v, stride, w, n, n_slices, nblk, partial, st); break;
    default: launch_moments<T, 4>(v, stride, w, n, n_slices, nblk, partial, st); break;
    }
}

}  // namespace pr

using namespace pr;

extern "C" size_t pr_moments_workspace(int64_t n, int32_t n_slices, int32_t max_order)
{
    if (n < 1 || n_slices < 1 || n_slices > 65535 || max_order < 1 || max_order > kMomMaxOrder) return 0;
    return (size_t)(moments_blocks(n, n_slices) * n_slices * max_order) * sizeof(double);
}

extern "C" pr_status pr_moments(pr_precision precision, const void* v, int64_t slice_stride, const double* w,
                                int64_t n, int32_t n_slices, int32_t max_order, double* out, void* workspace,
                                size_t workspace_bytes, void* stream)
{
    if (precision != PR_F32 && precision != PR_F64) return PR_ERR_INVALID_ARG;
    if (!v || !out || !workspace || n < 1 || n_slices < 1 || n_slices > 65535) return PR_ERR_INVALID_ARG;
    if (max_order < 1 || max_order > kMomMaxOrder || slice_stride < 0 || (n_slices > 1 && slice_stride < n))
        return PR_ERR_INVALID_ARG;
    if (!elem_aligned(workspace, 8) || !elem_aligned(v, elem_bytes(precision)) || !elem_aligned(w, 8) ||
        !elem_aligned(out, 8))
        return PR_ERR_INVALID_ARG;
    if (workspace_bytes < pr_moments_workspace(n, n_slices, max_order)) return PR_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t nblk = moments_blocks(n, n_slices);
    double* partial = static_cast<double*>(workspace);
    if (precision == PR_F32)
        launch_moments_q<float>(max_order, v, slice_stride, w, n, n_slices, nblk, partial, st);
    else
        launch_moments_q<double>(max_order, v, slice_stride, w, n, n_slices, nblk, partial, st);
    PR_CHECK_LAUNCH();
    const int64_t tot = (int64_t)n_slices * max_order;
    moments_finish_kernel<<<(unsigned)((tot + 3) / 4), 128, 0, st>>>(partial, nblk, n_slices, max_order, n,
                                                                        w ? 1 : 0, out);
    PR_CHECK_LAUNCH();
    return PR_OK;
}
