// coarse.cu -- coarse propagator C_dT (Section 2.2.2), the serial parareal
// update rho^{n+1} = J(C(rho^n), rho_f*, rho_c*) (Section 3.2.3, Eq.
// mm_sequential) with the iterators of Section 4, and the W1 distance.
//
// Everything here is FP64.  The macroscopic states are short (I <= 4096 bins,
// the serial update I <= 1024), so the work is latency-bound: a CTA or a
// cluster per state vector, and one cluster for the serial sweep over the
// slices.  Operations
// that decide exactness (edges, quantile interpolation, the monotone repair,
// reading the CDF back at the edges) are written with explicitly rounded
// intrinsics so that no multiply-add is fused.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "coarse_dev.cuh"
#include "pr_common.cuh"

namespace pr {

struct ChemRates {
    double k[6];
    bool printed;
};

struct CoarseHandle {
    GridDev g;
    double* P;   // row-major I x I
    int device;
};

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------

// Mean ybar of the chemical system's fast equilibrium (Section 2.2.3),
// phi(y) ~ exp(-int_0^y G'(s)/E(s) ds) / E(y), by the trapezoidal rule on
// y_j = j/2, j = 0..4000 (the inner integral cumulatively on the same grid).
// One CTA evaluates the integrands in parallel; the three sums keep the order
// of the grid (one thread each, from shared memory), so that only additions
// are left in the serial chains.
constexpr double kChemDy = 0.5;
constexpr int kChemJ = 4000;
constexpr int kChemThreads = 1024;
constexpr size_t kChemSmem = (size_t)2 * (kChemJ + 1) * sizeof(double);

__device__ __forceinline__ void chem_fast_terms(const double* k, bool printed, double y, double& ratio,
                                                double& log_e)
{
    const double y1 = y * (y - 1.0), y2 = y1 * (y - 2.0);
    const double net = k[0] - k[1] * y + k[2] * y1 - k[3] * y2;              // -G' (net rates)
    const double dg = printed ? -k[0] - k[1] * y + k[2] * y1 - k[3] * y2 : -net;
    const double e = 0.5 * (k[0] + k[1] * y + k[2] * y1 + k[3] * y2);
    ratio = dg / e;
    log_e = log(e);
}

__global__ void __launch_bounds__(kChemThreads) chem_ybar_kernel(ChemRates r, double* __restrict__ out)
{
    extern __shared__ __align__(16) double csm[];
    __shared__ double wmax[kChemThreads / 32];
    double* a = csm;                  // G'/E, then the integral, then phi
    double* b = csm + kChemJ + 1;     // log E
    const int t = threadIdx.x, T = blockDim.x;
    for (int j = t; j <= kChemJ; j += T) chem_fast_terms(r.k, r.printed, j * kChemDy, a[j], b[j]);
    __syncthreads();
    if (t == 0) {
        double integral = 0.0, prev = a[0];
        a[0] = 0.0;
        for (int j = 1; j <= kChemJ; ++j) {
            const double ratio = a[j];
            integral += 0.5 * kChemDy * (prev + ratio);
            prev = ratio;
            a[j] = integral;
        }
    }
    __syncthreads();
    double top = -INFINITY;
    for (int j = t; j <= kChemJ; j += T) {
        a[j] = -a[j] - b[j];          // log phi
        top = fmax(top, a[j]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
    if ((t & 31) == 0) wmax[t >> 5] = top;
    __syncthreads();
    for (int w = 0; w < T / 32; ++w) top = fmax(top, wmax[w]);
    for (int j = t; j <= kChemJ; j += T) a[j] = exp(a[j] - top);
    __syncthreads();
    if (t == 0 || t == 32) {          // the two sums in warps of their own
        double sum = 0.0;
        for (int j = 0; j <= kChemJ; ++j) {
            const double w = (j == 0 || j == kChemJ) ? 0.5 : 1.0;
            sum = t ? fma(w, a[j], sum) : fma(w * (j * kChemDy), a[j], sum);
        }
        b[t] = sum;
    }
    __syncthreads();
    if (t == 0) *out = b[0] / b[32];
}

// The generator times slice_dt by its three diagonals: sub[c] = A(c, c - 1),
// dia[c] = A(c, c), sup[c] = A(c, c + 1) (0 where there is no such column).
__global__ void generator_kernel(GridDev g, int kind, double lam, double beta, double eps, double tau_x, double k4,
                                 double k5, const double* __restrict__ ybar_ptr, double slice_dt,
                                 double* __restrict__ sub, double* __restrict__ dia, double* __restrict__ sup)
{
    const int I = g.bins;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= I) return;
    const bool chem = kind == PR_MODEL_CHEM || kind == PR_MODEL_CHEM_PRINTED;
    const double a = chem ? k4 * *ybar_ptr : 0.0;   // k4 ybar
    // Dbar(x): 1/beta, or (k4 ybar + k5 x)/2 for the chemical system
    auto dbar = [&](double x) { return chem ? 0.5 * (a + k5 * x) : 1.0 / beta; };
    // log rho_inf(x) = log(1/Dbar(x)) - int_0^x Fbar'/Dbar: Fbar(x)/Dbar for a
    // constant Dbar; for the chemical system 2x - (4a/k5) log(1 + k5 x/a)
    // (Fbar' = k5 x - a, net rates) or -2x (Fbar' = -(a + k5 x), as printed)
    auto fbar = [&](double x) {
        if (kind == PR_MODEL_ADVECTION) return x / eps;   // given directly (linear advection case)
        return kind == PR_MODEL_OU ? 0.5 * (1.0 - lam) * x * x
                                   : 0.25 * x * x * x * x - 0.5 * (1.0 - lam) * x * x;
    };
    auto log_rho_inf = [&](double x) {
        if (!chem) return log(1.0 / dbar(x)) - fbar(x) / dbar(x);
        const double integral = kind == PR_MODEL_CHEM ? 2.0 * x - (4.0 * a / k5) * log1p(k5 * x / a) : -2.0 * x;
        return log(1.0 / dbar(x)) - integral;
    };
    auto centre = [&](int k) { return 0.5 * (edge(g, k) + edge(g, k + 1)); };
    auto width = [&](int k) { return edge(g, k + 1) - edge(g, k); };
    double diag = 0.0, left = 0.0, right = 0.0;
    // left edge e = c: cell c loses phi_c
    if (c >= 1) {
        const int e = c;
        const double xe = edge(g, e);
        const double coef = dbar(xe) / (centre(e) - centre(e - 1));
        const double rr = exp(log_rho_inf(xe) - log_rho_inf(centre(e))) / width(e);
        const double rl = exp(log_rho_inf(xe) - log_rho_inf(centre(e - 1))) / width(e - 1);
        diag -= coef * rr / tau_x;
        left += coef * rl / tau_x;
    }
    // right edge e = c+1: cell c gains phi_{c+1}
    if (c + 1 <= I - 1) {
        const int e = c + 1;
        const double xe = edge(g, e);
        const double coef = dbar(xe) / (centre(e) - centre(e - 1));
        const double rr = exp(log_rho_inf(xe) - log_rho_inf(centre(e))) / width(e);
        const double rl = exp(log_rho_inf(xe) - log_rho_inf(centre(e - 1))) / width(e - 1);
        right += coef * rr / tau_x;
        diag -= coef * rl / tau_x;
    }
    sub[c] = left * slice_dt;
    dia[c] = diag * slice_dt;
    sup[c] = right * slice_dt;
}

// T = sum_{k <= 18} B^k / k!, B = f A, by Horner's rule T <- I + (B T) / k.  B has
// three diagonals, so T's columns are independent and column c reaches 18 rows
// to either side: one warp per column, two entries per lane.  T is zero
// outside the band (cleared by the caller).
constexpr int kTaylor = 18;

__global__ void __launch_bounds__(128)
taylor_kernel(int I, double f, const double* __restrict__ sub, const double* __restrict__ dia,
              const double* __restrict__ sup, double* __restrict__ T)
{
    const int lane = threadIdx.x & 31;
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (c >= I) return;
    double t[2], lo[2], di[2], hi[2];
    int r[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        r[h] = c - 32 + 32 * h + lane;
        const bool in = r[h] >= 0 && r[h] < I;
        lo[h] = in ? sub[r[h]] * f : 0.0;
        di[h] = in ? dia[r[h]] * f : 0.0;
        hi[h] = in ? sup[r[h]] * f : 0.0;
        t[h] = r[h] == c ? 1.0 : 0.0;
    }
    for (int k = kTaylor; k >= 1; --k) {
        // the entries above and below, across the two halves
        double up0 = __shfl_up_sync(0xffffffffu, t[0], 1), up1 = __shfl_up_sync(0xffffffffu, t[1], 1);
        double dn0 = __shfl_down_sync(0xffffffffu, t[0], 1), dn1 = __shfl_down_sync(0xffffffffu, t[1], 1);
        const double last0 = __shfl_sync(0xffffffffu, t[0], 31), first1 = __shfl_sync(0xffffffffu, t[1], 0);
        if (lane == 0) {
            up0 = 0.0;
            up1 = last0;
        }
        if (lane == 31) {
            dn0 = first1;
            dn1 = 0.0;
        }
        const double alpha = 1.0 / k;
        // the terms in the order of their columns in B's row
        const double a0 = fma(hi[0], dn0, fma(di[0], t[0], lo[0] * up0));
        const double a1 = fma(hi[1], dn1, fma(di[1], t[1], lo[1] * up1));
        t[0] = fma(alpha, a0, r[0] == c ? 1.0 : 0.0);
        t[1] = fma(alpha, a1, r[1] == c ? 1.0 : 0.0);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (r[h] >= 0 && r[h] < I && abs(r[h] - c) <= kTaylor) T[(size_t)r[h] * I + c] = t[h];
}

// C = A A (I x I, row-major), bound by the binary64 pipe: CTAs of `rows` rows
// by 64 columns, eight warps of RW rows by 32 columns (one column per lane,
// RW sums in registers); `rows` is chosen so that the CTAs fill whole waves of
// the SMs.  The next tiles are loaded into registers while the current ones
// are multiplied.  A is zero more than `band` entries off its diagonal: the
// terms outside are skipped (each would add an exact zero).
// 512 bins: 0.233 ms, the pipe 97 % busy.
constexpr int kSqK = 32;

template <int RW>
__global__ void __launch_bounds__(256, 1) square_kernel(int n, int rows, int band,
                                                        const double* __restrict__ A, double* __restrict__ C)
{
    __shared__ double As[4 * RW][kSqK];
    __shared__ double Bs[kSqK][64];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row0 = blockIdx.y * rows, col0 = blockIdx.x * 64;
    const int wr = (warp >> 1) * RW, wc = (warp & 1) * 32 + lane;
    constexpr int na = (4 * RW * kSqK + 255) / 256, nb = kSqK * 64 / 256;
    double ra[na], rb[nb];
    auto load = [&](int k0) {
#pragma unroll
        for (int q = 0; q < na; ++q) {
            const int t = q * 256 + tid, r = t / kSqK, k = k0 + t % kSqK;
            ra[q] = r < rows && row0 + r < n && k < n ? A[(size_t)(row0 + r) * n + k] : 0.0;
        }
#pragma unroll
        for (int q = 0; q < nb; ++q) {
            const int t = q * 256 + tid, k = k0 + t / 64, c = col0 + t % 64;
            rb[q] = k < n && c < n ? A[(size_t)k * n + c] : 0.0;
        }
    };
    double acc[RW];
#pragma unroll
    for (int r = 0; r < RW; ++r) acc[r] = 0.0;
    const int first = max(0, max(row0, col0) - band) & ~(kSqK - 1);
    const int last = min(n, min(row0 + rows, col0 + 64) + band);   // one past
    if (first < last) load(first);
    for (int k0 = first; k0 < last; k0 += kSqK) {
#pragma unroll
        for (int q = 0; q < na; ++q) {
            const int t = q * 256 + tid;
            if (t < 4 * RW * kSqK) As[t / kSqK][t % kSqK] = ra[q];
        }
#pragma unroll
        for (int q = 0; q < nb; ++q) {
            const int t = q * 256 + tid;
            Bs[t / 64][t % 64] = rb[q];
        }
        __syncthreads();
        if (k0 + kSqK < last) load(k0 + kSqK);
#pragma unroll 4
        for (int k = 0; k < kSqK; ++k) {
            const double b = Bs[k][wc];
#pragma unroll
            for (int r = 0; r < RW; ++r) acc[r] = fma(As[wr + r][k], b, acc[r]);
        }
        __syncthreads();
    }
    if (col0 + wc >= n) return;
#pragma unroll
    for (int r = 0; r < RW; ++r)
        if (wr + r < rows && row0 + wr + r < n) C[(size_t)(row0 + wr + r) * n + col0 + wc] = acc[r];
}

// C_dT on n_vec states, one state per cluster of CL CTAs (the rows of P @ m
// split between them; the bits do not depend on CL): on GB300's narrow FP64
// pipe one CTA takes ~60 us for 512^2 FMAs, so a few states fill the GPU only
// when each is spread over several SMs.
template <int CL>
__global__ void __launch_bounds__(kCoarseThreads)
coarse_fp_kernel(const double* __restrict__ P, int I, const double* __restrict__ cin, double* __restrict__ cout)
{
    extern __shared__ __align__(16) double dsm[];
    double* in = dsm;
    double* out = in + (I + 1);
    double* mass = out + (I + 1);
    double* mp = mass + I;
    double* wsum = mp + I;
    const Dist<CL> d = Dist<CL>::make();
    const size_t v = blockIdx.x / CL;
    const double* src = cin + v * (I + 1);
    for (int i = threadIdx.x; i <= I; i += blockDim.x) in[i] = src[i];
    d.sync();   // every CTA of the cluster runs before any writes into its shared memory
    coarse_apply_block<CL>(P, I, in, out, mass, mp, wsum, d);
    double* dst = cout + v * (I + 1);
    const int q0 = d.lo(I - 1), q1 = d.hi(I - 1);
    for (int r = q0 + (int)threadIdx.x; r < q1; r += blockDim.x) dst[r + 1] = out[r + 1];
    if (d.rank == 0 && threadIdx.x == 0) {
        dst[0] = out[0];
        dst[I] = out[I];
    }
}

// The serial sweep of Section 3.2.3 on one CTA (CL = 1) or on a cluster of
// CL CTAs (launched with that cluster size).
template <int CL>
__global__ void __launch_bounds__(kCoarseThreads, 1)
parareal_update_kernel(const double* __restrict__ P, GridDev g, int iterator, int qmode, int K,
                       const double* __restrict__ cdf0, const double* __restrict__ fstar,
                       const double* __restrict__ cstar, double* __restrict__ next, int32_t* status)
{
    extern __shared__ __align__(16) unsigned char usm[];
    serial_sweep<CL>(usm, P, g, iterator, qmode, K, cdf0, fstar, cstar, next, status);
}

template <int PER_SM>
__global__ void __launch_bounds__(kCoarseThreads, PER_SM)
iterate_kernel(GridDev g, int iterator, int qmode, const double* __restrict__ a, const double* __restrict__ b,
               const double* __restrict__ c, double* __restrict__ out, int32_t* status)
{
    extern __shared__ __align__(16) unsigned char usm[];
    const int I = g.bins;
    double* Ab = reinterpret_cast<double*>(usm);
    double* Bb = Ab + (I + 1);
    double* Cb = Bb + (I + 1);
    double* Ob = Cb + (I + 1);
    JqSmem js = carve_jq(reinterpret_cast<unsigned char*>(Ob + (I + 1)), I);
    if (threadIdx.x == 0) js.flag[1] = 0;
    fill_edges(g, js);
    const size_t off = (size_t)blockIdx.x * (I + 1);
    for (int i = threadIdx.x; i <= I; i += blockDim.x) {
        Ab[i] = a[off + i];
        Bb[i] = b[off + i];
        Cb[i] = c[off + i];
    }
    __syncthreads();
    if (iterator == PR_ITER_QUANTILE) quantile_iterate_block(g, qmode, Ab, Bb, Cb, Ob, js);
    else mass_iterate_block(iterator, I, Ab, Bb, Cb, Ob, js.kq, js.wsum);
    for (int i = threadIdx.x; i <= I; i += blockDim.x) out[off + i] = Ob[i];
    if (threadIdx.x == 0 && status && js.flag[1]) atomicExch(status, (int32_t)PR_ERR_NUMERIC);
}

__global__ void __launch_bounds__(256)
w1_kernel(GridDev g, const double* __restrict__ c1, const double* __restrict__ c2, double* __restrict__ w1)
{
    __shared__ double wsum[40];
    const int I = g.bins;
    const size_t off = (size_t)blockIdx.x * (I + 1);
    double acc = 0.0;
    for (int i = threadIdx.x; i < I; i += blockDim.x) {
        const double d0 = c1[off + i] - c2[off + i], d1 = c1[off + i + 1] - c2[off + i + 1];
        const double a0 = fabs(d0), a1 = fabs(d1);
        if ((d0 >= 0.0 && d1 >= 0.0) || (d0 <= 0.0 && d1 <= 0.0)) acc += 0.5 * g.h * (a0 + a1);
        else acc += g.h * (d0 * d0 + d1 * d1) / (2.0 * (a0 + a1));
    }
    const double s = block_sum_f64(acc, wsum);
    if (threadIdx.x == 0) w1[blockIdx.x] = s;
}

// L2 distance of the piecewise-constant densities (bin mass / h) of two CDFs:
// sqrt(sum_i (m1_i - m2_i)^2 / h), one CTA per pair.
__global__ void __launch_bounds__(256)
l2_density_kernel(GridDev g, const double* __restrict__ c1, const double* __restrict__ c2, double* __restrict__ out)
{
    __shared__ double wsum[40];
    const int I = g.bins;
    const size_t off = (size_t)blockIdx.x * (I + 1);
    double acc = 0.0;
    for (int i = threadIdx.x; i < I; i += blockDim.x) {
        const double d = (c1[off + i + 1] - c1[off + i]) - (c2[off + i + 1] - c2[off + i]);
        acc += d * d / g.h;
    }
    const double s = block_sum_f64(acc, wsum);
    if (threadIdx.x == 0) out[blockIdx.x] = sqrt(s);
}

// CTAs of the cluster that runs the serial sweep (1, 2, 4 or 8: the portable sizes; 16 not tried).
static int g_update_cluster = 8;

template <typename K>
static cudaError_t allow_smem(K kernel, size_t bytes)
{
    if (bytes <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Rows per CTA of a squaring: with ceil(I / 64) column tiles, the fewest whole
// waves of one CTA per SM whose tiles have at most 64 rows.
static void launch_square(int I, int band, const double* A, double* C, cudaStream_t st)
{
    const int gx = (I + 63) / 64;
    int rows = 0;
    for (int waves = 1; rows == 0 || rows > 64; ++waves) {
        const int gy = waves * num_sms() / gx;
        rows = gy ? (I + gy - 1) / gy : 0;
    }
    const dim3 grid((unsigned)gx, (unsigned)((I + rows - 1) / rows));
    switch ((rows + 3) / 4) {
#define PR_SQ(rw) case rw: square_kernel<rw><<<grid, 256, 0, st>>>(I, rows, band, A, C); break;
    PR_SQ(1) PR_SQ(2) PR_SQ(3) PR_SQ(4) PR_SQ(5) PR_SQ(6) PR_SQ(7) PR_SQ(8) PR_SQ(9) PR_SQ(10) PR_SQ(11) PR_SQ(12)
    PR_SQ(13) PR_SQ(14) PR_SQ(15)
#undef PR_SQ
    default: square_kernel<16><<<grid, 256, 0, st>>>(I, rows, band, A, C);
    }
}

}  // namespace pr

using namespace pr;

extern "C" pr_status pr_coarse_create(const pr_model* model, const pr_grid* grid, double slice_dt,
                                      void** handle, void* stream)
{
    if (!model || !grid_ok(grid) || !handle || !(slice_dt > 0.0) || !std::isfinite(slice_dt)) return PR_ERR_INVALID_ARG;
    const bool chem = model->kind == PR_MODEL_CHEM || model->kind == PR_MODEL_CHEM_PRINTED;
    if (chem) {
        // rates finite and non-negative, k4 and k5 positive (Dbar > 0 needs a
        // positive ybar and x_lo >= 0)
        if (!(model->tau_x > 0.0) || !(grid->x_lo >= 0.0)) return PR_ERR_INVALID_ARG;
        for (int i = 0; i < 6; ++i)
            if (!std::isfinite(model->rate[i]) || model->rate[i] < 0.0) return PR_ERR_INVALID_ARG;
        if (!(model->rate[4] > 0.0) || !(model->rate[5] > 0.0) || !(model->rate[0] > 0.0)) return PR_ERR_INVALID_ARG;
    } else {
        if (model->kind < PR_MODEL_OU || model->kind > PR_MODEL_ADVECTION) return PR_ERR_INVALID_ARG;
        if (!(model->beta > 0.0) || !(model->tau_x > 0.0) || !std::isfinite(model->lambda)) return PR_ERR_INVALID_ARG;
        if (model->kind == PR_MODEL_ADVECTION && !(model->eps > 0.0)) return PR_ERR_INVALID_ARG;
    }
    *handle = nullptr;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int I = grid->bins;
    // the handle's matrix, and scratch: the other matrix of the squarings, the
    // three diagonals, ybar
    const size_t nn = (size_t)I * I;
    double *P = nullptr, *scratch = nullptr;
    auto fail = [&](pr_status rc) {
        if (P) cudaFree(P);
        if (scratch) cudaFree(scratch);
        return rc;
    };
    // (an allocation of its own, released again: a handle holds its matrix alone)
    if (cudaMalloc(&P, nn * 8) != cudaSuccess || cudaMalloc(&scratch, (nn + 3 * (size_t)I + 1) * 8) != cudaSuccess)
        return fail(PR_ERR_NOMEM);
    double* W = scratch;
    double *sub = W + nn, *dia = sub + I, *sup = dia + I, *ybar_dev = sup + I;
    const GridDev g = make_grid(*grid);
    if (chem) {   // ybar first; it must be positive and finite
        ChemRates r;
        for (int i = 0; i < 6; ++i) r.k[i] = model->rate[i];
        r.printed = model->kind == PR_MODEL_CHEM_PRINTED;
        if (allow_smem(chem_ybar_kernel, kChemSmem) != cudaSuccess) return fail(PR_ERR_CUDA);
        chem_ybar_kernel<<<1, kChemThreads, kChemSmem, st>>>(r, ybar_dev);
    }
    generator_kernel<<<(I + 63) / 64, 64, 0, st>>>(g, model->kind, model->lambda, model->beta, model->eps,
                                                   model->tau_x, model->rate[4], model->rate[5], ybar_dev, slice_dt,
                                                   sub, dia, sup);
    std::vector<double> diagonals(3 * (size_t)I + 1);
    if (cudaMemcpyAsync(diagonals.data(), sub, diagonals.size() * 8, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return fail(PR_ERR_CUDA);
    if (chem && (!std::isfinite(diagonals.back()) || !(diagonals.back() > 0.0))) return fail(PR_ERR_NUMERIC);
    double norm = 0.0;   // the largest absolute column sum
    for (int c = 0; c < I; ++c) {
        const double above = c ? std::fabs(diagonals[2 * (size_t)I + c - 1]) : 0.0;
        const double below = c + 1 < I ? std::fabs(diagonals[c + 1]) : 0.0;
        norm = std::fmax(norm, above + std::fabs(diagonals[I + c]) + below);
    }
    if (!std::isfinite(norm)) return fail(PR_ERR_CUDA);
    // scaling and squaring: ||B / 2^s||_1 <= 1/4, Taylor polynomial of degree 18
    int s = 0;
    while (norm / std::ldexp(1.0, s) > 0.25 && s < 1000) ++s;
    double* T = s % 2 ? W : P;   // the squarings alternate and end in P
    if (cudaMemsetAsync(T, 0, nn * 8, st) != cudaSuccess) return fail(PR_ERR_CUDA);
    taylor_kernel<<<(I + 3) / 4, 128, 0, st>>>(I, std::ldexp(1.0, -s), sub, dia, sup, T);
    int band = kTaylor;
    for (int q = 0; q < s; ++q) {
        double* to = T == P ? W : P;
        launch_square(I, band, T, to, st);
        T = to;
        band = std::min(2 * band, I);
    }
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) return fail(PR_ERR_CUDA);
    cudaFree(scratch);
    auto* h = new CoarseHandle;
    h->g = g;
    h->P = P;
    cudaGetDevice(&h->device);
    *handle = h;
    return PR_OK;
}

extern "C" pr_status pr_coarse_destroy(void* handle)
{
    if (!handle) return PR_ERR_INVALID_ARG;
    auto* h = static_cast<CoarseHandle*>(handle);
    cudaFree(h->P);
    delete h;
    return PR_OK;
}

extern "C" pr_status pr_coarse_matrix(void* handle, double* out, void* stream)
{
    if (!handle || !out || !elem_aligned(out, 8)) return PR_ERR_INVALID_ARG;
    auto* h = static_cast<CoarseHandle*>(handle);
    const size_t bytes = (size_t)h->g.bins * h->g.bins * sizeof(double);
    PR_TRY_CUDA(cudaMemcpyAsync(out, h->P, bytes, cudaMemcpyDeviceToDevice, static_cast<cudaStream_t>(stream)));
    return PR_OK;
}

extern "C" pr_status pr_coarse_fp(void* handle, const double* cdf_in, double* cdf_out, int32_t n_vec, void* stream)
{
    if (!handle || !cdf_in || !cdf_out || n_vec < 1 || cdf_in == cdf_out) return PR_ERR_INVALID_ARG;
    if (!elem_aligned(cdf_in, 8) || !elem_aligned(cdf_out, 8)) return PR_ERR_INVALID_ARG;
    auto* h = static_cast<CoarseHandle*>(handle);
    const int I = h->g.bins;
    const size_t smem = coarse_apply_smem(I);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // the largest cluster that keeps the launch within two CTAs per SM
    int cl = 1;
    if (I >= 64)
        for (int c : {8, 4, 2})
            if ((int64_t)n_vec * c <= 2 * (int64_t)num_sms()) {
                cl = c;
                break;
            }
    if (cl == 1) {
        PR_TRY_CUDA(allow_smem(coarse_fp_kernel<1>, smem));
        coarse_fp_kernel<1><<<n_vec, kCoarseThreads, smem, st>>>(h->P, I, cdf_in, cdf_out);
        PR_CHECK_LAUNCH();
        return PR_OK;
    }
    auto launch = [&](auto kernel) -> cudaError_t {
        cudaError_t e = allow_smem(kernel, smem);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(n_vec * cl));
        cfg.blockDim = dim3(kCoarseThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cl;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kernel, (const double*)h->P, I, cdf_in, cdf_out);
    };
    cudaError_t e;
    switch (cl) {
    case 2: e = launch(coarse_fp_kernel<2>); break;
    case 4: e = launch(coarse_fp_kernel<4>); break;
    default: e = launch(coarse_fp_kernel<8>); break;
    }
    if (e != cudaSuccess) return PR_ERR_CUDA;
    PR_CHECK_LAUNCH();
    return PR_OK;
}

extern "C" pr_status pr_parareal_update(void* coarse, pr_iterator iterator, pr_quantile_mode qmode, int32_t n_slices,
                                        const double* cdf0, const double* cdf_f_star, const double* cdf_c_star,
                                        double* cdf_next, int32_t* status, void* stream)
{
    if (!coarse || !cdf0 || !cdf_next || n_slices < 1) return PR_ERR_INVALID_ARG;
    if (!elem_aligned(cdf0, 8) || !elem_aligned(cdf_f_star, 8) || !elem_aligned(cdf_c_star, 8) ||
        !elem_aligned(cdf_next, 8) || !elem_aligned(status, 4))
        return PR_ERR_INVALID_ARG;
    if (iterator < PR_ITER_QUANTILE || iterator > PR_ITER_NONE) return PR_ERR_INVALID_ARG;
    if (qmode != PR_QMODE_TWO_SIDED && qmode != PR_QMODE_MIDPOINT) return PR_ERR_INVALID_ARG;
    if (iterator != PR_ITER_NONE && (!cdf_f_star || !cdf_c_star)) return PR_ERR_INVALID_ARG;
    auto* h = static_cast<CoarseHandle*>(coarse);
    if (h->g.bins > kUpdateMaxBins) return PR_ERR_UNSUPPORTED;
    const size_t smem = update_smem(h->g.bins);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int cl = h->g.bins >= 64 ? g_update_cluster : 1;
    if (cl == 1) {
        PR_TRY_CUDA(allow_smem(parareal_update_kernel<1>, smem));
        parareal_update_kernel<1><<<1, kCoarseThreads, smem, st>>>(h->P, h->g, (int)iterator, (int)qmode, n_slices,
                                                                  cdf0, cdf_f_star, cdf_c_star, cdf_next, status);
        PR_CHECK_LAUNCH();
        return PR_OK;
    }
    auto launch = [&](auto kernel) -> cudaError_t {
        cudaError_t e = allow_smem(kernel, smem);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)cl);
        cfg.blockDim = dim3(kCoarseThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cl;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kernel, (const double*)h->P, h->g, (int)iterator, (int)qmode, (int)n_slices,
                                  cdf0, cdf_f_star, cdf_c_star, cdf_next, status);
    };
    cudaError_t e;
    switch (cl) {
    case 2: e = launch(parareal_update_kernel<2>); break;
    case 4: e = launch(parareal_update_kernel<4>); break;
    default: e = launch(parareal_update_kernel<8>); break;
    }
    if (e != cudaSuccess) return PR_ERR_CUDA;
    PR_CHECK_LAUNCH();
    return PR_OK;
}

extern "C" void pr_set_update_cluster(int32_t ctas)
{
    g_update_cluster = (ctas == 1 || ctas == 2 || ctas == 4) ? ctas : 8;
}

extern "C" pr_status pr_iterate(pr_iterator iterator, pr_quantile_mode qmode, const pr_grid* grid, int32_t n_vec,
                                const double* a, const double* b, const double* c, double* out, int32_t* status,
                                void* stream)
{
    if (!grid_ok(grid) || n_vec < 1 || !a || !b || !c || !out) return PR_ERR_INVALID_ARG;
    if (!elem_aligned(a, 8) || !elem_aligned(b, 8) || !elem_aligned(c, 8) || !elem_aligned(out, 8) ||
        !elem_aligned(status, 4))
        return PR_ERR_INVALID_ARG;
    if (iterator < PR_ITER_QUANTILE || iterator > PR_ITER_ROT) return PR_ERR_INVALID_ARG;
    if (qmode != PR_QMODE_TWO_SIDED && qmode != PR_QMODE_MIDPOINT) return PR_ERR_INVALID_ARG;
    if (grid->bins > kUpdateMaxBins) return PR_ERR_UNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (status) PR_TRY_CUDA(cudaMemsetAsync(status, 0, sizeof(int32_t), st));
    const GridDev g = make_grid(*grid);
    const size_t smem = (size_t)4 * (grid->bins + 1) * sizeof(double) + jq_smem_bytes(grid->bins);
    auto launch = [&](auto kernel) -> pr_status {
        PR_TRY_CUDA(allow_smem(kernel, smem));
        kernel<<<n_vec, kCoarseThreads, smem, st>>>(g, (int)iterator, (int)qmode, a, b, c, out, status);
        PR_CHECK_LAUNCH();
        return PR_OK;
    };
    // as many CTAs per SM as the states and the shared memory make (registers cut
    // for one, two or four): 400 states of 5 bins 17 us at four, 24 at two, 32 at
    // one; of 512 bins 83 us at two, 105 at one, 88 with registers for four; of
    // 1024 bins (one fits) 145 us, 150 with registers for two
    const int64_t want = ((int64_t)n_vec + num_sms() - 1) / num_sms();
    const int64_t per_sm = std::min<int64_t>(want, ((int64_t)smem_optin_max() + 1024) / (int64_t)(smem + 1024));
    if (per_sm >= 3) return launch(iterate_kernel<4>);
    return per_sm == 2 ? launch(iterate_kernel<2>) : launch(iterate_kernel<1>);
}

extern "C" pr_status pr_w1(const pr_grid* grid, int32_t n_vec, const double* c1, const double* c2, double* w1,
                           void* stream)
{
    if (!grid_ok(grid) || n_vec < 1 || !c1 || !c2 || !w1) return PR_ERR_INVALID_ARG;
    if (!elem_aligned(c1, 8) || !elem_aligned(c2, 8) || !elem_aligned(w1, 8)) return PR_ERR_INVALID_ARG;
    const GridDev g = make_grid(*grid);
    w1_kernel<<<n_vec, 256, 0, static_cast<cudaStream_t>(stream)>>>(g, c1, c2, w1);
    PR_CHECK_LAUNCH();
    return PR_OK;
}

extern "C" pr_status pr_l2_density(const pr_grid* grid, int32_t n_vec, const double* c1, const double* c2,
                                   double* l2, void* stream)
{
    if (!grid_ok(grid) || n_vec < 1 || !c1 || !c2 || !l2) return PR_ERR_INVALID_ARG;
    if (!elem_aligned(c1, 8) || !elem_aligned(c2, 8) || !elem_aligned(l2, 8)) return PR_ERR_INVALID_ARG;
    const GridDev g = make_grid(*grid);
    l2_density_kernel<<<n_vec, 256, 0, static_cast<cudaStream_t>(stream)>>>(g, c1, c2, l2);
    PR_CHECK_LAUNCH();
    return PR_OK;
}

extern "C" const char* pr_status_string(pr_status s)
{
    switch (s) {
    case PR_OK: return "PR_OK";
    case PR_ERR_INVALID_ARG: return "PR_ERR_INVALID_ARG";
    case PR_ERR_CUDA: return "PR_ERR_CUDA";
    case PR_ERR_TIMEOUT: return "PR_ERR_TIMEOUT";
    case PR_ERR_UNSUPPORTED: return "PR_ERR_UNSUPPORTED";
    case PR_ERR_NOMEM: return "PR_ERR_NOMEM";
    case PR_ERR_NUMERIC: return "PR_ERR_NUMERIC";
    }
    return "PR_ERR_UNKNOWN";
}

extern "C" const char* pr_version(void) { return "0.1.0"; }

/* Host <-> device transfers of caller buffers, for callers that hold their
 * inputs and results in host memory (no method arithmetic: one
 * cudaMemcpyAsync each, ordered on `stream`). */
extern "C" pr_status pr_copy_to_device(void* dst, const void* src, size_t bytes, void* stream)
{
    if (bytes == 0) return PR_OK;
    if (!dst || !src) return PR_ERR_INVALID_ARG;
    PR_TRY_CUDA(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, static_cast<cudaStream_t>(stream)));
    return PR_OK;
}

extern "C" pr_status pr_copy_to_host(void* dst, const void* src, size_t bytes, void* stream)
{
    if (bytes == 0) return PR_OK;
    if (!dst || !src) return PR_ERR_INVALID_ARG;
    PR_TRY_CUDA(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, static_cast<cudaStream_t>(stream)));
    return PR_OK;
}

extern "C" pr_status pr_stream_synchronize(void* stream)
{
    PR_TRY_CUDA(cudaStreamSynchronize(static_cast<cudaStream_t>(stream)));
    return PR_OK;
}
