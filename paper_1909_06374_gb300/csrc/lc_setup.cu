// lc_setup.cu -- setup stage of the generator (Sec. 2.1, first two steps):
// TK95 spectrum of the Eq. 3 PSD, its FP64 variance, the target amplitudes,
// and the ERDF draws by inverse CDF.
#include <algorithm>

#include "lc_draw.cuh"
#include "lc_internal.h"

namespace lc {

constexpr int kSpecBlock = 256;
constexpr int kSpecPerThread = 4;
constexpr int kSpecTile = kSpecBlock * kSpecPerThread;  // bins per block

// TK95 (Sec. 2.1; Sec. 3.2.5): f_j = j/(N dt) (App. A), P_j from Eq. 3 with
// A = 1, X_0 = 0, X_j = sqrt(P_j/2)(g_re + i g_im) for 0 < j < N/2 and the
// real Nyquist bin sqrt(P_{N/2}) g_re; g from Box-Muller on the two uniforms
// of Philox block j (stream 0).  Also the block's share of
// sigma^2 = X_{N/2}^2 + 2 sum_{0<j<N/2} |X_j|^2 (Parseval for the
// unnormalised inverse transform), reduced in a fixed order, and the same sum
// with |X_j|^2 replaced by P_j (the variance the PSD implies, for PSD target
// amplitudes).  coeffs = fixed amplitude: X_j = sqrt(P_j) e^{2 pi i U2},
// X_{N/2} = +-sqrt(P_{N/2}) with the sign of cos(2 pi U2).

// Coefficient j of a curve (c = 1/(N dt f_br), nh = N/2).  y_j = f_j / f_br =
// j c; Eq. 3 as 1 / (e^{a_lo ln y} + e^{a_hi ln y}) (one logarithm for both
// terms); the amplitude sqrt(P/2) sqrt(-2 ln U1) as one square root: these are
// the FP64 operations that the FP64-rate-bound kernels spend their time on
// (conversions of 64-bit integers are among them: the uniforms, 2 U2 and j are
// put together from their bits, with one exact subtraction each at most).  Two
// kernels compute the coefficients and two add their squares, by the number of
// a class's curves, so every operation that nvcc could contract with another is
// written down: a curve's amplitudes do not depend on its batch.
__device__ __forceinline__ double2 tk_bin(const CurveDev& cv, double c, bool fixed, uint64_t j, uint64_t nh, double& P)
{
    const uint4 w = philox(j, cv.curve_id, 0u, cv.seed);
    const double U1 = unit_open_fast(w.x, w.y), U2 = unit_open_fast(w.z, w.w);
    const double lu = fixed ? 0.0 : log(U1);  // rad^2 = -2 lu
    double sn, cs;
    sincospi(__hiloint2double(__double2hiint(U2) + 0x100000, __double2loint(U2)), &sn, &cs);  // 2 U2, by its exponent
    // j as a double: the low word of 2^52 + j, less 2^52 (j < 2^32, exact)
    const double ly = log(__dmul_rn(__dsub_rn(__hiloint2double(0x43300000, (int)(uint32_t)j), 0x1p52), c));
    P = __ddiv_rn(1.0, __dadd_rn(exp(__dmul_rn(cv.a_lo, ly)), exp(__dmul_rn(cv.a_hi, ly))));
    if (j < nh) {
        const double a = fixed ? __dsqrt_rn(P) : __dsqrt_rn(__dmul_rn(-P, lu));
        return make_double2(__dmul_rn(a, cs), __dmul_rn(a, sn));
    }
    const double a = fixed ? __dsqrt_rn(P) : __dsqrt_rn(__dmul_rn(__dmul_rn(-2.0, P), lu));
    return make_double2(fixed ? (cs < 0.0 ? -a : a) : __dmul_rn(a, cs), 0.0);
}

// acc + the share of coefficient j in the series' variance.
__device__ __forceinline__ double tk_add_power(double acc, double2 X, uint64_t j, uint64_t nh)
{
    if (j < nh) return __fma_rn(2.0, __fma_rn(X.x, X.x, __dmul_rn(X.y, X.y)), acc);
    return __fma_rn(X.x, X.x, acc);
}

// Tree sums of the block's kSpecBlock values (fixed order), in thread 0.
__device__ __forceinline__ void spec_block_sums(double (&red)[kSpecBlock], double (&red_p)[kSpecBlock])
{
    __syncthreads();
    for (int s = kSpecBlock / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            red[threadIdx.x] += red[threadIdx.x + s];
            red_p[threadIdx.x] += red_p[threadIdx.x + s];
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kSpecBlock)
k_tk_spectrum(const CurveDev* __restrict__ curves, const int* __restrict__ cls_curves,
              int blocks_per_curve, double2* __restrict__ spec, double* __restrict__ partial,
              double* __restrict__ partial_p)
{
    const int ci = blockIdx.x / blocks_per_curve;
    const int jb = blockIdx.x % blocks_per_curve;
    const CurveDev cv = curves[cls_curves[ci]];
    const uint64_t nh = 1ull << (cv.log2n - 1);
    const double c = 1.0 / ((double)(1ull << cv.log2n) * cv.dt * cv.f_br);
    const bool fixed = cv.coeffs == 1;
    double acc = 0.0, acc_p = 0.0;
#pragma unroll
    for (int q = 0; q < kSpecPerThread; ++q) {
        const uint64_t j = (uint64_t)jb * kSpecTile + (uint64_t)q * kSpecBlock + threadIdx.x;
        if (j > nh) continue;
        double2 X = make_double2(0.0, 0.0);
        if (j > 0) {
            double P;
            X = tk_bin(cv, c, fixed, j, nh, P);
            acc = tk_add_power(acc, X, j, nh);
            acc_p += j < nh ? 2.0 * P : P;
        }
        spec[cv.offh + j] = X;
    }
    __shared__ double red[kSpecBlock], red_p[kSpecBlock];
    red[threadIdx.x] = acc;
    red_p[threadIdx.x] = acc_p;
    spec_block_sums(red, red_p);
    if (threadIdx.x == 0) {
        partial[blockIdx.x] = red[0];
        partial_p[blockIdx.x] = red_p[0];
    }
}

// The same coefficients for a few short curves, whose tiles would occupy few
// SMs (an SM's FP64 rate gives 1024 bins in 46 us): one bin per thread and
// kFewBins bins per block; the partial sums, in the order of k_tk_spectrum's,
// by k_tk_sums.  PSD targets need the sum of P as well and take k_tk_spectrum.
constexpr int kFewBins = 64;
__global__ void __launch_bounds__(kFewBins) k_tk_bins(const CurveDev* __restrict__ curves,
                                                      const int* __restrict__ cls_curves, int blocks_per_curve,
                                                      double2* __restrict__ spec)
{
    const CurveDev& cv = curves[cls_curves[blockIdx.x / blocks_per_curve]];
    const uint64_t j = (uint64_t)(blockIdx.x % blocks_per_curve) * kFewBins + threadIdx.x;
    const uint64_t nh = 1ull << (cv.log2n - 1);
    if (j > nh) return;
    double2 X = make_double2(0.0, 0.0);
    if (j > 0) {
        double P;
        X = tk_bin(cv, 1.0 / ((double)(1ull << cv.log2n) * cv.dt * cv.f_br), cv.coeffs == 1, j, nh, P);
    }
    spec[cv.offh + j] = X;
}

__global__ void __launch_bounds__(kSpecBlock) k_tk_sums(const CurveDev* __restrict__ curves,
                                                        const int* __restrict__ cls_curves, int blocks_per_curve,
                                                        const double2* __restrict__ spec,
                                                        double* __restrict__ partial, double* __restrict__ partial_p)
{
    const int jb = blockIdx.x % blocks_per_curve;
    const CurveDev& cv = curves[cls_curves[blockIdx.x / blocks_per_curve]];
    const uint64_t nh = 1ull << (cv.log2n - 1);
    double2 X[kSpecPerThread];
#pragma unroll
    for (int q = 0; q < kSpecPerThread; ++q) {
        const uint64_t j = (uint64_t)jb * kSpecTile + (uint64_t)q * kSpecBlock + threadIdx.x;
        X[q] = j > 0 && j <= nh ? spec[cv.offh + j] : make_double2(0.0, 0.0);
    }
    double acc = 0.0;
#pragma unroll
    for (int q = 0; q < kSpecPerThread; ++q) {
        const uint64_t j = (uint64_t)jb * kSpecTile + (uint64_t)q * kSpecBlock + threadIdx.x;
        if (j > nh || j == 0) continue;
        acc = tk_add_power(acc, X[q], j, nh);
    }
    __shared__ double red[kSpecBlock], red_p[kSpecBlock];
    red[threadIdx.x] = acc;
    red_p[threadIdx.x] = 0.0;
    spec_block_sums(red, red_p);
    if (threadIdx.x == 0) {
        partial[blockIdx.x] = red[0];
        partial_p[blockIdx.x] = 0.0;
    }
}

// sigma (realised) and sigma_P (PSD) of each curve of a class: the partial
// sums added in block order.
constexpr int kSigmaWarps = 4;
__global__ void __launch_bounds__(32 * kSigmaWarps) k_sigma(const int* __restrict__ cls_curves, int ncurves,
                                                            int blocks_per_curve, const double* __restrict__ partial,
                                                            const double* __restrict__ partial_p,
                                                            double* __restrict__ sigma, double* __restrict__ sigma_p)
{
    // one warp per curve: 32 partials of each sum are loaded at once, then lane
    // 0 adds one sum and lane 1 the other (one thread per curve loading and
    // adding in turn: 4.3 ms for the 32769 partials of a 2^26 curve)
    __shared__ double v[kSigmaWarps][2][33];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ci = blockIdx.x * kSigmaWarps + w;
    if (ci >= ncurves) return;
    const double* __restrict__ p0 = partial + (size_t)ci * blocks_per_curve;
    const double* __restrict__ p1 = partial_p + (size_t)ci * blocks_per_curve;
    double s = 0.0;
    double n0 = lane < blocks_per_curve ? p0[lane] : 0.0, n1 = lane < blocks_per_curve ? p1[lane] : 0.0;
    for (int b = 0; b < blocks_per_curve; b += 32) {
        v[w][0][lane] = n0;
        v[w][1][lane] = n1;
        __syncwarp();
        if (b + 32 + lane < blocks_per_curve) {  // the next ones, while these are added
            n0 = p0[b + 32 + lane];
            n1 = p1[b + 32 + lane];
        }
        const int n = min(32, blocks_per_curve - b);
        if (lane < 2)
            for (int q = 0; q < n; ++q) s += v[w][lane][q];
        __syncwarp();
    }
    if (lane == 0) sigma[cls_curves[ci]] = sqrt(s);
    if (lane == 1) sigma_p[cls_curves[ci]] = sqrt(s);
}

// Target amplitudes of the normalised TK95 series: A_j = |X_j| / sigma, A_0 = 0;
// with PSD targets A_j = sqrt(P_j) / sigma_P.
// One block covers kAmpTile bins of one curve (blockIdx.x = curve of the
// class x chunks per curve + chunk), so no thread divides by N/2 + 1.
constexpr int kAmpTile = 1024;
template <typename T>
__global__ void __launch_bounds__(256) k_amplitudes(const CurveDev* __restrict__ curves,
                                                    const int* __restrict__ cls_curves, int chunks, uint32_t log2n,
                                                    const double2* __restrict__ spec,
                                                    const double* __restrict__ sigma,
                                                    const double* __restrict__ sigma_p, T* __restrict__ A)
{
    const uint64_t nh1 = (1ull << (log2n - 1)) + 1;
    const int c = cls_curves[blockIdx.x / chunks];
    const CurveDev& cv = curves[c];
    const uint64_t j0 = (uint64_t)(blockIdx.x % chunks) * kAmpTile;
    const bool psd = cv.targets == 1;
    const double inv = 1.0 / (psd ? sigma_p[c] : sigma[c]);
    const double cy = 1.0 / ((double)(1ull << log2n) * cv.dt * cv.f_br);
    for (uint64_t j = j0 + threadIdx.x; j < j0 + kAmpTile && j < nh1; j += blockDim.x) {
        double a = 0.0;
        if (j > 0 && psd) {
            const double ly = log((double)j * cy);
            a = sqrt(1.0 / (exp(cv.a_lo * ly) + exp(cv.a_hi * ly))) * inv;
        } else if (j > 0) {
            const double2 X = spec[cv.offh + j];
            a = sqrt(X.x * X.x + X.y * X.y) * inv;
        }
        A[cv.offh + j] = (T)a;
    }
}

__global__ void k_erdf_constants(const CurveDev* __restrict__ curves, int ncurves, ErdfConst* __restrict__ out)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncurves) return;
    ErdfConst k = erdf_constants(curves[c]);
    k.f = draw_constants(k);
    out[c] = k;
}

// Tables of the float draws, copied to shared memory by every block.
__device__ const DrawTables g_draw_tables = make_draw_tables();
__device__ __forceinline__ void load_draw_tables(DrawTables* t)
{
    for (int i = threadIdx.x; i < (int)(sizeof(DrawTables) / 4); i += blockDim.x)
        ((uint32_t*)t)[i] = ((const uint32_t*)&g_draw_tables)[i];
}

// The FP64 sequence for the draws that the float path leaves undecided.
__device__ __noinline__ float erdf_draw_decide(const ErdfConst& k, double U) { return (float)erdf_draw(k, U); }
__device__ __noinline__ float erdf_draw_tab_decide(const double* F, double umin, double h, double lo, double hi,
                                                   double U)
{
    return (float)erdf_draw_tab(F, umin, h, lo, hi, U);
}

// ERDF draws (Sec. 2.1 second step; inverse CDF instead of slice sampling):
// draw k uses Philox block k/2 of stream 1, words (w0,w1) for even k and
// (w2,w3) for odd k; lambda is computed in FP64.
__global__ void k_erdf_draws_fp64(const CurveDev* __restrict__ curves, const int* __restrict__ cls_curves,
                             int ncurves, uint32_t log2n, const ErdfConst* __restrict__ ek,
                             double* __restrict__ x)
{
    const uint64_t half = 1ull << (log2n - 1);
    const uint64_t total = (uint64_t)ncurves * half;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const int ci = (int)(t >> (log2n - 1));
        const uint64_t q = t & (half - 1);
        const int c = cls_curves[ci];
        const CurveDev& cv = curves[c];
        if (cv.kind != 0) continue;  // tabulated shapes: k_erdf_draws_tab
        const ErdfConst k = ek[c];
        const uint4 w = philox(q, cv.curve_id, 1u, cv.seed);
        const double l0 = erdf_draw(k, unit_open(w.x, w.y));
        const double l1 = erdf_draw(k, unit_open(w.z, w.w));
        x[cv.off + 2 * q] = l0;
        x[cv.off + 2 * q + 1] = l1;
    }
}

// The same draws rounded to float (lc_draw.cuh): a block inverts `pairs`
// consecutive Philox blocks of one curve.  Bound by the FP64 pipe still (5 to 9
// operations per draw, ~120 before) and by issue: 255 curves of 2^16 samples
// 5.11 -> 0.65 ms, the 1.9e8 draws of a ragged batch 57.9 -> 7.2 ms.
__global__ void __launch_bounds__(256) k_erdf_draws(const CurveDev* __restrict__ curves,
                                                    const int* __restrict__ cls_curves, int chunks, uint32_t pairs,
                                                    const ErdfConst* __restrict__ ek, float* __restrict__ x)
{
    __shared__ DrawTables t;
    __shared__ ErdfConst k;
    load_draw_tables(&t);
    const int c = cls_curves[blockIdx.x / chunks];
    const CurveDev& cv = curves[c];
    if (cv.kind != 0) return;  // tabulated shapes: k_erdf_draws_tab
    for (int i = threadIdx.x; i < (int)(sizeof(ErdfConst) / 4); i += blockDim.x)
        ((uint32_t*)&k)[i] = ((const uint32_t*)(ek + c))[i];
    const uint64_t cid = cv.curve_id, seed = cv.seed;
    const uint32_t q0 = (uint32_t)(blockIdx.x % chunks) * pairs;
    float2* __restrict__ out = (float2*)(x + cv.off);
    __syncthreads();
    const DrawConst d = k.f;
    for (uint32_t q = q0 + threadIdx.x; q < q0 + pairs; q += blockDim.x) {
        const uint4 w = philox(q, cid, 1u, seed);
        const double U0 = unit_open_fast(w.x, w.y), U1 = unit_open_fast(w.z, w.w);
        float l0, l1;
        const bool ok0 = erdf_draw_fast(t, k, d, U0, l0);
        const bool ok1 = erdf_draw_fast(t, k, d, U1, l1);
        if (!ok0) l0 = erdf_draw_decide(k, U0);
        if (!ok1) l1 = erdf_draw_decide(k, U1);
        out[q] = make_float2(l0, l1);
    }
}

// CDF tables of the tabulated ERDF shapes, one block per curve: Simpson's rule
// on every interval, (f(u_k) + 4 f(u_k + h/2) + f(u_{k+1})) h/6 with u_k = umin
// + k h, in parallel, then their sum in order by one thread.  Bound by the FP64
// rate: 2 densities per interval instead of 3 (766 curves, 1.55 -> 1.13 ms).
__global__ void __launch_bounds__(256) k_erdf_table(const CurveDev* __restrict__ curves,
                                                    const int* __restrict__ tab_curves, double* __restrict__ tab)
{
    __shared__ double I[kErdfTable];
    const CurveDev& cv = curves[tab_curves[blockIdx.x]];
    {
        // a thread's intervals are consecutive, so an interval's right end
        // point is the next one's left (the same u, hence the same density)
        constexpr int kPer = kErdfTable / 256;
        const double h = erdf_table_step(cv);
        const double h6 = __ddiv_rn(h, 6.0);
        const int k0 = threadIdx.x * kPer;
        double u0 = __dadd_rn(cv.umin, __dmul_rn((double)k0, h)), f0 = erdf_density(cv, u0);
        for (int k = k0; k < k0 + kPer; ++k) {
            const double u1 = __dadd_rn(cv.umin, __dmul_rn((double)(k + 1), h)), f1 = erdf_density(cv, u1);
            double sum = __dadd_rn(f0, __dmul_rn(4.0, erdf_density(cv, __dadd_rn(u0, __dmul_rn(0.5, h)))));
            sum = __dadd_rn(sum, f1);
            I[k] = __dmul_rn(sum, h6);
            u0 = u1;
            f0 = f1;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double* F = tab + cv.tab;
        double acc = 0.0;
        F[0] = 0.0;
#pragma unroll 8
        for (int k = 0; k < kErdfTable; ++k) {
            acc = __dadd_rn(acc, I[k]);
            F[k + 1] = acc;
        }
    }
}

// Draws of the tabulated shapes: a block stages its curve's table in shared
// memory and inverts `pairs` Philox blocks (same stream and word use as
// k_erdf_draws); float draws by lc_draw.cuh (766 curves of 2^16 samples 5.57
// -> 1.98 ms).
template <typename T>
__global__ void __launch_bounds__(256) k_erdf_draws_tab(const CurveDev* __restrict__ curves,
                                                        const int* __restrict__ tab_cls_curves, int chunks,
                                                        uint64_t pairs, const ErdfConst* __restrict__ ek,
                                                        const double* __restrict__ tab, T* __restrict__ x)
{
    __shared__ double F[kErdfTable + 1];
    __shared__ DrawTables t;
    const int c = tab_cls_curves[blockIdx.x / chunks];
    const uint64_t q0 = (uint64_t)(blockIdx.x % chunks) * pairs;
    const CurveDev& cv = curves[c];
    for (int i = threadIdx.x; i <= kErdfTable; i += blockDim.x) F[i] = tab[cv.tab + i];
    if (sizeof(T) == 4) load_draw_tables(&t);
    __syncthreads();
    const double klo = ek[c].lo, khi = ek[c].hi, umin = cv.umin;
    const DrawConst d = ek[c].f;
    const double h = erdf_table_step(cv);
    for (uint64_t q = q0 + threadIdx.x; q < q0 + pairs; q += blockDim.x) {
        const uint4 w = philox(q, cv.curve_id, 1u, cv.seed);
        const double U0 = unit_open_fast(w.x, w.y), U1 = unit_open_fast(w.z, w.w);
        T l0, l1;
        if constexpr (sizeof(T) == 4) {
            const bool ok0 = erdf_draw_tab_fast(t, F, umin, h, d, U0, l0);
            const bool ok1 = erdf_draw_tab_fast(t, F, umin, h, d, U1, l1);
            if (!ok0) l0 = erdf_draw_tab_decide(F, umin, h, klo, khi, U0);
            if (!ok1) l1 = erdf_draw_tab_decide(F, umin, h, klo, khi, U1);
        } else {
            l0 = erdf_draw_tab(F, umin, h, klo, khi, U0);
            l1 = erdf_draw_tab(F, umin, h, klo, khi, U1);
        }
        x[cv.off + 2 * q] = l0;
        x[cv.off + 2 * q + 1] = l1;
    }
}

// ------------------------------------------------------------ launchers
static int grid_for(uint64_t work, int block)
{
    uint64_t g = (work + block - 1) / block;
    const uint64_t cap = 152ull * 16;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

int spec_blocks_per_curve(uint32_t log2n)
{
    const uint64_t nh1 = (1ull << (log2n - 1)) + 1;
    return (int)((nh1 + kSpecTile - 1) / kSpecTile);
}

int launch_tk_spectrum(const Plan& p, const ClassInfo& k, cudaStream_t st)
{
    const int bpc = spec_blocks_per_curve(k.log2n);
    double* part = p.d_partial + k.partial_off;
    double* part_p = p.d_partial + p.partial_total + k.partial_off;
    // fewer tiles than two per SM: spread over the GPU bin by bin
    bool few = (int64_t)k.ncurves * bpc < 152 * 2;
    for (int i = 0; few && i < k.ncurves; ++i) few = p.h_curves[k.h_curves[i]].targets == 0;
    if (few) {
        const int bb = (int)(((1ull << (k.log2n - 1)) + kFewBins) / kFewBins);
        k_tk_bins<<<k.ncurves * bb, kFewBins, 0, st>>>(p.d_curves, k.d_curves, bb, p.d_spec);
        k_tk_sums<<<k.ncurves * bpc, kSpecBlock, 0, st>>>(p.d_curves, k.d_curves, bpc, p.d_spec, part, part_p);
    } else {
        k_tk_spectrum<<<k.ncurves * bpc, kSpecBlock, 0, st>>>(p.d_curves, k.d_curves, bpc, p.d_spec, part, part_p);
    }
    k_sigma<<<(k.ncurves + kSigmaWarps - 1) / kSigmaWarps, 32 * kSigmaWarps, 0, st>>>(
        k.d_curves, k.ncurves, bpc, part, part_p, p.d_sigma, p.d_sigma + p.ncurves);
    return few ? 3 : 2;
}

template <typename T>
void launch_amplitudes(const Plan& p, const ClassInfo& k, cudaStream_t st)
{
    const uint64_t nh1 = (1ull << (k.log2n - 1)) + 1;
    const int chunks = (int)((nh1 + kAmpTile - 1) / kAmpTile);
    k_amplitudes<T><<<k.ncurves * chunks, 256, 0, st>>>(p.d_curves, k.d_curves, chunks, k.log2n, p.d_spec,
                                                        p.d_sigma, p.d_sigma + p.ncurves, (T*)p.d_A);
}

void launch_erdf_constants(const Plan& p, cudaStream_t st)
{
    k_erdf_constants<<<(int)((p.ncurves + 127) / 128), 128, 0, st>>>(p.d_curves, (int)p.ncurves, p.d_erdf);
}

void launch_erdf_tables(const Plan& p, cudaStream_t st)
{
    if (p.ntab) k_erdf_table<<<(int)p.ntab, 256, 0, st>>>(p.d_curves, p.d_tab_curves, p.d_tab);
}

template <typename T>
void launch_erdf_draws(const Plan& p, const ClassInfo& k, cudaStream_t st)
{
    if (k.ntab < k.ncurves) {
        const uint64_t work = (uint64_t)k.ncurves << (k.log2n - 1);
        if constexpr (sizeof(T) == 8) {
            k_erdf_draws_fp64<<<grid_for(work, 256), 256, 0, st>>>(p.d_curves, k.d_curves, k.ncurves, k.log2n,
                                                                   p.d_erdf, (double*)p.d_x);
        } else {
            // eight Philox blocks per thread, fewer while the grid would not fill the GPU
            const uint64_t half = 1ull << (k.log2n - 1);
            uint64_t pairs = std::min<uint64_t>(half, 2048);
            while (pairs > 256 && work / pairs < 152 * 8) pairs /= 2;
            const int chunks = (int)(half / pairs);
            k_erdf_draws<<<k.ncurves * chunks, 256, 0, st>>>(p.d_curves, k.d_curves, chunks, (uint32_t)pairs,
                                                             p.d_erdf, (float*)p.d_x);
        }
    }
    if (k.ntab) {
        // up to 8192 Philox blocks (16384 draws) per block of threads, fewer
        // while the grid would not fill the GPU
        const uint64_t half = 1ull << (k.log2n - 1);
        uint64_t pairs = half < 8192 ? half : 8192;
        while (pairs > 512 && (half / pairs) * k.ntab < 152 * 4) pairs /= 2;
        const int chunks = (int)(half / pairs);
        k_erdf_draws_tab<T><<<k.ntab * chunks, 256, 0, st>>>(p.d_curves, k.d_tab_curves, chunks, pairs, p.d_erdf,
                                                             p.d_tab, (T*)p.d_x);
    }
}

template void launch_amplitudes<float>(const Plan&, const ClassInfo&, cudaStream_t);
template void launch_amplitudes<double>(const Plan&, const ClassInfo&, cudaStream_t);
template void launch_erdf_draws<float>(const Plan&, const ClassInfo&, cudaStream_t);
template void launch_erdf_draws<double>(const Plan&, const ClassInfo&, cudaStream_t);

}  // namespace lc
