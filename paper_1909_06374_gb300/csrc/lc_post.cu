// lc_post.cu -- estimators of App. A on batches of generated series: the
// periodogram (Eq. A2, and the fractional rms normalisation of Eq. A4) and the
// structure function (Eq. A6), used for the ensemble checks of Sec. 3.2.5.
//
// Both read a series laid out like a plan's state (curve c at sum_{c'<c} N),
// e.g. the output of lc_generate.  The periodogram reuses the plan's
// half-length complex FFT (the series packed as z_m = x_{2m} + i x_{2m+1}) and
// unpacks |X_j|^2; the structure function is a direct sum over the pairs at
// each lag.
#include <algorithm>

#include "lc_internal.h"

namespace lc {

// |X_j|^2 of a real series from its packed half-length transform Z:
// X_0 = Re Z_0 + Im Z_0, X_M = Re Z_0 - Im Z_0, X_{M/2} = conj Z_{M/2}, and for
// 0 < k < M/2: X_k = E + W^k O, X_{M-k} = conj(E - W^k O) with
// E = (Z_k + conj Z_{M-k})/2, O = (Z_k - conj Z_{M-k})/(2i).
// P_j = |X_j|^2 2/N^2 (Eq. A2) or |X_j|^2 2 dt N / X_0^2 (Eq. A4, X_0 = N mu).
//
// One block takes `pairs` conjugate pairs of one curve (launch_periodogram).  A
// float bin's power takes two FP64 operations (three for Eq. A4) of the 2 per
// clock and SM, whose pipe is the limit (86% busy): its conversions and Eq. A2's scale, a power of two, are put
// together from bits.  2048 curves of 2^16 samples, transform included: 1.11 ms with FP64
// conversions and scaling (Eq. A4, with a division per bin: 1.81), 0.846 (0.902)
// with these.  Two pairs per thread: the kernel alone takes 405 us there, with
// 1, 4 or 16 pairs 440, 546 and 535 (256 FP64 curves of 2^16: 179, 184, 178 and
// 184).
constexpr uint32_t kPgPairs = 512;

// (x^2 + y^2) 2^-sh, rounded once: a float's square is exact in FP64.
__device__ __forceinline__ double power_of(float x, float y, int sh)
{
    const uint32_t a = __float_as_uint(x) & 0x7fffffffu, b = __float_as_uint(y) & 0x7fffffffu;
    if (a - 0x00800000u >= 0x7f000000u || b - 0x00800000u >= 0x7f000000u)  // zeros, subnormal, Inf, NaN
        return ((double)x * x + (double)y * y) * pow2_scale(1.0, -sh);
    // normal floats' bits, the exponent rebased: |x| and |x| 2^-sh in FP64
    const uint32_t one = 896u << 20, scaled = (uint32_t)(896 - sh) << 20;
    const double xd = __hiloint2double((int)((a >> 3) + one), (int)(a << 29));
    const double yd = __hiloint2double((int)((b >> 3) + one), (int)(b << 29));
    const double xs = __hiloint2double((int)((a >> 3) + scaled), (int)(a << 29));
    const double ys = __hiloint2double((int)((b >> 3) + scaled), (int)(b << 29));
    return __fma_rn(xd, xs, __dmul_rn(yd, ys));
}
__device__ __forceinline__ double power_of(double x, double y, int sh)
{
    return (x * x + y * y) * pow2_scale(1.0, -sh);
}

template <typename T>
__global__ void __launch_bounds__(256) k_periodogram(const int* __restrict__ cls_curves,
                                                     const CurveDev* __restrict__ curves, uint32_t pairs,
                                                     uint32_t log2M, const void* __restrict__ tw,
                                                     const void* __restrict__ Zin, int rms, double* __restrict__ P)
{
    using V = cplx<T>;
    const uint32_t half = 1u << (log2M - 1);
    const uint32_t M = 1u << log2M;
    const double nd = 2.0 * (double)M;
    const V* __restrict__ rt = (const V*)tw;
    const uint32_t chunks = max(half / pairs, 1u);
    const CurveDev& cv = curves[cls_curves[blockIdx.x / chunks]];
    const uint32_t k0 = blockIdx.x % chunks * pairs;
    const V* __restrict__ Z = (const V*)Zin + (cv.off >> 1);
    double* __restrict__ out = P + cv.offh;
    // 2 / N^2 = 2^-sh, or the rms normalisation (by one thread: its division is
    // as many FP64 operations as a pair's bins)
    const int sh = rms ? 0 : 2 * (int)log2M + 1;
    __shared__ double rms_scale;
    if (rms) {
        if (threadIdx.x == 0) {
            const V z0 = Z[0];
            const double X0 = (double)(z0.x + z0.y);
            rms_scale = 2.0 * cv.dt * nd / (X0 * X0);
        }
        __syncthreads();
    }
    const double scale = rms ? rms_scale : 1.0;
    auto power = [&](T x, T y) -> double {
        const double v = power_of(x, y, sh);
        return rms ? v * scale : v;
    };
    const uint32_t k1 = min(half, k0 + pairs);
#pragma unroll 4
    for (uint32_t k = k0 + threadIdx.x; k < k1; k += 256) {
        if (k == 0) {
            const V z0 = Z[0];
            const V zh = Z[half];
            out[0] = power(z0.x + z0.y, (T)0);
            out[M] = power(z0.x - z0.y, (T)0);
            out[half] = power(zh.x, zh.y);
        } else {
            const V za = Z[k], zb = Z[M - k];
            const V W = rt[k];
            V E; E.x = (T)0.5 * (za.x + zb.x); E.y = (T)0.5 * (za.y - zb.y);
            V O; O.x = (T)0.5 * (za.y + zb.y); O.y = (T)-0.5 * (za.x - zb.x);
            const V WO = cmul(W, O);
            const V Xk = cadd(E, WO);
            const V Xm = csub(E, WO);  // conj(X_{M-k}); the modulus is the same
            out[k] = power(Xk.x, Xk.y);
            out[M - k] = power(Xm.x, Xm.y);
        }
    }
}

// SF(tau)^2 of Eq. A6 of FP32 curves: the mean over the N - tau pairs of
// (x_i - x_{i+tau})^2, added up as runs of up to 64 squares 256 samples apart
// in float, then the runs of a segment (sum_runs), then the segments in FP64.
// A block takes one segment of 256 MM samples of a curve, MM = 64 or N/256,
// and `per` of the lags: its x_i stay in registers over all of them, so a pair
// costs one load (of x_{i+tau}, mostly from L1: neighbouring lags read
// overlapping windows), a subtraction and a multiply-add, all of a run's loads
// independent.  256 curves of 2^16 samples at 53 lags: 0.23 ms (3.8e12
// pairs/s), bound by the loads through L1 (68% of its throughput, 96% of them
// hits; issue 57%); one block per (curve, lag) that walks the whole curve, two
// loads per pair and nothing kept: 3.14 ms.
constexpr int kSfBatch = 16;  // lags whose runs are added up together

// Sum of the 256 runs at r (>= 0, or NaN) by a warp, in lane 0.  Added as
// integers, 2^-54 of the largest run's power of two as unit: exact for the runs
// above 2^-31 of it, and below 2^-46 of the sum in all (255 FP64 additions:
// 2^-45), over the whole range of float.  256 curves of 2^16 samples at 53 lags
// 232 us, with FP64 additions (16 clocks per warp operation) 258; 2000 curves of
// 2^10 at 27 lags 61 against 117.  Infinities and NaN go there.
__device__ __forceinline__ double sum_runs(const float* r)
{
    const int lane = threadIdx.x & 31;
    uint32_t top = 0u;
#pragma unroll
    for (int q = 0; q < 8; ++q) top = max(top, __float_as_uint(r[lane + 32 * q]));
    top = __reduce_max_sync(0xffffffffu, top);
    if (top >= 0x7f800000u) {
        double sum = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) sum += (double)r[lane + 32 * q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
        return sum;
    }
    const uint32_t et = max(top >> 23, 1u);
    unsigned long long acc = 0u;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const uint32_t v = __float_as_uint(r[lane + 32 * q]), e = v >> 23;
        const uint32_t m = e ? (v & 0x7fffffu) | 0x800000u : v;
        acc += ((unsigned long long)m << 31) >> min(et - max(e, 1u), 63u);
    }
    // the lanes' 58 bits in three parts whose sums fit a word
    const uint32_t p0 = __reduce_add_sync(0xffffffffu, (uint32_t)acc & 0x7ffffffu);
    const uint32_t p1 = __reduce_add_sync(0xffffffffu, (uint32_t)(acc >> 27) & 0x7ffffffu);
    const uint32_t p2 = __reduce_add_sync(0xffffffffu, (uint32_t)(acc >> 54));
    acc = p0 + ((unsigned long long)p1 << 27) + ((unsigned long long)p2 << 54);
    return (double)acc * __hiloint2double((int)((1023u + et - 181u) << 20), 0);
}

template <int MM>
__global__ void __launch_bounds__(256, 2)
    k_structure_runs(const int* __restrict__ cls_curves, const CurveDev* __restrict__ curves, uint32_t log2n, int segs,
                     int groups, int per, int nlags, const uint32_t* __restrict__ lags, const float* __restrict__ x,
                     double* __restrict__ part, double* __restrict__ out)
{
    __shared__ float sh[kSfBatch][256];
    const int t = threadIdx.x;
    const int g = (int)(blockIdx.x % (uint32_t)groups);
    const int seg = (int)((blockIdx.x / (uint32_t)groups) % (uint32_t)segs);
    const int c = cls_curves[blockIdx.x / (uint32_t)groups / (uint32_t)segs];
    const uint32_t n = 1u << log2n, s0 = (uint32_t)seg * (256u * MM), i0 = s0 + (uint32_t)t;
    const uint64_t off = curves[c].off;
    const float* __restrict__ xc = x + off;
    const int l0 = g * per, l1 = min(nlags, l0 + per);
    float xi[MM];
#pragma unroll
    for (int m = 0; m < MM; ++m) xi[m] = i0 + 256u * m < n ? xc[i0 + 256u * m] : 0.0f;
    for (int lb = l0; lb < l1; lb += kSfBatch) {
        const int nb = min(kSfBatch, l1 - lb);
        for (int b = 0; b < nb; ++b) {
            const uint32_t tau = lags[lb + b], np = n - tau;
            const float* __restrict__ xt = xc + i0 + tau;
            float run = 0.0f;
            if (s0 + 256u * MM <= np) {
#pragma unroll
                for (int m = 0; m < MM; ++m) {
                    const float d = xi[m] - xt[256 * m];
                    run += d * d;
                }
            } else {
#pragma unroll 8
                for (int m = 0; m < MM; ++m) {
                    if (i0 + 256u * m < np) {
                        const float d = xc[i0 + 256u * m] - xt[256 * m];
                        run += d * d;
                    }
                }
            }
            sh[b][t] = run;
        }
        __syncthreads();
        for (int b = t >> 5; b < nb; b += 8) {
            const double sum = sum_runs(sh[b]);
            if ((t & 31) == 0) {
                if (segs == 1) out[(size_t)c * nlags + lb + b] = sum / (double)(n - lags[lb + b]);
                else part[off / 2 + (size_t)(lb + b) * segs + seg] = sum;
            }
        }
        __syncthreads();
    }
}

// The segments' sums of one (curve, lag) per warp, in a fixed order.
__global__ void __launch_bounds__(128) k_structure_sum(const int* __restrict__ cls_curves,
                                                       const CurveDev* __restrict__ curves, int ncurves,
                                                       uint32_t log2n, int segs, int nlags,
                                                       const uint32_t* __restrict__ lags,
                                                       const double* __restrict__ part, double* __restrict__ out)
{
    const int lane = threadIdx.x & 31;
    const size_t w = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= (size_t)ncurves * nlags) return;
    const int c = cls_curves[w / nlags], l = (int)(w % nlags);
    const double* __restrict__ p = part + curves[c].off / 2 + (size_t)l * segs;
    double acc = 0.0;
    for (int i = lane; i < segs; i += 32) acc += p[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) out[(size_t)c * nlags + l] = acc / (double)((1ull << log2n) - lags[l]);
}

// SF(tau)^2 of FP64 curves, one (curve, lag) per block (bound by the FP64
// rate).  Each thread adds runs of 64 strided squares; the block sums in a
// fixed order.
template <typename T>
__global__ void __launch_bounds__(256) k_structure_function(const CurveDev* __restrict__ curves, int nlags,
                                                            const uint32_t* __restrict__ lags,
                                                            const T* __restrict__ x, double* __restrict__ out)
{
    const int c = blockIdx.x / nlags;
    const int l = blockIdx.x % nlags;
    const CurveDev& cv = curves[c];
    const uint64_t tau = lags[l];
    const uint64_t npairs = (1ull << cv.log2n) - tau;
    const T* __restrict__ xc = x + cv.off;
    double acc = 0.0;
    T run = 0;
    int cnt = 0;
    for (uint64_t i = threadIdx.x; i < npairs; i += blockDim.x) {
        const T d = xc[i] - xc[i + tau];
        run += d * d;
        if (++cnt == 64) {
            acc += (double)run;
            run = 0;
            cnt = 0;
        }
    }
    acc += (double)run;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    __shared__ double wpart[8];
    if ((threadIdx.x & 31) == 0) wpart[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += wpart[w];
        out[(size_t)c * nlags + l] = s / (double)npairs;
    }
}

// FP32 structure function of one class.  The partial sums of curves of several
// segments go to the FFT buffer (8 nlags N / 2^14 <= 2 N bytes per curve).  A
// block takes all lags where the curves' segments give four blocks per SM, a
// share of them where not.
static void launch_structure(const Plan& p, const ClassInfo& k, int nlags, const float* x, double* out,
                             cudaStream_t st)
{
    const int segs = k.log2n > 14 ? 1 << (k.log2n - 14) : 1;
    const int64_t units = (int64_t)k.ncurves * segs;
    int groups = (int)std::min<int64_t>(nlags, std::max<int64_t>(1, (152 * 4 + units - 1) / units));
    const int per = (nlags + groups - 1) / groups;
    groups = (nlags + per - 1) / per;
    const unsigned blocks = (unsigned)(units * groups);
    double* part = (double*)p.d_f;
#define LC_SF(MM)                                                                                                  \
    k_structure_runs<MM><<<blocks, 256, 0, st>>>(k.d_curves, p.d_curves, k.log2n, segs, groups, per, nlags, p.d_lags, \
                                                 x, part, out)
    if (k.log2n >= 14) LC_SF(64);
    else if (k.log2n == 13) LC_SF(32);
    else if (k.log2n == 12) LC_SF(16);
    else if (k.log2n == 11) LC_SF(8);
    else LC_SF(4);
#undef LC_SF
    if (segs > 1)
        k_structure_sum<<<(unsigned)(((size_t)k.ncurves * nlags + 3) / 4), 128, 0, st>>>(
            k.d_curves, p.d_curves, k.ncurves, k.log2n, segs, nlags, p.d_lags, part, out);
}

// kPgPairs pairs per block where that gives two blocks per SM, one per thread
// where not: with their transform, one 2^16 FP32 curve 19 us (4096 pairs per
// block: 29), 64 of 2^14 24 (35), one 2^16 FP64 curve 32 (56).
template <typename T>
static void launch_periodogram(const Plan& p, const ClassInfo& k, const void* Z, int rms, double* out, cudaStream_t st)
{
    const uint64_t half = 1ull << (k.log2n - 2);
    uint32_t pairs = kPgPairs;
    while (pairs > 256 && k.ncurves * half < 152ull * 2 * pairs) pairs /= 2;
    const unsigned blocks = (unsigned)(k.ncurves * std::max<uint64_t>(half / pairs, 1));
    k_periodogram<T><<<blocks, 256, 0, st>>>(k.d_curves, p.d_curves, pairs, k.log2n - 1, k.d_tw, Z, rms, out);
}

template <typename T>
static void run_periodogram(Plan& p, const void* x, int rms, double* out, cudaStream_t st)
{
    for (auto& k : p.classes) {
        // x is only read: the passes ping-pong between d_f and d_keysB
        void* Z = launch_fft<T>(p, k, false, const_cast<void*>(x), p.d_f, nullptr, false, st, nullptr, p.d_keysB);
        launch_periodogram<T>(p, k, Z, rms, out, st);
    }
}

}  // namespace lc

using namespace lc;

extern "C" {

lc_status lc_periodogram(lc_plan plan, const void* x, int rms, double* out_p, void* stream)
{
    if (!plan || !x || !out_p) { set_error("null plan, x or out_p"); return LC_ERR_INVALID; }
    DeviceGuard g(plan->device);
    StreamJoin j(*plan, stream);
    if (plan->prec == LC_FP32) run_periodogram<float>(*plan, x, rms, out_p, plan->stream);
    else run_periodogram<double>(*plan, x, rms, out_p, plan->stream);
    LC_CK(cudaGetLastError());
    return LC_OK;
}

lc_status lc_structure_function(lc_plan plan, const void* x, const uint32_t* lags, size_t nlags, double* out_sf2,
                                void* stream)
{
    if (!plan || !x || !lags || !out_sf2) { set_error("null plan, x, lags or out_sf2"); return LC_ERR_INVALID; }
    if (nlags < 1 || nlags > kMaxLags) { set_error("nlags must be in [1, 4096]"); return LC_ERR_INVALID; }
    uint32_t nmin = 0xffffffffu;
    for (auto& k : plan->classes) nmin = std::min(nmin, 1u << k.log2n);
    for (size_t l = 0; l < nlags; ++l) {
        if (lags[l] < 1 || lags[l] >= nmin) {
            set_error("lag " + std::to_string(l) + " outside [1, N) of the shortest curve");
            return LC_ERR_INVALID;
        }
    }
    const uint64_t blocks = (uint64_t)plan->ncurves * nlags;
    if (blocks > 0x7fffffffull) { set_error("ncurves * nlags too large"); return LC_ERR_INVALID; }
    DeviceGuard g(plan->device);
    StreamJoin j(*plan, stream);
    // pageable source: the copy is staged before the call returns
    LC_CK(cudaMemcpyAsync(plan->d_lags, lags, nlags * sizeof(uint32_t), cudaMemcpyHostToDevice, plan->stream));
    if (plan->prec == LC_FP32)
        for (auto& k : plan->classes) launch_structure(*plan, k, (int)nlags, (const float*)x, out_sf2, plan->stream);
    else
        k_structure_function<double><<<(unsigned)blocks, 256, 0, plan->stream>>>(
            plan->d_curves, (int)nlags, plan->d_lags, (const double*)x, out_sf2);
    LC_CK(cudaGetLastError());
    return LC_OK;
}

}  // extern "C"
