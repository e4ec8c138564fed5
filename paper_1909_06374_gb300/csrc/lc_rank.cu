// lc_rank.cu -- the rank-order replacement (x[position] = s[rank]) and the sort
// of the draws for curves that one CTA ranks whole (lc_rank.cuh): one launch
// and one read of the values in place of the LSD passes' three launches and
// 24 to 40 B per value each.  FP64 curves of 2^10 .. 2^14 samples (the values,
// the positions of shared bins' members, counters and starts take 208 KB at 2^14);
// FP32 ones of 2^10 .. 2^12, whose iterations the fused kernels run, for their
// draws and on the multi-kernel path (2^13 on: the sample sort).
// Bound by latency on the one SM of a curve (512 FP64 curves of 2^14: issue 34%,
// ALU 38%, stalls on global loads first, one CTA of 32 warps per SM).  One FP64
// curve of 2^14 samples, transforms included: 119 us per iteration with eight
// LSD passes (24 launches), 94 with FP64 conversions and comparisons here, 72
// with integer ones.
#include "lc_internal.h"
#include "lc_rank.cuh"

namespace lc {

namespace {

struct RankArgs {
    const int* cls_curves;
    const CurveDev* curves;
    const uint32_t* eff_iters;
    const int* d_iter;  // null: every curve active
    const void* src;
    const void* s_in;   // sorted draws (replacement)
    void* out;          // new state, or the sorted values
    float* bounds;      // kRankBounds floats per curve of the class, from the iteration before; may be null
};

template <typename T, int LOG2L>
struct RankCta {
    static constexpr int TH = LOG2L >= 13 ? 1024 : 512;
    static constexpr int BPV = LOG2L == 14 ? 2 : 4;
    using R = RankShape<T, LOG2L, TH, BPV>;
    static constexpr size_t CNT = sizeof(T) << LOG2L;
    static constexpr size_t WST = CNT + R::CNT;
    static constexpr size_t SLOT = WST + R::WST;
    static constexpr size_t SEG = SLOT + R::SLOT;
    static constexpr size_t SPL = SEG + R::SEG;
    static constexpr size_t BYTES = SPL + R::SPL;
    // resident CTAs per SM that the ranking's registers allow; the crowded
    // curves' sort, which takes more, gives way
    static constexpr int MINB = LOG2L <= 11 ? 3 : LOG2L == 12 ? 2 : 1;
    static_assert(BYTES <= 227 * 1024 && R::NSEG + 1 <= kRankBounds, "one CTA's shared memory");
};

// VALUES: out = the sorted values; else out[position] = s_in[rank].  out may be
// src: every value is in shared memory before the first barrier.
template <typename T, int LOG2L, bool VALUES>
__global__ void __launch_bounds__(RankCta<T, LOG2L>::TH, RankCta<T, LOG2L>::MINB) k_rank_cta(const RankArgs a)
{
    using C = RankCta<T, LOG2L>;
    using K = typename key_of<T>::type;
    constexpr int TH = C::TH, L = 1 << LOG2L, PER = L / TH;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t wsum[TH / 32];
    const int tid = threadIdx.x;
    const int c = a.cls_curves[blockIdx.x];
    if (a.d_iter && (uint32_t)(*a.d_iter) >= a.eff_iters[c]) return;
    const uint64_t off = a.curves[c].off;
    const K* src = (const K*)a.src + off;
    T* out = (T*)a.out + off;
    RankMem<T> m;
    m.mem = nullptr;
    m.cnt = (uint32_t*)(smem + C::CNT);
    m.wst = (uint16_t*)(smem + C::WST);
    m.slot = (uint16_t*)(smem + C::SLOT);
    m.seg = (float2*)(smem + C::SEG);
    m.spl = (float*)(smem + C::SPL);
    m.wsum = wsum;
    float* bounds = a.bounds ? a.bounds + (size_t)blockIdx.x * kRankBounds : nullptr;
    K* key = (K*)smem;  // the values' bits at their positions
#pragma unroll
    for (int j = 0; j < PER; ++j) key[tid + j * TH] = src[tid + j * TH];
    const bool warm = bounds && a.d_iter && *a.d_iter > 0;
    if (warm && tid <= C::R::NSEG) m.spl[tid] = bounds[tid];
    __syncthreads();
    uint32_t rk[PER];
    auto any = [&](int i) { return value_bits(key[i]); };
    auto val = [&](int j) { return any(tid + j * TH); };
    if (cta_rank<T, LOG2L, TH, C::BPV, true>(m, warm, val, any, rk)) {
        if (VALUES) {
#pragma unroll
            for (int j = 0; j < PER; ++j) out[rk[j]] = key_value(rank_key(val(j)));  // within one curve: L2 joins them
        } else {
            const T* __restrict__ s = (const T*)a.s_in + off;
#pragma unroll
            for (int j = 0; j < PER; ++j) out[tid + j * TH] = s[rk[j]];
        }
        if (bounds && tid <= C::R::NSEG) bounds[tid] = m.spl[tid];
    } else {  // crowded bins (many equal values): sorted whole
        __syncthreads();
        K v[PER];
#pragma unroll
        for (int j = 0; j < PER; ++j) v[j] = rank_key(val(j));
        __syncthreads();
        const SortPairs<K> sp{key, m.slot};
#pragma unroll
        for (int j = 0; j < PER; ++j) sp.store(tid + j * TH, {v[j], (uint32_t)(tid + j * TH)});
        __syncthreads();
        if constexpr (VALUES) {
            const SortValues<K> sv{key};
            cta_bitonic<TH>(sv, L);
#pragma unroll
            for (int j = 0; j < PER; ++j) out[tid + j * TH] = key_value(sv.load(tid + j * TH));
        } else {
            cta_bitonic<TH>(sp, L);
            const T* __restrict__ s = (const T*)a.s_in + off;
#pragma unroll
            for (int j = 0; j < PER; ++j) out[sp.load(tid + j * TH).p] = s[tid + j * TH];
        }
        if (bounds && tid <= C::R::NSEG) bounds[tid] = 0.0f;  // the next iteration finds them useless
    }
}

template <typename T, int LOG2L>
cudaError_t rank_attr()
{
    const int smem = (int)RankCta<T, LOG2L>::BYTES;
    cudaError_t e =
        cudaFuncSetAttribute(k_rank_cta<T, LOG2L, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_rank_cta<T, LOG2L, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e;
}

template <typename T, int LOG2L>
void go(const RankArgs& a, int ncurves, bool values, cudaStream_t st)
{
    using C = RankCta<T, LOG2L>;
    if (values) k_rank_cta<T, LOG2L, true><<<ncurves, C::TH, C::BYTES, st>>>(a);
    else k_rank_cta<T, LOG2L, false><<<ncurves, C::TH, C::BYTES, st>>>(a);
}

}  // namespace

bool rank_cta_supported(lc_precision prec, uint32_t log2n)
{
    return log2n >= 10 && log2n <= (prec == LC_FP32 ? 12u : 14u);
}

cudaError_t rank_kernel_attributes()
{
    cudaError_t e = cudaSuccess;
    if (e == cudaSuccess) e = rank_attr<float, 10>();
    if (e == cudaSuccess) e = rank_attr<float, 11>();
    if (e == cudaSuccess) e = rank_attr<float, 12>();
    if (e == cudaSuccess) e = rank_attr<double, 10>();
    if (e == cudaSuccess) e = rank_attr<double, 11>();
    if (e == cudaSuccess) e = rank_attr<double, 12>();
    if (e == cudaSuccess) e = rank_attr<double, 13>();
    if (e == cudaSuccess) e = rank_attr<double, 14>();
    return e;
}

template <typename T>
void launch_rank_cta(const Plan& p, const ClassInfo& k, const void* src, bool values, void* x_out, bool gated,
                     cudaStream_t st)
{
    RankArgs a{};
    a.cls_curves = k.d_curves;
    a.curves = p.d_curves;
    a.eff_iters = p.d_eff_iters;
    a.d_iter = gated ? p.d_iter : nullptr;
    a.src = src;
    a.s_in = p.d_s;
    a.out = values ? p.d_s : (x_out ? x_out : p.d_x);
    a.bounds = gated ? k.d_bounds : nullptr;
    switch (k.log2n) {
    case 10: go<T, 10>(a, k.ncurves, values, st); break;
    case 11: go<T, 11>(a, k.ncurves, values, st); break;
    case 12: go<T, 12>(a, k.ncurves, values, st); break;
    default:
        if constexpr (sizeof(T) == 8) {
            if (k.log2n == 13) go<T, 13>(a, k.ncurves, values, st);
            else go<T, 14>(a, k.ncurves, values, st);
        }
    }
}
template void launch_rank_cta<float>(const Plan&, const ClassInfo&, const void*, bool, void*, bool, cudaStream_t);
template void launch_rank_cta<double>(const Plan&, const ClassInfo&, const void*, bool, void*, bool, cudaStream_t);

}  // namespace lc
