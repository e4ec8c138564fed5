// lc_dft.cuh -- in-register DFTs of R <= 16 points for the FFT passes.
#pragma once
#include "lc_common.cuh"

namespace lc {

__host__ __device__ constexpr int ilog2c(int r) { return r <= 1 ? 0 : 1 + ilog2c(r >> 1); }
__host__ __device__ constexpr int bitrev_c(int v, int bits)
{
    return bits == 0 ? 0 : (((v & 1) << (bits - 1)) | bitrev_c(v >> 1, bits - 1));
}

// cos(2 pi t / 16)
__device__ __forceinline__ double cos16(int t)
{
    switch (t & 15) {
    case 0: return 1.0;
    case 1: return 0.92387953251128675613;
    case 2: return 0.70710678118654752440;
    case 3: return 0.38268343236508977173;
    case 4: return 0.0;
    case 5: return -0.38268343236508977173;
    case 6: return -0.70710678118654752440;
    case 7: return -0.92387953251128675613;
    case 8: return -1.0;
    case 9: return -0.92387953251128675613;
    case 10: return -0.70710678118654752440;
    case 11: return -0.38268343236508977173;
    case 12: return 0.0;
    case 13: return 0.38268343236508977173;
    case 14: return 0.70710678118654752440;
    default: return 0.92387953251128675613;
    }
}

// b * e^{-+ 2 pi i t/16} (+ for the inverse transform); t is a compile-time
// constant at every call site, so the branches fold away.
template <typename T, bool INV>
__device__ __forceinline__ cplx<T> rot16(cplx<T> b, int t)
{
    cplx<T> r;
    if (t == 0) return b;
    if (t == 4) {
        if (INV) { r.x = -b.y; r.y = b.x; } else { r.x = b.y; r.y = -b.x; }
        return r;
    }
    if (t == 8) { r.x = -b.x; r.y = -b.y; return r; }
    const T c = (T)cos16(t);
    const T s = INV ? (T)cos16(t + 12) : -(T)cos16(t + 12);  // sin(2 pi t/16) = cos(2 pi (t - 4)/16)
    r.x = b.x * c - b.y * s;
    r.y = b.x * s + b.y * c;
    return r;
}

// Bit-reversal permutation with indices fixed at compile time (keeps the
// array in registers).
template <int I, int R, typename V>
struct BitrevSwaps {
    static __device__ __forceinline__ void run(V (&u)[R])
    {
        constexpr int J = bitrev_c(I, ilog2c(R));
        if constexpr (J > I) { V t = u[I]; u[I] = u[J]; u[J] = t; }
        BitrevSwaps<I + 1, R, V>::run(u);
    }
};
template <int R, typename V>
struct BitrevSwaps<R, R, V> {
    static __device__ __forceinline__ void run(V (&)[R]) {}
};

// out[q] = sum_r u[r] e^{-+ 2 pi i r q / R}: radix-2 decimation in time on the
// bit-reversed input.
template <typename T, int R, bool INV>
__device__ __forceinline__ void dft_regs(cplx<T> (&u)[R])
{
    constexpr int LR = ilog2c(R);
    BitrevSwaps<0, R, cplx<T>>::run(u);
#pragma unroll
    for (int s = 1; s <= LR; ++s) {
        const int m = 1 << s, h = m >> 1;
#pragma unroll
        for (int g = 0; g < R; g += m) {
#pragma unroll
            for (int j = 0; j < h; ++j) {
                const cplx<T> a = u[g + j];
                const cplx<T> b = rot16<T, INV>(u[g + j + h], j * (16 / m));
                u[g + j] = cadd(a, b);
                u[g + j + h] = csub(a, b);
            }
        }
    }
}

// -------------------------------------------------------- fixed rounding
// The iteration ranks what the transforms return, so a transform has to round
// the same way in every kernel that computes it (two tile sizes, one class or
// several per launch), however the compiler would contract its products.
// These forms write every rounding down; the products that FMA leaves unrounded
// are the ones of the kernels' plain expressions as nvcc contracts them.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// a b with one product of each component rounded first: a.y b.y of the real
// part, and of the imaginary part a.y b.x (cmul_a) or a.x b.y (cmul_b).
template <typename V> __device__ __forceinline__ V cmul_a(V a, V b)
{
    V r;
    r.x = fma_rn(a.x, b.x, -mul_rn(a.y, b.y));
    r.y = fma_rn(a.x, b.y, mul_rn(a.y, b.x));
    return r;
}
template <typename V> __device__ __forceinline__ V cmul_b(V a, V b)
{
    V r;
    r.x = fma_rn(a.x, b.x, -mul_rn(a.y, b.y));
    r.y = fma_rn(a.y, b.x, mul_rn(a.x, b.y));
    return r;
}

// a +- b as one packed operation (two float roundings, one issue slot): the
// three transform kernels of an iteration of 4096 x 2^16 samples 1.754 -> 1.735
// ms, of one 2^17 curve 15.9 -> 15.2 us.
__device__ __forceinline__ unsigned long long pack2(float2 a)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long a)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ float2 add_fixed(float2 a, float2 b)
{
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}
__device__ __forceinline__ float2 sub_fixed(float2 a, float2 b)
{
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}
__device__ __forceinline__ double2 add_fixed(double2 a, double2 b)
{
    return make_double2(__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y));
}
__device__ __forceinline__ double2 sub_fixed(double2 a, double2 b)
{
    return make_double2(__dsub_rn(a.x, b.x), __dsub_rn(a.y, b.y));
}

// rot16 with every rounding written down.
template <typename T, bool INV>
__device__ __forceinline__ cplx<T> rot16_fixed(cplx<T> b, int t)
{
    cplx<T> r;
    if (t == 0) return b;
    if (t == 4) {
        r.x = INV ? -b.y : b.y;
        r.y = INV ? b.x : -b.x;
        return r;
    }
    const T c = (T)cos16(t);
    const T s = INV ? (T)cos16(t + 12) : -(T)cos16(t + 12);
    const bool x1 = t == 6 && !INV, y1 = t != 2;
    r.x = x1 ? fma_rn(-b.y, s, mul_rn(b.x, c)) : fma_rn(b.x, c, -mul_rn(b.y, s));
    r.y = y1 ? fma_rn(b.y, c, mul_rn(b.x, s)) : fma_rn(b.x, s, mul_rn(b.y, c));
    return r;
}

// dft_regs with every rounding written down.
template <typename T, int R, bool INV>
__device__ __forceinline__ void dft_fixed(cplx<T> (&u)[R])
{
    constexpr int LR = ilog2c(R);
    BitrevSwaps<0, R, cplx<T>>::run(u);
#pragma unroll
    for (int s = 1; s <= LR; ++s) {
        const int m = 1 << s, h = m >> 1;
#pragma unroll
        for (int g = 0; g < R; g += m) {
#pragma unroll
            for (int j = 0; j < h; ++j) {
                const cplx<T> a = u[g + j];
                const cplx<T> b = rot16_fixed<T, INV>(u[g + j + h], j * (16 / m));
                u[g + j] = add_fixed(a, b);
                u[g + j + h] = sub_fixed(a, b);
            }
        }
    }
}

}  // namespace lc
