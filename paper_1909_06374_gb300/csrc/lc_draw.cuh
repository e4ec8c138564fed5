// lc_draw.cuh -- single-precision ERDF draws without FP64 transcendentals.
//
// A float draw is the FP64 draw of erdf_draw / erdf_draw_tab rounded to 24
// bits.  The FP64 logarithm, quotients and exponential behind it are ~120
// double operations, and this GPU runs 2 of them per clock and SM against 128
// float ones.  Here the argument of the logarithm (or the table's u) is formed
// with the FP64 sequence's own operations (5 to 9 of them), and log2(lambda)
// and lambda are then carried in pairs of floats (head + tail, error-free
// sums and products after Dekker 1971 and Knuth, TAOCP 4.2.2; table-driven
// reductions after Tang, ACM TOMS 1989/1990).  With log2(lambda) = E = B + L K,
// relative errors of lambda (times ln 2 where they are E's):
//   2^-39  the float polynomial of 2^g: its terms reach 2^-16, rounded to
//          2^-40 a few times, and the first one left out is 2^-44;
//   (|E| + kc) 2^-44  B, K, the pair product L K and L itself, each to 2^-46 of
//          its share (log_pair: 2^-45 + 2^-47 |L|, times K).
// exp2_pair allows four times that, 2^-37 + (|E| + kc) 2^-42, beside which the
// FP64 sequence's own rounding (2^-50) does not count.  Where every value
// within that bound rounds to the same float, that float is the draw; otherwise
// (about 1 draw in 2^11) the caller runs the FP64 sequence.  So the draws keep
// their bits.  FP64 pipe 86% busy (512 curves of 2^16).
#pragma once
#include "lc_common.cuh"

namespace lc {

// Compile-time tables: natural log by the atanh series and 2^x by Taylor, in
// double (error below 2^-50, the pairs keep 2^-48).
constexpr double ct_log(double x)  // x in (0.5, 2)
{
    const double s = (x - 1.0) / (x + 1.0), z = s * s;
    double p = 0.0;
    for (int k = 41; k >= 1; k -= 2) p = p * z + 1.0 / k;
    return 2.0 * s * p;
}
constexpr double ct_exp2(double x)  // |x| <= 1/2
{
    const double y = x * 0.69314718055994530942;
    double p = 1.0;
    for (int k = 20; k >= 1; --k) p = 1.0 + p * y / k;
    return p;
}

constexpr int kDrawLog = 128;  // intervals of [1, 2)
constexpr int kDrawExp = 64;   // steps of 2^x per unit
struct DrawTables {
    float c[kDrawLog], lh[kDrawLog], ll[kDrawLog];      // c ~ 1/m, -log c as head + tail
    float eh[kDrawExp + 1], el[kDrawExp + 1];           // 2^{(j - 32)/64} as head + tail
};
constexpr DrawTables make_draw_tables()
{
    DrawTables t{};
    for (int i = 0; i < kDrawLog; ++i) {
        t.c[i] = (float)(1.0 / (1.0 + (i + 0.5) / kDrawLog));
        const double l = -ct_log((double)t.c[i]);
        t.lh[i] = (float)l;
        t.ll[i] = (float)(l - (double)t.lh[i]);
    }
    for (int j = 0; j <= kDrawExp; ++j) {
        const double e = ct_exp2((double)(j - kDrawExp / 2) / kDrawExp);
        t.eh[j] = (float)e;
        t.el[j] = (float)(e - (double)t.eh[j]);
    }
    return t;
}

#define LC_LN2F 0x1.62e430p-1f            // ln 2 = LC_LN2F + LC_LN2F_LO (to 2^-50)
#define LC_LN2F_LO (-0x1.05c610p-29f)

// s + e = a + b exactly (Knuth).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Natural logarithm of a positive normal double as head + tail, absolute
// error below 2^-45 + 2^-47 |log x|.
__device__ __forceinline__ void log_pair(const DrawTables& t, double x, float& h, float& l)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const float e = (float)((int)(b >> 52) - 1023);
    const float mh = __uint_as_float(0x3f800000u | ((uint32_t)(b >> 29) & 0x7fffffu));
    const float ml = __fmul_rn((float)((uint32_t)b & 0x1fffffffu), 0x1p-52f);
    const int i = (int)(b >> 45) & (kDrawLog - 1);
    const float c = t.c[i];
    // r = m c - 1 = rh + rl, |r| <= 2^-8
    const float p = __fmul_rn(mh, c);
    const float pe = __fmaf_rn(ml, c, __fmaf_rn(mh, c, -p));
    const float d = __fsub_rn(p, 1.0f);  // exact
    const float rh = __fadd_rn(d, pe);
    const float rl = __fsub_rn(pe, __fsub_rn(rh, d));
    // log(1 + r) = r - r^2/2 + r^3/3 - r^4/4 + r^5/5 - ...
    const float q = __fmul_rn(rh, rh);
    const float qe = __fmaf_rn(rh, rh, -q);
    float tail = __fmaf_rn(rh, 0.2f, -0.25f);
    tail = __fmaf_rn(rh, tail, 0x1.555556p-2f);
    tail = __fmul_rn(__fmul_rn(q, rh), tail);
    const float low = __fadd_rn(tail, __fmaf_rn(-rh, rl, __fmaf_rn(-0.5f, qe, rl)));
    const float hi = __fmaf_rn(-0.5f, q, rh);
    const float he = __fmaf_rn(-0.5f, q, __fsub_rn(rh, hi));
    // + e ln 2 - log c
    const float eh = __fmul_rn(e, LC_LN2F);
    const float el = __fmaf_rn(e, LC_LN2F_LO, __fmaf_rn(e, LC_LN2F, -eh));
    float s1, t1, s2, t2;
    two_sum(eh, t.lh[i], s1, t1);
    two_sum(s1, hi, s2, t2);
    const float lo = __fadd_rn(__fadd_rn(t1, t2), __fadd_rn(__fadd_rn(el, t.ll[i]), __fadd_rn(he, low)));
    h = __fadd_rn(s2, lo);
    l = __fsub_rn(lo, __fsub_rn(h, s2));
}

// 2^{B + L K} rounded to float when that is certain: true and the value, or
// false (the caller takes the FP64 sequence).  B, L, K as head + tail; kc =
// |K| + |B| scales the error bound, lo and hi are the clamp limits.
__device__ __forceinline__ bool exp2_pair(const DrawTables& t, float Bh, float Bl, float Lh, float Ll, float Kh,
                                          float Kl, float kc, float lo, float hi, float& out)
{
    const float ph = __fmul_rn(Lh, Kh);
    const float pe = __fadd_rn(__fmaf_rn(Lh, Kh, -ph), __fmaf_rn(Lh, Kl, __fmul_rn(Ll, Kh)));
    float s, e;
    two_sum(Bh, ph, s, e);
    e = __fadd_rn(__fadd_rn(e, Bl), pe);
    const float Eh = __fadd_rn(s, e);
    const float El = __fsub_rn(e, __fsub_rn(Eh, s));
    if (!(fabsf(Eh) < 120.0f)) return false;  // also NaN
    const float n = rintf(Eh);
    const float f = __fsub_rn(Eh, n);         // exact, |f| <= 1/2
    const float jf = rintf(__fmul_rn(f, (float)kDrawExp));
    const float g = __fmaf_rn(jf, -1.0f / kDrawExp, f);  // exact, |g| <= 2^-7
    const int j = (int)jf + kDrawExp / 2;
    // y = 2^{g + El} - 1 = z + z^2/2 + ..., z = (g + El) ln 2
    const float zh = __fmul_rn(g, LC_LN2F);
    const float zl = __fmaf_rn(El, LC_LN2F, __fmaf_rn(g, LC_LN2F_LO, __fmaf_rn(g, LC_LN2F, -zh)));
    float q = __fmaf_rn(zh, 0x1.555556p-5f, 0x1.555556p-3f);
    q = __fmul_rn(__fmul_rn(zh, zh), __fmaf_rn(zh, q, 0.5f));
    const float w = __fadd_rn(q, __fmaf_rn(zl, __fadd_rn(zh, q), zl));
    const float yh = __fadd_rn(zh, w);
    const float yl = __fsub_rn(w, __fsub_rn(yh, zh));
    const float Th = t.eh[j], Tl = t.el[j];
    const float mh = __fmul_rn(Th, yh);
    const float me = __fmaf_rn(Th, yl, __fmaf_rn(Th, yh, -mh));
    const float r = __fadd_rn(Th, mh);
    const float rl = __fadd_rn(__fsub_rn(mh, __fsub_rn(r, Th)), __fadd_rn(me, __fmaf_rn(Tl, yh, Tl)));
    const float m = __fmaf_rn(__fadd_rn(fabsf(Eh), kc), 0x1p-42f, 0x1p-37f);
    const float f1 = __fadd_rn(r, __fadd_rn(rl, m)), f2 = __fadd_rn(r, __fsub_rn(rl, m));
    out = __uint_as_float(__float_as_uint(f1) + ((uint32_t)(int)n << 23));
    return f1 == f2 && out > lo && out < hi;
}

__device__ __forceinline__ void split_pair(double x, float& h, float& l)
{
    h = (float)x;
    l = (float)(x - (double)h);
}

__device__ inline DrawConst draw_constants(const ErdfConst& k)
{
    const double log2_10 = 0x1.a934f0979a371p+1;
    DrawConst d;
    split_pair(log2_10, d.Uh, d.Ul);
    split_pair(log2_10 * k.ub, d.Bh, d.Bl);
    split_pair(k.a1nz ? log2_10 / k.c1 : 0.0, d.K1h, d.K1l);
    split_pair(k.a2nz ? log2_10 / k.c2 : 0.0, d.K2h, d.K2l);
    // |K| and |B| at their largest
    d.kc = fabsf(d.Bh) + fmaxf(fmaxf(fabsf(d.K1h), fabsf(d.K2h)), d.Uh);
    d.lo = (float)k.lo * (1.0f + 0x1p-20f);
    d.hi = (float)k.hi * (1.0f - 0x1p-20f);
    return d;
}

// (w0, w1) -> U as unit_open, with one FP64 operation: 1 + u 2^-52 less
// 1 - 2^-53 (exact).
__device__ __forceinline__ double unit_open_fast(uint32_t w0, uint32_t w1)
{
    const unsigned long long x = ((unsigned long long)w1 << 32) | w0;
    const double d = __longlong_as_double((long long)((x >> 12) | 0x3ff0000000000000ull));
    return __dsub_rn(d, 0x1.fffffffffffffp-1);
}

// Float draw of the sharp broken power law for uniform U; false where the
// FP64 sequence has to decide.
__device__ __forceinline__ bool erdf_draw_fast(const DrawTables& t, const ErdfConst& k, const DrawConst& d, double U,
                                               float& out)
{
    const double v = __dmul_rn(U, k.Msum);
    const bool below = v < k.M1;
    double arg;
    float add = 0.0f;
    bool power = true;
    if (below) {
        power = k.a1nz != 0;
        arg = power ? __dadd_rn(k.e1, __dmul_rn(k.c1, v)) : __dadd_rn(k.umin, v);
    } else {
        const double r = __dsub_rn(v, k.M1);
        power = k.a2nz != 0;
        if (power) {
            const double y = __dmul_rn(k.c2, r);
            arg = __dadd_rn(1.0, y);
            add = (float)__dsub_rn(y, __dsub_rn(arg, 1.0));  // 1 + y = arg + add exactly
        } else {
            arg = __dadd_rn(k.ub, r);
        }
    }
    float Lh, Ll, Kh, Kl, Bh, Bl;
    if (power) {
        // positive, normal, and 1 + y distinct from 1
        if (!(arg > 1e-30) || arg > 1e30 || (!below && arg == 1.0)) return false;
        log_pair(t, arg, Lh, Ll);
        Ll = __fadd_rn(Ll, __fdividef(add, (float)arg));
        Kh = below ? d.K1h : d.K2h;
        Kl = below ? d.K1l : d.K2l;
        Bh = d.Bh;
        Bl = d.Bl;
    } else {
        split_pair(arg, Lh, Ll);
        Kh = d.Uh;
        Kl = d.Ul;
        Bh = Bl = 0.0f;
    }
    return exp2_pair(t, Bh, Bl, Lh, Ll, Kh, Kl, d.kc, d.lo, d.hi, out);
}

// Float draw of a tabulated shape (erdf_draw_tab): the same FP64 v, interval
// and differences; the position inside the interval as a quotient of pairs.
// The bisection compares the bits of non-negative doubles, whose order is
// theirs.
__device__ __forceinline__ bool erdf_draw_tab_fast(const DrawTables& t, const double* F, double umin, double h,
                                                   const DrawConst& d, double U, float& out)
{
    const double v = __dmul_rn(U, F[kErdfTable]);
    const long long vb = __double_as_longlong(v);
    int a = 0;
#pragma unroll
    for (int w = kErdfTable / 2; w > 0; w >>= 1)
        if (__double_as_longlong(F[a + w]) <= vb) a += w;
    const double num = __dsub_rn(v, F[a]), den = __dsub_rn(F[a + 1], F[a]);
    if (!(den > 1e-30) || den > 1e30) return false;
    float nh, nl, dh, dl;
    split_pair(num, nh, nl);
    split_pair(den, dh, dl);
    const float rc = __frcp_rn(dh);
    const float q = __fmul_rn(nh, rc);
    const float r = __fmul_rn(__fadd_rn(__fmaf_rn(-q, dh, nh), __fmaf_rn(-q, dl, nl)), rc);
    // u = (umin + a h) + (q + r) h
    float uh, ul, hh, hl, Lh, Ll;
    split_pair(__fma_rn((double)a, h, umin), uh, ul);
    split_pair(h, hh, hl);
    const float ph = __fmul_rn(q, hh);
    const float pe = __fadd_rn(__fmaf_rn(q, hh, -ph), __fmaf_rn(q, hl, __fmul_rn(r, hh)));
    two_sum(uh, ph, Lh, Ll);
    Ll = __fadd_rn(Ll, __fadd_rn(pe, ul));
    return exp2_pair(t, 0.0f, 0.0f, Lh, Ll, d.Uh, d.Ul, d.kc, d.lo, d.hi, out);
}

}  // namespace lc
