// lc_rank.cuh -- exact stable ranks of one curve's values by one CTA.
//
// The range of the values is cut into NSEG segments of about equally many
// values (bounds: the ranks of the iteration before, else a sorted sample), a
// segment into equal bins by linear interpolation -- both monotone in the
// value -- with BPV bins per value on average.  Bins are counted with shared-
// memory atomics (8-bit counters, four to a word; the returned count is the
// value's slot in its bin) and scanned; a value alone in its bin has the bin's
// start as rank, the others (22% at four bins per value, 39% at two) compare
// themselves with the members of their bin by (value, position).  A thread
// keeps the values at its own positions, so a rank carries no payload and the
// replacement x[position] = s[rank] stores no scattered words.
//
// Any bounds give exact ranks; they only have to keep the bins sparse.  Where a
// bin gets more than kCrowd values the bounds are taken from a sorted sample,
// and if that leaves a crowded bin too (many equal values) the caller sorts
// the curve whole.
//
// Bound by issue and shared-memory latency: ~100 thread instructions per value
// against ~400 for four 8-bit LSD passes.  4096 curves of 2^12 x 100
// iterations (7 ms of it transforms): 48.1 ms with LSD passes, 26.5 ms with
// two 16-bit bins per value and 256 threads, 22.4 ms as it stands (search tree
// 19.2 -> 18.6 ms of iterations, three CTAs per SM at 42 registers 22.4).
#pragma once
#include "lc_dft.cuh"

namespace lc {

constexpr uint32_t kCrowd = 96;  // values of a bin at most (8-bit counters)

template <typename T, int LOG2L, int TH, int BPV>
struct RankShape {
    static constexpr int L = 1 << LOG2L;
    static constexpr int PER = L / TH;                   // values per thread
    static constexpr int NSEG = L / 16 < 256 ? L / 16 : 256;
    static constexpr int LPS = L / NSEG;                 // values per segment
    static constexpr int BPS = BPV * LPS;                // bins per segment
    static constexpr int SAMPLE = L < 1024 ? L : 1024;   // values of the sorted sample
    static constexpr int WORDS = L * BPV / 4;            // counter words
    static constexpr int WPT = WORDS / TH;               // of a thread in the scan
    static_assert(WPT >= 1 && BPV * L <= 65536 && NSEG <= TH && LOG2L <= 14, "16-bit bins, starts and positions");
    // bytes of the parts
    static constexpr size_t CNT = (size_t)4 * WORDS;     // counters; the sample while it is sorted
    static constexpr size_t WST = (size_t)2 * WORDS;     // start of each counter word's first bin
    static constexpr size_t SLOT = (size_t)2 * L;        // positions of shared bins' members
    static constexpr size_t SEG = (size_t)8 * NSEG;      // lower bound, bins per unit value
    static constexpr size_t SPL = (size_t)8 * NSEG + 16; // NSEG + 1 bounds, then their search tree
    static_assert(CNT >= 4 * SAMPLE, "room for the sample");
};

// A float that does not decrease with the value, and the value's order key:
// for doubles by integer operations (an SM converts, adds and compares 2
// doubles per clock: one 2^14 curve's iteration 94 us with them).
__device__ __forceinline__ float rank_float(float v) { return v; }
__device__ __forceinline__ float rank_float(double v)
{
    // rounded towards zero, exponents beyond float's clamped
    const int hi = __double2hiint(v), lo = __double2loint(v);
    const int e = (hi & 0x7fffffff) - (896 << 20);  // exponent and mantissa head
    const int m = e < 0 ? 0 : e >= (255 << 20) ? 0x7f7fffff : (e << 3) | (int)((uint32_t)lo >> 29);
    return __int_as_float((hi & 0x80000000) | m);
}
__device__ __forceinline__ uint32_t rank_key(float v) { return order_key(v); }
__device__ __forceinline__ unsigned long long rank_key(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? (b == 0x8000000000000000ull ? b : ~b) : b | 0x8000000000000000ull;  // -0 as +0
}

// Shared-memory parts of the ranking; mem (null: members' values are fetched by
// position) holds the keys of the members of shared bins (the caller's values
// may lie there: they are in `val` by then).
template <typename T>
struct RankMem {
    typename key_of<T>::type* mem;
    uint32_t* cnt;
    uint16_t* wst;
    uint16_t* slot;
    float2* seg;
    float* spl;
    uint32_t* wsum;  // one word per warp
};

// Place of element i of a shared array that cta_bitonic sorts: threads that take
// eight neighbours each meet no bank conflict.
template <typename V>
__device__ __forceinline__ int sorted_at(int i)
{
    return i ^ ((i >> (sizeof(V) == 8 ? 4 : 5)) & 7);
}

// What cta_bitonic sorts: values, or keys with positions (by key, then position).
template <typename V>
struct SortValues {
    V* v;
    using E = V;
    __device__ __forceinline__ E load(int i) const { return v[sorted_at<V>(i)]; }
    __device__ __forceinline__ void store(int i, E e) const { v[sorted_at<V>(i)] = e; }
    static __device__ __forceinline__ bool less(E a, E b) { return a < b; }
};
template <typename K>
struct SortPairs {
    K* key;
    uint16_t* pos;
    struct E {
        K k;
        uint32_t p;
    };
    __device__ __forceinline__ E load(int i) const { return {key[sorted_at<K>(i)], pos[sorted_at<uint16_t>(i)]}; }
    __device__ __forceinline__ void store(int i, E e) const
    {
        key[sorted_at<K>(i)] = e.k;
        pos[sorted_at<uint16_t>(i)] = (uint16_t)e.p;
    }
    static __device__ __forceinline__ bool less(E a, E b) { return a.k < b.k || (a.k == b.k && a.p < b.p); }
};

// B strides of the bitonic network, the smallest `low`, in registers; `k` the
// length of the runs that they merge.
template <int TH, int B, typename A>
__device__ __forceinline__ void bitonic_strides(const A& a, int n, int k, int low)
{
    constexpr int G = 1 << B;
    for (int i = threadIdx.x; i < n / G; i += TH) {
        const int e = ((i & ~(low - 1)) << B) | (i & (low - 1));
        const bool up = (e & k) == 0;
        typename A::E v[G];
#pragma unroll
        for (int q = 0; q < G; ++q) v[q] = a.load(e + q * low);
#pragma unroll
        for (int h = G / 2; h > 0; h >>= 1) {
#pragma unroll
            for (int q = 0; q < G; ++q) {
                if (q & h) continue;
                if (A::less(v[q + h], v[q]) == up) {
                    const typename A::E t = v[q];
                    v[q] = v[q + h];
                    v[q + h] = t;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < G; ++q) a.store(e + q * low, v[q]);
    }
    __syncthreads();
}

// Ascending bitonic sort of n = 2^m elements, three strides per pass over
// shared memory.  Bound by issue (about 12 instructions per exchange of pairs).
// Ranks of 512 FP64 curves of 2^14 equal values: 891 us with a stride per pass,
// 648 as it stands (eight LSD passes 498, distinct values 235); 1024 FP32
// curves of 2^12 226, 181 (107, 58).
template <int TH, typename A>
__device__ __forceinline__ void cta_bitonic(const A& a, int n)
{
    for (int m = 1; (1 << m) <= n; ++m) {
        int l = m;  // strides left
        if (m % 3 == 1) bitonic_strides<TH, 1>(a, n, 1 << m, 1 << (l -= 1));
        else if (m % 3 == 2) bitonic_strides<TH, 2>(a, n, 1 << m, 1 << (l -= 2));
        while (l > 0) bitonic_strides<TH, 3>(a, n, 1 << m, 1 << (l -= 3));
    }
}

// rk[j] = rank of the value val(j), which stands at position threadIdx.x + j TH
// (any(i): the value at position i, BY_POS: in shared memory throughout).  warm:
// spl holds bounds.  False: crowded, no ranks.  Leaves the next bounds in spl;
// ends with a block barrier.
template <typename T, int LOG2L, int TH, int BPV, bool BY_POS, typename F, typename G>
__device__ __forceinline__ bool cta_rank(const RankMem<T>& m, bool warm, F&& val, G&& any,
                                         uint32_t (&rk)[(1 << LOG2L) / TH])
{
    using R = RankShape<T, LOG2L, TH, BPV>;
    constexpr int L = R::L, PER = R::PER, NSEG = R::NSEG, LPS = R::LPS, BPS = R::BPS, WPT = R::WPT;
    constexpr int G4 = PER < 4 ? PER : 4;  // values whose searches overlap
    constexpr int LN = ilog2c(NSEG);
    float* const tree = m.spl + NSEG + 4;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (bool sampled = !warm;; sampled = true) {
        if (sampled) {
            constexpr int SN = R::SAMPLE, ST = L / SN;
            const SortValues<float> smp{(float*)m.cnt};
            for (int i = tid; i < SN; i += TH) smp.store(i, rank_float(any(i * ST + ST / 2)));
            __syncthreads();
            cta_bitonic<TH>(smp, SN);
            if (tid < NSEG) m.spl[tid] = smp.load(tid * (SN / NSEG));
            if (tid == 0) m.spl[NSEG] = smp.load(SN - 1);
            // a value of which the sample has twice a crowded bin's share: no
            // need to count (its atomics would queue at one word)
            constexpr int SHARE = 2 * (int)kCrowd * SN / L;
            bool tied = false;
            for (int i = tid; i + SHARE < SN; i += TH) tied |= smp.load(i) == smp.load(i + SHARE);
            if (__syncthreads_or(tied)) return false;
        }
        for (int i = tid; i < R::WORDS; i += TH) m.cnt[i] = 0u;
        if (tid < NSEG) {
            const float hi = m.spl[tid + 1];
            float lo = m.spl[tid];
            if (tid == 0) lo -= hi - lo;  // room for values beyond the bounds
            const float w = tid == NSEG - 1 ? 2.0f * (hi - lo) : hi - lo;
            m.seg[tid] = make_float2(lo, w > 0.0f ? __fdividef((float)BPS, w) : 0.0f);
            // the bounds as a search tree, level after level: a level of up to
            // 32 nodes meets no bank conflict (halving the sorted bounds
            // directly meets up to eight; 30 wavefronts a search against 11)
            if (tid > 0) {
                const int l = 31 - __clz(tid);
                tree[tid] = m.spl[(2 * (tid - (1 << l)) + 1) << (LN - 1 - l)];
            }
        }
        __syncthreads();
        bool crowded = false;
#pragma unroll
        for (int j0 = 0; j0 < PER; j0 += G4) {
            float f[G4];
            int k[G4];
#pragma unroll
            for (int j = 0; j < G4; ++j) {
                f[j] = rank_float(val(j0 + j));
                k[j] = 1;
            }
#pragma unroll
            for (int l = 0; l < LN; ++l)
#pragma unroll
                for (int j = 0; j < G4; ++j) k[j] = 2 * k[j] + (f[j] >= tree[k[j]] ? 1 : 0);
#pragma unroll
            for (int j = 0; j < G4; ++j) {
                k[j] -= NSEG;
                const float2 g = m.seg[k[j]];
                const int q = max(0, min(__float2int_rz((f[j] - g.x) * g.y), BPS - 1));  // NaN -> 0
                const uint32_t u = (uint32_t)(k[j] * BPS + q), sh = (u & 3u) << 3;
                const uint32_t old = (atomicAdd(&m.cnt[u >> 2], 1u << sh) >> sh) & 255u;
                crowded |= old >= kCrowd;  // seen before the counter could overflow
                rk[j0 + j] = u | (old << 16);
            }
        }
        if (!__syncthreads_or(crowded)) break;
        if (sampled) return false;
    }
    {
        // starts: exclusive scan over the counter words, WPT consecutive ones per thread
        // (wide shared loads: a thread's words lie side by side)
        uint32_t c[WPT], sum = 0;
        if constexpr (WPT % 4 == 0) {
#pragma unroll
            for (int i = 0; i < WPT; i += 4) *(uint4*)&c[i] = *(const uint4*)(m.cnt + WPT * tid + i);
        } else {
#pragma unroll
            for (int i = 0; i < WPT; ++i) c[i] = m.cnt[WPT * tid + i];
        }
#pragma unroll
        for (int i = 0; i < WPT; ++i) {
            const uint32_t n = __dp4a(c[i], 0x01010101u, 0u);
            c[i] = sum;
            sum += n;
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) m.wsum[warp] = incl;
        __syncthreads();
        uint32_t run = incl - sum;
#pragma unroll
        for (int w = 0; w < TH / 32; ++w) run += w < warp ? m.wsum[w] : 0u;
        if constexpr (WPT % 4 == 0) {
#pragma unroll
            for (int i = 0; i < WPT; i += 4)
                *(uint2*)(m.wst + WPT * tid + i) = make_uint2((run + c[i]) | ((run + c[i + 1]) << 16),
                                                              (run + c[i + 2]) | ((run + c[i + 3]) << 16));
        } else {
#pragma unroll
            for (int i = 0; i < WPT; ++i) m.wst[WPT * tid + i] = (uint16_t)(run + c[i]);
        }
    }
    __syncthreads();
    // rk = start | members << 16 | slot << 24; shared bins' members leave value and position
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const uint32_t u = rk[j] & 0xffffu, old = rk[j] >> 16, sh = (u & 3u) << 3;
        const uint32_t w = m.cnt[u >> 2];
        const uint32_t s0 = __dp4a(w & ((1u << sh) - 1u), 0x01010101u, (uint32_t)m.wst[u >> 2]);
        const uint32_t c = (w >> sh) & 255u;
        if (c > 1u) {
            if (!BY_POS) m.mem[s0 + old] = rank_key(val(j));
            m.slot[s0 + old] = (uint16_t)(tid + j * TH);
        }
        rk[j] = s0 | (c << 16) | (old << 24);
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const uint32_t s0 = rk[j] & 0xffffu, c = (rk[j] >> 16) & 255u;
        uint32_t r = s0;
        if (c > 1u) {
            // the member after the own slot: all there is to compare with in a pair
            const typename key_of<T>::type v = rank_key(val(j));
            uint32_t o = rk[j] >> 24;
            for (uint32_t i = 1; i < c; ++i) {
                o = o + 1u == c ? 0u : o + 1u;
                typename key_of<T>::type y;
                if (BY_POS) y = rank_key(any((int)m.slot[s0 + o]));
                else y = m.mem[s0 + o];
                r += y < v ? 1u : 0u;
                if (y == v) r += (int)m.slot[s0 + o] < tid + j * TH ? 1u : 0u;
            }
        }
        rk[j] = r;
        if ((r & (LPS - 1)) == 0u || r == (uint32_t)L - 1u) {
            const float f = rank_float(val(j));
            if ((r & (LPS - 1)) == 0u) m.spl[r / LPS] = f;
            if (r == (uint32_t)L - 1u) m.spl[NSEG] = f;
        }
    }
    __syncthreads();
    return true;
}

}  // namespace lc
