// Register-side pieces of the transfer under independent X/Z noise
// (mld_xz.cu): gates on one bit of a state held in registers, the exchange of
// register and lane bits, rescaling.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mld_gate.cuh"

namespace mld {
namespace xz {

// Twice FP32: hi + lo, |lo| <= ulp(hi)/2. The transfer has products and sums of
// non-negative numbers only, so nothing cancels.
struct Twin {
    float hi, lo;
};
// (The _rn intrinsics keep the compiler from contracting a product into the
// sum whose rounding error the next lines take.)
__device__ __forceinline__ Twin renormal(float s, float e) {
    const float hi = __fadd_rn(s, e);
    return Twin{hi, __fsub_rn(e, __fsub_rn(hi, s))};
}
// a + b = s + returned error (Knuth's two-sum)
__device__ __forceinline__ float sum_error(float a, float b, float s) {
    const float t = __fsub_rn(s, a);
    return __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}
__device__ __forceinline__ Twin times(Twin a, Twin b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.lo, b.lo, e);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    return renormal(p, e);
}
__device__ __forceinline__ double times(double a, double b) { return a * b; }
// a x + b y
__device__ __forceinline__ Twin dot(Twin a, Twin x, Twin b, Twin y) {
    const float p = __fmul_rn(a.hi, x.hi), q = __fmul_rn(b.hi, y.hi);
    float e = __fmaf_rn(a.hi, x.hi, -p), f = __fmaf_rn(b.hi, y.hi, -q);
    e = __fmaf_rn(a.hi, x.lo, e);
    f = __fmaf_rn(b.hi, y.lo, f);
    e = __fmaf_rn(a.lo, x.hi, e);
    f = __fmaf_rn(b.lo, y.hi, f);
    const float s = __fadd_rn(p, q);
    return renormal(s, __fadd_rn(sum_error(p, q, s), __fadd_rn(e, f)));
}
__device__ __forceinline__ double dot(double a, double x, double b, double y) { return fma(a, x, b * y); }
__device__ __forceinline__ Twin plus(Twin a, Twin b) {
    const float s = __fadd_rn(a.hi, b.hi);
    return renormal(s, __fadd_rn(sum_error(a.hi, b.hi, s), __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ double plus(double a, double b) { return a + b; }
template <typename T>
__device__ __forceinline__ T make(double x);
template <>
__device__ __forceinline__ double make<double>(double x) { return x; }
template <>
__device__ __forceinline__ Twin make<Twin>(double x) {
    const float hi = (float)x;
    return Twin{hi, (float)(x - (double)hi)};
}
__device__ __forceinline__ Twin scaled(Twin a, float s) { return Twin{a.hi * s, a.lo * s}; }   // s a power of two
__device__ __forceinline__ double scaled(double a, double s) { return a * s; }
template <typename T>
struct ScaleOf { using type = double; };
template <>
struct ScaleOf<Twin> { using type = float; };

// c_ab = f[a] g[b] under the representative.
template <typename T>
struct Weights {
    T c00, c10, c01, c11;
};

// new[n] = sum_o f[o ^ n] g[prev ^ o] old[o] on register bit TB of a state of
// RB bits; prev is register bit PREV (-1: none).
template <int RB, int TB, int PREV>
__device__ __forceinline__ void gate_on(double (&v)[1 << RB], Weights<double> w) {
#pragma unroll
    for (int i = 0; i < (1 << RB); ++i) {
        if (i >> TB & 1) continue;
        const bool p = PREV >= 0 && (i >> (PREV >= 0 ? PREV : 0) & 1);
        const double x = v[i], y = v[i | 1 << TB];
        v[i] = dot(p ? w.c01 : w.c00, x, p ? w.c10 : w.c11, y);
        v[i | 1 << TB] = dot(p ? w.c11 : w.c10, x, p ? w.c00 : w.c01, y);
    }
}

// Register bits T, T+1, .., END-1 (prev is the bit below; none below 0).
template <int RB, int TB, int END, class W>
__device__ __forceinline__ void gates_rising(double (&v)[1 << RB], const W& w) {
    if constexpr (TB < END) {
        gate_on<RB, TB, TB - 1>(v, w(TB));
        gates_rising<RB, TB + 1, END>(v, w);
    }
}
// Register bits TB, TB-1, .., 0 (prev is the bit above).
template <int RB, int TB, class W>
__device__ __forceinline__ void gates_falling(double (&v)[1 << RB], const W& w) {
    if constexpr (TB >= 0) {
        gate_on<RB, TB, TB + 1>(v, w(TB));
        gates_falling<RB, TB - 1>(v, w);
    }
}

// The same on the top register bit, prev in bit 0, followed by a rotation of
// the index (the top bit becomes bit 0): one body serves every row pair in
// turn. a, b: weights of old[0], old[1] for new[n], by [prev][n].
template <int RB, typename T>
__device__ __forceinline__ void gate_and_rotate(T (&v)[1 << RB], const T (&a)[2][2], const T (&b)[2][2]) {
    constexpr int R = 1 << RB;
    T out[R];
#pragma unroll
    for (int i = 0; i < R / 2; ++i) {
        out[2 * i] = dot(a[i & 1][0], v[i], b[i & 1][0], v[i + R / 2]);
        out[2 * i + 1] = dot(a[i & 1][1], v[i], b[i & 1][1], v[i + R / 2]);
    }
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = out[i];
}
template <int RB>
__host__ __device__ constexpr int reversed(int i) {
    int r = 0;
    for (int t = 0; t < RB; ++t) r |= (i >> t & 1) << (RB - 1 - t);
    return r;
}

// Before the exchange register bit t is row pair RB-1-t: the pairs below LB
// (the top register bits) become lane bits, the lane bits (pair H-1-u) become
// register bits MID+u (pair RB on top, so that it comes next), the MID pairs
// between follow below. A vector holds the values of consecutive MID pairs.
template <int LB, int RB>
__host__ __device__ constexpr int store_index(int k, int m) {
    // pairs 0..LB-1 from k (bit j = pair j), pairs LB..RB-1 from m (bit j-LB)
    int i = 0;
    for (int j = 0; j < RB; ++j) i |= ((j < LB ? k >> j : m >> (j - LB)) & 1) << (RB - 1 - j);
    return i;
}
template <int LB, int RB>
__host__ __device__ constexpr int load_index(int k, int m) {
    // bit u of the writer's lane k is pair H-1-u; bit t of m is pair LB+t
    int i = k << (RB - LB);
    for (int t = 0; t < RB - LB; ++t) i |= (m >> t & 1) << (RB - LB - 1 - t);
    return i;
}

template <int BYTES>
struct Vec;
template <>
struct Vec<8> { using type = float2; };
template <>
struct Vec<16> { using type = float4; };

template <class S, typename T>
__device__ __forceinline__ void exchange_store(unsigned char* X, const T (&v)[1 << S::RB], int lane) {
    using V = typename Vec<S::VB>::type;
    constexpr int PER = S::VB / (int)sizeof(T);
    V* x = reinterpret_cast<V*>(X) + lane;
#pragma unroll
    for (int k = 0; k < S::LANES; ++k)
#pragma unroll
        for (int s = 0; s < S::SLOTS; ++s) {
            V t;
            T* e = reinterpret_cast<T*>(&t);
#pragma unroll
            for (int m = 0; m < PER; ++m) e[m] = v[store_index<S::LB, S::RB>(k, s * PER + m)];
            x[(s * S::LANES + k) * S::STRIDE] = t;
        }
}
template <class S, typename T>
__device__ __forceinline__ void exchange_load(const unsigned char* X, T (&v)[1 << S::RB], int lane) {
    using V = typename Vec<S::VB>::type;
    constexpr int PER = S::VB / (int)sizeof(T);
    const V* x = reinterpret_cast<const V*>(X) + lane * S::STRIDE;
#pragma unroll
    for (int k = 0; k < S::LANES; ++k)
#pragma unroll
        for (int s = 0; s < S::SLOTS; ++s) {
            const V t = x[s * S::LANES * S::STRIDE + k];
            const T* e = reinterpret_cast<const T*>(&t);
#pragma unroll
            for (int m = 0; m < PER; ++m) v[load_index<S::LB, S::RB>(k, s * PER + m)] = e[m];
        }
}

template <int LANES>
__device__ __forceinline__ void unit_sync(int unit) {
    if constexpr (LANES > 32)
        asm volatile("bar.sync %0, %1;" ::"r"(1 + unit), "n"(LANES) : "memory");
    else
        __syncwarp();
}

// Entries are kept near the top of the exponent range. Between two rescalings
// they grow by at most 2^H (1 + odds <= 2 a gate). An operation loses at most
// a few of the smallest subnormals, 2^14 of them in an entry by the next
// rescaling; entries of at least 2^-low there keep their accuracy.
template <typename T>
struct Range;
template <>
struct Range<double> {
    static constexpr int top = 900;
    static constexpr uint32_t low = (uint32_t)(1023 - 980) << 20;
    static __device__ __forceinline__ double start() { return __hiloint2double((1023 + top) << 20, 0); }
    // bits of the largest entry: its high word, which orders alike
    static __device__ __forceinline__ uint32_t bits(double v) { return (uint32_t)__double2hiint(v); }
    static __device__ __forceinline__ double rescale(uint32_t m, int& e2) {
        int up = m ? top + 1023 - (int)(m >> 20) : 0;
        up = up > 1000 ? 1000 : up;
        e2 -= up;
        return __hiloint2double((1023 + up) << 20, 0);
    }
};
template <>
struct Range<Twin> {
    static constexpr int top = gate::kTop;
    static constexpr uint32_t low = (uint32_t)(127 - 80) << 23;
    static __device__ __forceinline__ Twin start() { return Twin{gate::top_scale(), 0.f}; }
    static __device__ __forceinline__ uint32_t bits(Twin v) { return __float_as_uint(v.hi); }
    static __device__ __forceinline__ float rescale(uint32_t m, int& e2) { return gate::rescale<>(m, e2); }
};
template <typename T, int N>
__device__ __forceinline__ uint32_t max_bits(const T (&v)[N]) {
    uint32_t m = Range<T>::bits(v[0]);
#pragma unroll
    for (int i = 0; i < N; i += 2) m = __vimax3_u32(m, Range<T>::bits(v[i]), Range<T>::bits(v[i + 1]));
    return m;
}
template <typename T, int N>
__device__ __forceinline__ uint32_t min_bits(const T (&v)[N]) {
    uint32_t m = Range<T>::bits(v[0]);
#pragma unroll
    for (int i = 0; i < N; i += 2) m = __vimin3_u32(m, Range<T>::bits(v[i]), Range<T>::bits(v[i + 1]));
    return m;
}

// z = m 2^e, m in [sqrt(1/2), sqrt(2)), by its bits (z > 0); e is added.
__device__ __forceinline__ double mantissa(double z, int& e) {
    if (__double2hiint(z) < 1 << 20) {                    // subnormal
        z *= 18014398509481984.0;                         // 2^54
        e -= 54;
    }
    const int hi = __double2hiint(z), frac = hi & 0xfffff;
    const int up = frac >= 0x6a09e;
    e += (hi >> 20) - 1023 + up;
    return __hiloint2double(frac | (1023 - up) << 20, __double2loint(z));
}
// ln(z m) + e ln 2, the exponents joined first (z is kept near 2^top, and
// ln z and e ln 2 would cancel to a few hundred ulps of their difference).
__device__ __forceinline__ double log_of(double z, double m, int e) {
    if (!(z > 0.0) || !(z < INFINITY)) return z > 0.0 ? z : -INFINITY;
    m = mantissa(mantissa(z, e) * m, e);
    return log(m) + (double)e * 0.69314718055994530942;
}

// A qubit's two weights as odds: t[0] of a flip, t[1] of none, the larger one 1;
// returns the larger probability.
__device__ __forceinline__ double odds_of(double* t, float p) {
    const double x = p, y = 1.0 - x;
    t[0] = x > y ? 1.0 : x / y;
    t[1] = x > y ? y / x : 1.0;
    return x > y ? x : y;
}
__device__ __forceinline__ double odds_of(Twin* t, float p) {
    // 1 - p is a float for p > 1/2, and a pair below
    const bool flips = p > 0.5f;
    const float q = __fsub_rn(1.f, p), small = flips ? q : p, hi = flips ? p : q;
    const float lo = flips ? 0.f : __fsub_rn(__fsub_rn(1.f, q), p);
    const float r = __fdiv_rn(small, hi);
    const float rest = __fmaf_rn(-r, lo, __fmaf_rn(-r, hi, small));
    const Twin odds = renormal(r, __fdiv_rn(rest, hi)), one = Twin{1.f, 0.f};
    t[0] = flips ? one : odds;
    t[1] = flips ? odds : one;
    return (double)hi + (double)lo;
}

__device__ __forceinline__ double value_of(double z) { return z; }
__device__ __forceinline__ double value_of(Twin z) { return (double)z.hi + (double)z.lo; }
__device__ __forceinline__ double shuffled(double z, int o) { return __shfl_xor_sync(0xffffffffu, z, o); }
__device__ __forceinline__ Twin shuffled(Twin z, int o) {
    return Twin{__shfl_xor_sync(0xffffffffu, z.hi, o), __shfl_xor_sync(0xffffffffu, z.lo, o)};
}

}  // namespace xz
}  // namespace mld
