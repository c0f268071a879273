// Column transfer of the generator picture as one 2x2 gate per qubit.
//
// On every interior corner column exactly one of the two end plaquettes is a
// check, so the boundary state of the untruncated sweep (Eq. 7 summed column
// by column) has d bits: one per row position. Qubit (r, c) acts on position
// r alone: in an even column it replaces the plaquette above-left of it by the
// one below-right (rows rising), in an odd column the one below-left by the
// one above-right (rows falling), and
//     new[0] = a old[0] + b old[1],  new[1] = b old[0] + a old[1],
// where (a, b) = (w[flip = 0][ctrl], w[1][ctrl]) are the probabilities of the
// Paulis that the two plaquettes' XOR (flip) and the neighbouring positions'
// XOR (ctrl = bit r-1 ^ bit r+1) give on top of the representative. Position r
// carries X-type plaquettes for even r (flip = x part, ctrl = z part), Z-type
// for odd r. Corner columns 0 and d hold Z-type plaquettes only: even
// positions are 0 there. Every term is non-negative, so each entry keeps FP32
// relative accuracy.
//
// Layout: the middle position M = (d-1)/2 is the half of a float2, so packed
// f32x2 arithmetic applies to every other position; the positions on one side
// of M index the registers, those on the other side the lanes. Bit t of either
// index is the position at distance t + 1 from M. A column runs inward (the
// register side towards M), through M, exchanges the two sides (a transpose
// through shared memory, the only exchange a column needs) and runs outward.
// The next column starts on the side where this one ends, so seen from the
// registers every column is the same program.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mld {
namespace gate {

__device__ __forceinline__ uint64_t as_u64(float2 v) { return *reinterpret_cast<uint64_t*>(&v); }
__device__ __forceinline__ float2 as_f2(uint64_t v) { return *reinterpret_cast<float2*>(&v); }

// Packed FP32 pairs: each half rounds like the scalar operation; one issue
// slot instead of two (the FMA pipe's rate is the same).
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(as_u64(a)), "l"(as_u64(b)), "l"(as_u64(c)));
    return as_f2(d);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(as_u64(a)), "l"(as_u64(b)));
    return as_f2(d);
}
__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }

// Weights of a qubit under its representative: x = w[0][0], y = w[0][1],
// z = w[1][0], w = w[1][1] ([flip][ctrl]).
__device__ __forceinline__ float4 permuted(float4 v, uint32_t e) {      // e = ctrl bit | flip bit << 1
    const bool c = e & 1, f = e & 2;
    const float a = c ? v.y : v.x, b = c ? v.x : v.y, g = c ? v.w : v.z, h = c ? v.z : v.w;
    return f ? make_float4(g, h, a, b) : make_float4(a, b, g, h);
}
// A noise row (p_I, p_X, p_Y, p_Z) as [flip][ctrl] of a position's parity.
__device__ __forceinline__ float4 flip_ctrl(float4 p, bool x_flips) {
    return x_flips ? make_float4(p.x, p.w, p.y, p.z) : make_float4(p.x, p.y, p.w, p.z);
}

// Gate on index bit T of P; the control's other bits are T+1 (if below NB)
// and T-1, or the half of the pair for T = 0.
template <int NB, int T>
__device__ __forceinline__ void gate_bit(float2 (&P)[1 << NB], float4 w) {
    float2 A[2], B[2];
    if (T == 0) {
        A[0] = make_float2(w.x, w.y);
        A[1] = make_float2(w.y, w.x);
        B[0] = make_float2(w.z, w.w);
        B[1] = make_float2(w.w, w.z);
    } else {
        A[0] = dup(w.x);
        A[1] = dup(w.y);
        B[0] = dup(w.z);
        B[1] = dup(w.w);
    }
#pragma unroll
    for (int k = 0; k < (1 << NB); ++k) {
        if (k & (1 << T)) continue;
        const int c = ((T + 1 < NB ? k >> (T + 1) : 0) ^ (T > 0 ? k >> (T > 0 ? T - 1 : 0) : 0)) & 1;
        const float2 x = P[k], y = P[k | (1 << T)];
        P[k] = fma2(A[c], x, mul2(B[c], y));
        P[k | (1 << T)] = fma2(B[c], x, mul2(A[c], y));
    }
}

// Gate on the pair's position; control = index bit 0 (what else it depends on
// is folded into w).
template <int NB>
__device__ __forceinline__ void gate_pair(float2 (&P)[1 << NB], float4 w) {
#pragma unroll
    for (int k = 0; k < (1 << NB); ++k) {
        const float a = (k & 1) ? w.y : w.x, b = (k & 1) ? w.w : w.z;
        const float x = P[k].x, y = P[k].y;
        P[k].x = fmaf(a, x, b * y);
        P[k].y = fmaf(b, x, a * y);
    }
}

template <int NB, int T, class W>
__device__ __forceinline__ void gates_down(float2 (&P)[1 << NB], const W& w) {      // T, T-1, .., 0
    gate_bit<NB, T>(P, w(T));
    if constexpr (T > 0) gates_down<NB, T - 1>(P, w);
}
template <int NB, int T, class W>
__device__ __forceinline__ void gates_up(float2 (&P)[1 << NB], const W& w) {        // T, T+1, .., NB-1
    gate_bit<NB, T>(P, w(T));
    if constexpr (T + 1 < NB) gates_up<NB, T + 1>(P, w);
}

// First column, the positions of the index bits: before it even positions are
// 0 and odd ones free, so the state grows from what the earlier positions gave.
// cur[k]: entries over index bits below T (and the pair); an even position
// leaves a second entry per value o of the next position's old bit.
template <int NB, int T, class W>
struct Grow {
    static __device__ __forceinline__ void even(float2 (&P)[1 << NB], const float2* cur, const W& w) {
        const float4 v = w(T);
        if constexpr (T == NB - 1) {
#pragma unroll
            for (int k = 0; k < (1 << T); ++k) {
                const int c = T > 0 ? (k >> (T > 0 ? T - 1 : 0)) & 1 : 0;
                const float2 A = T == 0 ? make_float2(v.x, v.y) : dup(c ? v.y : v.x);
                const float2 B = T == 0 ? make_float2(v.z, v.w) : dup(c ? v.w : v.z);
                P[k] = mul2(A, cur[k]);
                P[k | (1 << T)] = mul2(B, cur[k]);
            }
        } else {
            float2 ext[4 << T];
#pragma unroll
            for (int k = 0; k < (1 << T); ++k) {
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    const int c = o ^ (T > 0 ? (k >> (T > 0 ? T - 1 : 0)) & 1 : 0);
                    const float2 A = T == 0 ? (o ? make_float2(v.y, v.x) : make_float2(v.x, v.y)) : dup(c ? v.y : v.x);
                    const float2 B = T == 0 ? (o ? make_float2(v.w, v.z) : make_float2(v.z, v.w)) : dup(c ? v.w : v.z);
                    ext[2 * k + o] = mul2(A, cur[k]);
                    ext[2 * (k | (1 << T)) + o] = mul2(B, cur[k]);
                }
            }
            Grow<NB, T + 1, W>::odd(P, ext, w);
        }
    }
    static __device__ __forceinline__ void odd(float2 (&P)[1 << NB], const float2* ext, const W& w) {
        const float4 v = w(T);
        float2 out[2 << T];
#pragma unroll
        for (int k = 0; k < (1 << T); ++k) {
            const int c = T > 0 ? (k >> (T > 0 ? T - 1 : 0)) & 1 : 0;
            const float2 A = T == 0 ? make_float2(v.x, v.y) : dup(c ? v.y : v.x);
            const float2 B = T == 0 ? make_float2(v.z, v.w) : dup(c ? v.w : v.z);
            out[k] = fma2(A, ext[2 * k], mul2(B, ext[2 * k + 1]));
            out[k | (1 << T)] = fma2(B, ext[2 * k], mul2(A, ext[2 * k + 1]));
        }
        if constexpr (T == NB - 1) {
#pragma unroll
            for (int k = 0; k < (1 << NB); ++k) P[k] = out[k];
        } else {
            Grow<NB, T + 1, W>::even(P, out, w);
        }
    }
};

// ln z + e ln 2 for z >= 0. ln of the mantissa m in [sqrt(1/2), sqrt(2)) from
// the series of 2 atanh((m-1)/(m+1)), the quotient to twice FP32 precision, so
// that the error stays below 2e-9 (1.8e-9 over all mantissas, the operations
// run on the host; an FP64 log is some 25 instructions of a
// pipe with 1/64 of the FP32 rate: at d = 5 it would cost more than the sweep).
__device__ __forceinline__ double ln_scaled(float z, int e) {
    if (!(z > 0.f)) return -INFINITY;
    int ex = 0;
    if (z < 1.17549435e-38f) {
        z *= 16777216.f;
        ex = -24;
    }
    const uint32_t bits = __float_as_uint(z);
    ex += (int)(bits >> 23) - 127;
    float m = __uint_as_float((bits & 0x7fffffu) | 0x3f800000u);
    if (m > 1.41421354f) {
        m *= 0.5f;
        ex += 1;
    }
    const float num = m - 1.f;                       // exact
    const float den = m + 1.f;
    const float den_lo = m - (den - 1.f);            // m + 1 = den + den_lo
    const float r = __frcp_rn(den);
    const float s = num * r;
    const float rem = fmaf(-s, den_lo, fmaf(-s, den, num));
    const float q = s * s;
    float t = fmaf(q, 2.f / 13.f, 2.f / 11.f);       // 2 s (1/3 s^2 + 1/5 s^4 + ..), |s| < 0.172
    t = fmaf(t, q, 2.f / 9.f);
    t = fmaf(t, q, 2.f / 7.f);
    t = fmaf(t, q, 2.f / 5.f);
    t = fmaf(t, q, 2.f / 3.f);
    const float tail = fmaf(t * q, s, 2.f * rem * r);
    return fma((double)(e + ex), 0.69314718055994530942, (double)(2.f * s) + (double)tail);
}

// Power-of-two rescaling by the largest entry m >= 0 (as its bit pattern) to
// about 2^100: no gate lets an entry grow (a + b <= 1), so the whole exponent
// range below is left for entries that later columns favour (at p = 1e-5 and
// d = 11 these lie up to e^-110 below the largest). Returns the factor and
// takes its logarithm off the exponent.
constexpr int kTop = 100;
template <int TOP = kTop>
__device__ __forceinline__ float rescale(uint32_t mbits, int& e2) {
    int up = mbits ? TOP + 127 - (int)(mbits >> 23) : 0;
    up = up > 127 ? 127 : up;
    e2 -= up;
    return __uint_as_float((uint32_t)(127 + up) << 23);
}
// The scale of the first column.
__device__ __forceinline__ float top_scale() { return __uint_as_float((uint32_t)(127 + kTop) << 23); }

template <int N>
__device__ __forceinline__ float max_of(const float2 (&P)[N]) {
    float m = fmaxf(P[0].x, P[0].y);
#pragma unroll
    for (int k = 1; k < N; ++k) m = fmaxf(fmaxf(m, P[k].x), P[k].y);
    return m;
}

}  // namespace gate
}  // namespace mld
