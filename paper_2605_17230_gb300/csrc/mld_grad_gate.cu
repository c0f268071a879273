// Adjoint of the column transfer (mld_gate.cuh): ln Z_l of every class and
// sum_l dlogP_l d ln Z_l / d p for every qubit, d = 3..11 at untruncated chi.
//
// A unit is (syndrome, l_Z), 2^M lanes (M = (d-1)/2) holding the state and the
// adjoint state in registers, 2^(d-M) entries each. Forward: the states at
// every column's start go to the unit's global slice (L2). Z is linear in
// every gate's weights, and the two classes l_X share all columns but the
// last, so their adjoint states, weighted dlogP_l / Z_l, are added at the
// start of the last column and swept back as one: per column, the forward
// gates are run again from the stored state, and each gate, last to first,
// gives its weight sums (old state times adjoint state, by flip and control)
// and carries the adjoint back (the gate is symmetric). The old state of a
// gate is recomputed from a checkpoint at most three gates back: two per side
// of the column's exchange, in shared memory.
//
// Range: the adjoint state is rescaled by a power of two after every column
// and the forward sweep's rescalings are left out of it (both go to the FP64
// factor of the weight sums). No gate lets an entry grow, so neither state
// leaves its top however rare the syndrome is, and the weight sums stay finite.
// Entries keep FP32 accuracy down to 2^-180 of the largest. Below, a class may
// lose its paths; the sums of a gate, weighted, then miss the upstream
// gradient that they add up to, and the unit adds nothing from there on
// (MLD_ERR_NUMERIC).
//
// Accuracy: a gate's weighted sums add up to the upstream gradients of the two
// classes, up to the roundings of the states between the gate and Z. The first
// gate of each side of a column measures the ratio (in FP32 pairs) and the
// sums of that side are corrected by it. Of classes whose gradients oppose each
// other by more than a twentieth the common ratio would multiply what sets
// their own apart, so they are swept back one after the other. Against 64 bits,
// batch gradient of an unlabelled loss, 512 shots: d = 3 3.4e-8 (without 9.2e-8,
// a sweep per class divided by each column's own overlap 4.4e-8), d = 5 2.8e-8
// (8.9e-8, 4.9e-8), d = 7 4.0e-8 (8.8e-8, 5.0e-8), d = 9 4.3e-8 (1.2e-7, 8.1e-8);
// single shots with gradients 1, -1 of two classes, of their terms: d = 7 8.4e-8
// (1.8e-7, 1.1e-7), d = 9 1.1e-7 (2.4e-7, 1.3e-7).
//
// Bound: at d <= 9 issue and shared memory (50% of the issue slots, 62% of the
// shared-memory cycles at d = 7: state loads, exchanges, the sums over lanes);
// at d = 11 the fetching of its own straight-line program (93 KB) by five
// resident warps an SM. Measured on GB300, against one block per (syndrome,
// class) with its states in shared memory: d = 7, 65,536 syndromes 0.63 ms
// (6.1; 0.56 without the correction; 1.0 where all units hold opposed classes);
// d = 9, 16,384 syndromes 0.87 ms (8.6; 0.72 without it and the rescaling of the
// adjoint state; 1.47 opposed); d = 11, 2,049 syndromes 1.0 ms (7.4; 1.9
// opposed). A column as a list of operations run by an
// interpreter (one copy of each gate's code) was slower: 0.92, 1.18, 1.90 ms.
//
// Gradients are summed per unit slot in FP64 in a fixed order, the slots by a
// second kernel: reruns give the same bits.
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "mld_gate.cuh"
#include "mld_grad.h"
#include "mld_internal.h"
#include "mld_xz.cuh"

namespace mld {
namespace {

using namespace gate;
using xz::Twin;

// Tops of the states and of the adjoint states (a class's paths need the range
// below both): a weight sum adds up to 2^d products of the two, below
// 2^(54 + 1 + 54 + 1 + 11).
constexpr int kGradTop = 54, kAdjointTop = 54;
// Classes whose adjoint states at the start of the last column differ by more
// than this are swept back one at a time (they would not fit one range), and
// so are those whose gradients add up to less than this part of their moduli.
constexpr double kApart = 8.673617379884035e-19;        // 2^-60
constexpr float kOpposed = 0.9f;

template <int D>
struct GradLanes {
    static constexpr int N = D * D;
    static constexpr int M = (D - 1) / 2;
    static constexpr int R = 1 << M;                    // float2 per lane
    static constexpr int LANES = 1 << M;
    static constexpr int UPW = 32 / LANES;              // units a warp sweeps at a time
    static constexpr int SPW = UPW > 1 ? UPW / 2 : 1;   // syndromes of a warp
    static constexpr int WORDS = (N - 1 + 63) / 64;
    static constexpr int WARPS = D == 11 ? 2 : 4;       // of a block
    static constexpr int STRIDE = LANES + 1;
    static constexpr int XCH = LANES * STRIDE;          // float2; also holds the state after the exchange
    static constexpr int STATE = R * LANES;             // float2
    static constexpr int HI = (M + 2) / 2;              // checkpoint of the M + 1 gates before the exchange
    static constexpr int HO = (M + 1) / 2;              // and of the M after it
    static constexpr int UNIT = XCH + 2 * STATE;        // float2 of shared memory
    static constexpr size_t kWarpBytes =
        (size_t)UPW * UNIT * 8 + (size_t)UPW * N * 4 * 8 + (size_t)UPW * (D + 2) * 4 + SPW * D * 4;
    static constexpr size_t kTable = (size_t)N * 16 * (D == 11 ? 1 : 4);
    static constexpr size_t kBytes = kTable + WARPS * ((kWarpBytes + 15) & ~(size_t)15);
    static constexpr int64_t kSlice = (int64_t)(D + 1) * STATE;      // float2 of a unit's global slice
};

__host__ __device__ constexpr int grad_row(int d, int c, int j) { return (c & 1) ? d - 1 - j : j; }

// x 2^e by its exponent field (FP64 arithmetic has 1/64 of the FP32 rate);
// subnormal values and results are 0, infinities and NaN stay, and what would
// overflow stays finite.
__device__ __forceinline__ double scaled(double x, int e) {
    const int hi = __double2hiint(x), at = (hi >> 20) & 0x7ff;
    if (at == 0x7ff) return x;
    const int to = at + e;
    if (at == 0 || to <= 0) return 0.0;
    return __hiloint2double((hi & ~(0x7ff << 20)) | (to < 0x7fe ? to : 0x7fe) << 20, __double2loint(x));
}
// The same in FP32, to infinity.
__device__ __forceinline__ float scaled(float x, int e) {
    const int bits = __float_as_int(x), at = (bits >> 23) & 0xff, to = at + e;
    if (at == 0 || to <= 0) return 0.f;
    return to < 0xff ? __int_as_float((bits & ~(0xff << 23)) | to << 23) : copysignf(INFINITY, x);
}

template <int M>
__device__ __forceinline__ void load_state(float2 (&P)[1 << M], const float2* s, int lane) {
#pragma unroll
    for (int k = 0; k < (1 << M); ++k) P[k] = s[(k << M) + lane];
}
template <int M>
__device__ __forceinline__ void store_state(const float2 (&P)[1 << M], float2* s, int lane) {
#pragma unroll
    for (int k = 0; k < (1 << M); ++k) s[(k << M) + lane] = P[k];
}

// Weight sums of one gate and the adjoint before it: s[2 f + c].
template <int M, int T>
__device__ __forceinline__ void back_bit(const float2 (&P)[1 << M], float2 (&G)[1 << M], float4 w, float (&s)[4]) {
    float2 A[2], B[2], F0[2], F1[2];
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
    F0[0] = F0[1] = F1[0] = F1[1] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < (1 << M); ++k) {
        if (k & (1 << T)) continue;
        const int c = ((T + 1 < M ? k >> (T + 1) : 0) ^ (T > 0 ? k >> (T > 0 ? T - 1 : 0) : 0)) & 1;
        const float2 x = P[k], y = P[k | (1 << T)], g0 = G[k], g1 = G[k | (1 << T)];
        F0[c] = fma2(x, g0, fma2(y, g1, F0[c]));
        F1[c] = fma2(y, g0, fma2(x, g1, F1[c]));
        G[k] = fma2(A[c], g0, mul2(B[c], g1));
        G[k | (1 << T)] = fma2(B[c], g0, mul2(A[c], g1));
    }
    if (T == 0) {                                       // the halves' controls differ
        s[0] = F0[0].x + F0[1].y;
        s[1] = F0[0].y + F0[1].x;
        s[2] = F1[0].x + F1[1].y;
        s[3] = F1[0].y + F1[1].x;
    } else {
        s[0] = F0[0].x + F0[0].y;
        s[1] = F0[1].x + F0[1].y;
        s[2] = F1[0].x + F1[0].y;
        s[3] = F1[1].x + F1[1].y;
    }
}
template <int M>
__device__ __forceinline__ void back_pair(const float2 (&P)[1 << M], float2 (&G)[1 << M], float4 w, float (&s)[4]) {
    s[0] = s[1] = s[2] = s[3] = 0.f;
#pragma unroll
    for (int k = 0; k < (1 << M); ++k) {
        const int c = k & 1;
        const float a = c ? w.y : w.x, b = c ? w.w : w.z;
        const float x = P[k].x, y = P[k].y, g0 = G[k].x, g1 = G[k].y;
        s[c] = fmaf(x, g0, fmaf(y, g1, s[c]));
        s[2 + c] = fmaf(y, g0, fmaf(x, g1, s[2 + c]));
        G[k].x = fmaf(a, g0, b * g1);
        G[k].y = fmaf(b, g0, a * g1);
    }
}

// What a warp's lanes know of their unit.
template <int D>
struct Lane {
    using S = GradLanes<D>;
    static constexpr int M = S::M;
    const float4* tab;
    float2* xch;            // exchange buffer, then the state after the exchange
    float2* ck_in;          // checkpoints
    float2* ck_out;
    float2* slice;          // states at the columns' starts [c], and the adjoint sum of the last column
    double* acc;            // [n][4]
    float* scale;           // rescaling within each column
    const uint32_t* words;  // representative bits by column
    int lane, lz;

    __device__ __forceinline__ uint32_t bit(int t) const { return (uint32_t)(lane >> t) & 1u; }
    // Z on row 0 (l_Z); X on the last column (l_X)
    __device__ __forceinline__ uint32_t word(int c, int lx) const {
        uint32_t w = words[c] ^ (lz ? ((c & 1) ? 1u << (2 * (D - 1)) : 1u) : 0u);
        if (lx) {
#pragma unroll
            for (int j = 0; j < D; ++j) w ^= 1u << (2 * j + ((j & 1) ? 0 : 1));
        }
        return w;
    }
    __device__ __forceinline__ float4 weight(int c, int j, uint32_t w, uint32_t toggle) const {
        const uint32_t e = ((w >> (2 * j)) & 3) ^ toggle;
        return D == 11 ? permuted(tab[c * D + j], e) : tab[(c * D + j) * 4 + e];
    }
    // weights of step J: the lane's control folded in at the middle, the
    // column's rescaling at the first step after the exchange
    template <int J>
    __device__ __forceinline__ float4 step_weight(int c, uint32_t w, float sc) const {
        float4 v = weight(c, J, w, J == M ? bit(0) : 0u);
        if (J == M + 1) v = make_float4(v.x * sc, v.y * sc, v.z * sc, v.w * sc);
        return v;
    }
    template <int J>
    __device__ __forceinline__ void step(float2 (&P)[1 << M], int c, uint32_t w, float sc) const {
        const float4 v = step_weight<J>(c, w, sc);
        if constexpr (J < M)
            gate_bit<M, M - 1 - J>(P, v);
        else if constexpr (J == M)
            gate_pair<M>(P, v);
        else
            gate_bit<M, J - M - 1>(P, v);
    }
    template <int FROM, int TO>
    __device__ __forceinline__ void steps(float2 (&P)[1 << M], int c, uint32_t w, float sc) const {
        if constexpr (FROM < TO) {
            step<FROM>(P, c, w, sc);
            steps<FROM + 1, TO>(P, c, w, sc);
        }
    }
    __device__ __forceinline__ void exchange(float2 (&P)[1 << M]) const {
        __syncwarp();
#pragma unroll
        for (int k = 0; k < (1 << M); ++k) xch[lane * S::STRIDE + k] = P[k];
        __syncwarp();
#pragma unroll
        for (int k = 0; k < (1 << M); ++k) P[k] = xch[k * S::STRIDE + lane];
        __syncwarp();
    }
    // bits of the unit's largest entry, from the lanes' (>= 0)
    __device__ __forceinline__ static uint32_t unit_max(float x) {
        uint32_t mx = __float_as_uint(x);
        if constexpr (S::LANES == 32) {
            mx = __reduce_max_sync(0xffffffffu, mx);
        } else {
#pragma unroll
            for (int o = S::LANES / 2; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        return mx;
    }
    // the whole column; scale[slot] keeps its rescaling
    __device__ __forceinline__ void column(float2 (&P)[1 << M], int c, uint32_t w, int slot, int& e2) const {
        steps<0, M + 1>(P, c, w, 1.f);
        const float sc = rescale<kGradTop>(unit_max(max_of(P)), e2);
        if (lane == 0) scale[slot] = sc;
        exchange(P);
        steps<M + 1, D>(P, c, w, sc);
    }
    // What a column's weight sums are multiplied by: the column's rescaling is
    // a factor of those of step M+1 and of all before it (early), not of G.
    struct Factors {
        double late, early;
        Twin unit, want;            // what a gate's weighted sums times (unit 2^e) come to
        float slack, trust;         // by how much they may miss it; and to be corrected
        int e_late, e_early;
        float drift;                // what they miss, of them
        bool lost;
    };
    // Step J backwards: P is the state before it.
    template <int J>
    __device__ __forceinline__ void back(const float2 (&P)[1 << M], float2 (&G)[1 << M], int c, uint32_t w,
                                         Factors& by) const {
        float s[4];
        const float4 v = step_weight<J>(c, w, 1.f);
        if constexpr (J < M)
            back_bit<M, M - 1 - J>(P, G, v, s);
        else if constexpr (J == M)
            back_pair<M>(P, G, v, s);
        else
            back_bit<M, J - M - 1>(P, G, v, s);
        if (J == M && bit(0)) {                          // the lane's share of the control
            float t = s[0];
            s[0] = s[1];
            s[1] = t;
            t = s[2];
            s[2] = s[3];
            s[3] = t;
        }
        // sums over the unit's lanes; lane 2 f + c (bits swapped: 0, 2, 1, 3)
        // ends with s[2 f + c]
        float v0, v1;
        {
            const bool up = lane & 1;
            const float k0 = up ? s[2] : s[0], k1 = up ? s[3] : s[1];
            v0 = k0 + __shfl_xor_sync(0xffffffffu, up ? s[0] : s[2], 1);
            v1 = k1 + __shfl_xor_sync(0xffffffffu, up ? s[1] : s[3], 1);
        }
        const int r = grad_row(D, c, J), q = r * D + c;
        const uint32_t e = (w >> (2 * J)) & 3;
        // (the first gate of each side: its weighted sums have to give what the
        // unit adds; the ratio takes the roundings between here and Z out)
        const auto check = [&](float a, float b, float a2 = 0.f, float b2 = 0.f) {
            const auto product = [](float x, float w) {
                const float p = __fmul_rn(x, w);
                return Twin{p, __fmaf_rn(x, w, -p)};
            };
            Twin t = product(a, b);
            if (M == 1) t = xz::plus(t, product(a2, b2));
#pragma unroll
            for (int o = 1; o < S::LANES && o < 4; o <<= 1) t = xz::plus(t, xz::shuffled(t, o));
            const int e = J > M + 1 ? by.e_late : by.e_early;
            t.hi = scaled(__shfl_sync(0xffffffffu, t.hi, 0, S::LANES), e);
            t.lo = scaled(__shfl_sync(0xffffffffu, t.lo, 0, S::LANES), e);
            t = xz::times(t, by.unit);
            const float miss = (by.want.hi - t.hi) + (by.want.lo - t.lo);
            if (fabsf(miss) > by.slack) {
                by.lost = true;
                by.late = by.early = 0.0;
            }
            by.drift = by.trust > 0.f && fabsf(miss) <= by.trust ? miss / t.hi : 0.f;
        };
        const float4 y = J == M && bit(0) ? make_float4(v.y, v.x, v.w, v.z) : v;      // as the sums: without the lane's share
        if constexpr ((J == D - 1 || J == M) && M == 1) check(v0, (lane & 1) ? y.z : y.x, v1, (lane & 1) ? y.w : y.y);
        const auto add = [&](int f, int cc, float x) {
            const int ff = f ^ (int)(e >> 1), c2 = cc ^ (int)(e & 1);
            const int xx = (r & 1) ? c2 : ff, zz = (r & 1) ? ff : c2;
            acc[4 * q + (xx ? (zz ? 2 : 1) : (zz ? 3 : 0))] += (double)fmaf(x, by.drift, x) * (J > M + 1 ? by.late : by.early);
        };
        if constexpr (M == 1) {
            add(lane & 1, 0, v0);
            add(lane & 1, 1, v1);
        } else {
            const bool up = lane & 2;
            float x = (up ? v1 : v0) + __shfl_xor_sync(0xffffffffu, up ? v0 : v1, 2);
#pragma unroll
            for (int o = 4; o < S::LANES; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if constexpr (J == D - 1 || J == M)
                check(x, lane < 4 ? ((lane & 1) ? ((lane & 2) ? y.w : y.z) : ((lane & 2) ? y.y : y.x)) : 0.f);
            if (lane < 4) add(lane & 1, lane >> 1, x);
        }
    }
    // Steps J-1, .., FROM backwards, the state before step FROM being in base.
    template <int FROM, int J>
    __device__ __forceinline__ void back_from(const float2* base, float2 (&G)[1 << M], int c, uint32_t w, float sc,
                                              Factors& by) const {
        if constexpr (J > FROM) {
            float2 P[1 << M];
            load_state<M>(P, base, lane);
            steps<FROM, J - 1>(P, c, w, sc);
            back<J - 1>(P, G, c, w, by);
            back_from<FROM, J - 1>(base, G, c, w, sc, by);
        }
    }
    // Column c backwards: G after it -> G before it; factor 2^ge G is the
    // derivative of the loss by the state (unit is the same factor, with the
    // upstream gradients want, on a common scale). Returns whether the range
    // was lost.
    __device__ __forceinline__ bool back_column(float2 (&G)[1 << M], int c, uint32_t w, int slot, double factor, int& ge,
                                                Twin unit, Twin want, float slack, float trust) const {
        const float sc = scale[slot];
        Factors by;
        by.unit = unit;
        by.want = want;
        by.slack = slack;
        by.trust = trust;
        by.lost = false;
        by.e_late = ge;
        by.late = scaled(factor, ge);
        ge += (int)(__float_as_uint(sc) >> 23) - 127;
        by.e_early = ge;
        by.early = scaled(factor, ge);
        {
            float2 P[1 << M];
            load_state<M>(P, slice + (size_t)c * S::STATE, lane);
            steps<0, S::HI>(P, c, w, sc);
            store_state<M>(P, ck_in, lane);
            steps<S::HI, M + 1>(P, c, w, sc);
            exchange(P);
            store_state<M>(P, xch, lane);
            steps<M + 1, M + 1 + S::HO>(P, c, w, sc);
            store_state<M>(P, ck_out, lane);
        }
        back_from<M + 1 + S::HO, D>(ck_out, G, c, w, sc, by);
        back_from<M + 1, M + 1 + S::HO>(xch, G, c, w, sc, by);
        exchange(G);
        back_from<S::HI, M + 1>(ck_in, G, c, w, sc, by);
        back_from<0, S::HI>(slice + (size_t)c * S::STATE, G, c, w, sc, by);
        float m = 0.f;
#pragma unroll
        for (int k = 0; k < (1 << M); ++k) m = fmaxf(m, fmaxf(fabsf(G[k].x), fabsf(G[k].y)));
        const float up = rescale<kAdjointTop>(unit_max(m), ge);
#pragma unroll
        for (int k = 0; k < (1 << M); ++k) G[k] = mul2(dup(up), G[k]);
        return by.lost;
    }
};

template <int D>
__global__ void __launch_bounds__(32 * GradLanes<D>::WARPS, D == 11 ? 3 : (D == 9 ? 3 : 4))
grad_gate_kernel(GradDenseArgs g) {
    using S = GradLanes<D>;
    constexpr int M = S::M, N = S::N;
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, wl = tid & 31;
    float4* tab = reinterpret_cast<float4*>(smem);
    {
        bool ok = true;
        for (int i = tid; i < N; i += 32 * S::WARPS) {
            const int c = i / D, j = i % D, r = grad_row(D, c, j);
            const float4 p = reinterpret_cast<const float4*>(g.noise)[r * D + c];
            const float sum = (p.x + p.y) + (p.z + p.w);
            ok = ok && p.x >= 0.f && p.y >= 0.f && p.z >= 0.f && p.w >= 0.f && fabsf(sum - 1.f) <= 1e-6f;
            const float4 v = flip_ctrl(p, (r & 1) == 0);
            if (D == 11)
                tab[i] = v;
            else
                for (uint32_t e = 0; e < 4; ++e) tab[4 * i + e] = permuted(v, e);
        }
        if (!ok && blockIdx.x == 0) atomicOr(g.status, 1 << MLD_ERR_INVALID_ARG);
    }
    unsigned char* mine = smem + S::kTable + (size_t)warp * ((S::kWarpBytes + 15) & ~(size_t)15);
    float2* states = reinterpret_cast<float2*>(mine);
    double* accs = reinterpret_cast<double*>(states + (size_t)S::UPW * S::UNIT);
    float* scales = reinterpret_cast<float*>(accs + (size_t)S::UPW * N * 4);
    uint32_t* words = reinterpret_cast<uint32_t*>(scales + S::UPW * (D + 2));
    for (int i = wl; i < S::UPW * N * 4; i += 32) accs[i] = 0.0;
    __syncthreads();

    const int u = wl / S::LANES;
    const int64_t gw = (int64_t)blockIdx.x * S::WARPS + warp, nw = (int64_t)gridDim.x * S::WARPS;
    Lane<D> L;
    L.tab = tab;
    L.xch = states + (size_t)u * S::UNIT;
    L.ck_in = L.xch + S::XCH;
    L.ck_out = L.ck_in + S::STATE;
    L.slice = reinterpret_cast<float2*>(g.lws) + (gw * S::UPW + u) * S::kSlice;
    L.acc = accs + (size_t)u * N * 4;
    L.scale = scales + u * (D + 2);
    L.lane = wl % S::LANES;
    const int lane = L.lane;
    // entries of the ends: even positions 0 (position of pair M, register bit t at its side's distance t + 1)
    bool lane_end = true;
#pragma unroll
    for (int t = 0; t < M; ++t) lane_end = lane_end && !(((M + 1 + t) & 1) == 0 && L.bit(t));
    const auto end_state = [&](float2 (&P)[1 << M], float v) {
#pragma unroll
        for (int k = 0; k < (1 << M); ++k) {
            bool zero = false;
#pragma unroll
            for (int t = 0; t < M; ++t) zero = zero || (((M + 1 + t) & 1) == 0 && (k >> t & 1));
            const float x = zero || !lane_end ? 0.f : v;
            P[k] = make_float2(x, (M & 1) == 0 ? 0.f : x);
        }
    };

    const int64_t units = 2 * g.B, chunks = (units + S::UPW - 1) / S::UPW;
    for (int64_t chunk = gw; chunk < chunks; chunk += nw) {
        const int64_t unit = chunk * S::UPW + u;
        const bool live = unit < units;
        const int64_t b = (live ? unit : units - 1) >> 1;
        L.lz = (int)(unit & 1);
        __syncwarp();
        for (int s = 0; s < S::SPW; ++s) {
            const int64_t bs = S::UPW > 1 ? chunk * S::SPW + s : b;
            const uint64_t* syn = g.syn + (bs < g.B ? bs : g.B - 1) * S::WORDS;
            const int l = wl < 2 * D ? wl : 0;
#pragma unroll
            for (int c = 0; c < D; ++c) {
                const int r = grad_row(D, c, l >> 1), z = ((l & 1) ^ r ^ 1) & 1;     // even rows: flip = x
                const uint64_t* mk = g.dmask + ((size_t)(r * D + c) * 2 + z) * S::WORDS;
                uint64_t x = 0;
#pragma unroll
                for (int w = 0; w < S::WORDS; ++w) x ^= syn[w] & mk[w];
                const uint32_t word = __ballot_sync(0xffffffffu, wl < 2 * D && (__popcll(x) & 1));
                if (wl == 0) words[s * D + c] = word;
            }
        }
        __syncwarp();
        L.words = words + (u >> 1) * D;

        // forward: the state at each column's start to the slice; the last
        // column once per l_X (one call site each way: the program of
        // d = 11 inlined twice takes 1.73 ms instead of 1.49)
        float2 P[1 << M];
        end_state(P, __uint_as_float((uint32_t)(127 + kGradTop) << 23));
        int e2 = -kGradTop, ez[2];
        float z[2];
#pragma unroll 1
        for (int pass = 0; pass <= D; ++pass) {
            const int c = pass < D ? pass : D - 1;
            if (pass < D)
                store_state<M>(P, L.slice + (size_t)c * S::STATE, lane);
            else
                load_state<M>(P, L.slice + (size_t)c * S::STATE, lane);
            int e = e2;
            L.column(P, c, L.word(c, pass == D), pass, e);
            if (c < D - 1) {
                e2 = e;
                continue;
            }
            float2 m[1 << M];
            end_state(m, 1.f);
            float sum = 0.f;
#pragma unroll
            for (int k = 0; k < (1 << M); ++k) sum = fmaf(P[k].x, m[k].x, fmaf(P[k].y, m[k].y, sum));
#pragma unroll
            for (int o = 1; o < S::LANES; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (pass == D) {
                z[1] = sum;
                ez[1] = e;
            } else {
                z[0] = sum;
                ez[0] = e;
            }
        }
        if (g.logP && live && lane < 2) {
            const float zz = lane ? z[1] : z[0];
            g.logP[2 * unit + lane] = zz < INFINITY ? ln_scaled(zz, lane ? ez[1] : ez[0]) : (double)NAN;
        }
        if (!g.dlogP) continue;
        // weights of the two classes' adjoints; a class of probability zero (or not finite) has none
        const double u0 = live ? g.dlogP[2 * (live ? unit : 0)] : 0.0, u1 = live ? g.dlogP[2 * (live ? unit : 0) + 1] : 0.0;
        const bool ok0 = u0 != 0.0 && z[0] > 0.f && z[0] < INFINITY, ok1 = u1 != 0.0 && z[1] > 0.f && z[1] < INFINITY;
        if (!__any_sync(0xffffffffu, ok0 || ok1)) continue;
        // the last column for l_X = 0 and 1, each with its own factor; then the
        // others for the sum of the two adjoint states, the smaller one scaled
        // to the larger one's factor (or one after the other: a second pass)
        float2 G[1 << M];
        float2* first = L.slice + (size_t)D * S::STATE;
        float2* second = first - S::STATE;               // the last column's start, read by then
        double c0 = ok0 ? u0 / (double)z[0] : 0.0, c1 = ok1 ? u1 / (double)z[1] : 0.0;
        const int top = 1023 - max(ok0 ? (__double2hiint(u0) >> 20) & 0x7ff : 0, ok1 ? (__double2hiint(u1) >> 20) & 0x7ff : 0);
        Twin want0 = xz::make<Twin>(ok0 ? scaled(u0, top) : 0.0), want1 = xz::make<Twin>(ok1 ? scaled(u1, top) : 0.0);
        const float moduli = fabsf(want0.hi) + fabsf(want1.hi), slack = 0.125f * moduli;
        double factor = 0.0;
        const Twin none{0.f, 0.f};
        Twin per = none, want = none;
        float trust = 0.f;
        bool apart = false, lost = false;
        int ge = 0, ge0 = 0, ge1 = 0, passes = 1;
#pragma unroll 1
        for (int pass = 0; pass < passes; ++pass) {
#pragma unroll 1
            for (int step = pass ? 2 : 0; step <= D; ++step) {
                const int c = step < 2 ? D - 1 : D - step;
                if (step <= 2) {
                    bool one = step == 1;
                    float share = 0.f;
                    if (step == 2) {
                        // f 2^e of the two: the larger, and the smaller's share of it
                        one = fabs(scaled(c1, ge1 - ge0)) > fabs(c0);
                        const double small = one ? scaled(c0, ge0 - ge1) : scaled(c1, ge1 - ge0), big = one ? c1 : c0;
                        const double ratio = small == 0.0 ? 0.0 : small / big;
                        apart = small != 0.0 && (fabs(ratio) < kApart || fabsf(want0.hi + want1.hi) < kOpposed * moduli);
                        if (pass == 0) passes = __any_sync(0xffffffffu, apart) ? 2 : 1;
                        if (pass == 1) one = !one;
                        share = pass || apart ? 0.f : (float)ratio;
                    }
                    factor = pass && !apart ? 0.0 : (one ? c1 : c0);
                    per = xz::make<Twin>(scaled(factor, top));
                    want = pass && !apart ? none : (one ? want1 : want0);
                    if (step == 2 && pass == 0 && !apart) want = xz::plus(want0, want1);
                    trust = 0.125f * fabsf(want.hi);
                    ge = step < 2 ? -kAdjointTop : (one ? ge1 : ge0);
                    if (step < 2) {
                        end_state(G, __uint_as_float((uint32_t)(127 + kAdjointTop) << 23));
                    } else {
                        const float2 *g = one ? second : first, *h = one ? first : second;
#pragma unroll
                        for (int k = 0; k < (1 << M); ++k)
                            G[k] = fma2(dup(share), h[(k << M) + lane], g[(k << M) + lane]);
                    }
                }
                if (L.back_column(G, c, L.word(c, step == 1), step == 1 ? D : c, factor, ge, per, want, slack, trust)) {
                    lost = true;
                    factor = 0.0;
                    per = want = none;
                    trust = 0.f;
                    if (step < 2) {
                        (step ? c1 : c0) = 0.0;
                        (step ? want1 : want0) = none;
                    }
                }
                if (step < 2) {
                    store_state<M>(G, step ? second : first, lane);
                    (step ? ge1 : ge0) = ge;
                }
            }
        }
        if (lost && lane == 0) atomicOr(g.status, 1 << MLD_ERR_NUMERIC);
    }
    // the warp's units in order, then the block's warps: one partial sum a block
    __syncthreads();
    double* part = reinterpret_cast<double*>(reinterpret_cast<float2*>(g.lws) +
                                             (int64_t)gridDim.x * S::WARPS * S::UPW * S::kSlice) +
                   (int64_t)blockIdx.x * N * 4;
    for (int i = tid; i < N * 4; i += 32 * S::WARPS) {
        double s = 0.0;
        for (int w = 0; w < S::WARPS; ++w) {
            const double* a = reinterpret_cast<const double*>(
                smem + S::kTable + (size_t)w * ((S::kWarpBytes + 15) & ~(size_t)15) + (size_t)S::UPW * S::UNIT * 8);
            for (int v = 0; v < S::UPW; ++v) s += a[(size_t)v * N * 4 + i];
        }
        part[i] = s;
    }
}

// One block per gradient entry: thread t sums the blocks t, t + 256, .. in
// order, then a fixed tree.
__global__ void __launch_bounds__(256) grad_sum_kernel(const double* __restrict__ part, int64_t blocks, int n4,
                                                       double* __restrict__ dnoise) {
    __shared__ double sums[256];
    const int e = blockIdx.x, t = threadIdx.x;
    double s = 0.0;
    for (int64_t b = t; b < blocks; b += 256) s += part[b * n4 + e];
    sums[t] = s;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (t < h) sums[t] += sums[t + h];
        __syncthreads();
    }
    if (t == 0) dnoise[e] += sums[0];
}

constexpr int kMaxDevices = 64;

template <int D>
int64_t blocks_d(int64_t B) {
    using S = GradLanes<D>;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
    static std::atomic<int> resident[kMaxDevices];
    int n = resident[dev].load(std::memory_order_acquire);
    if (n == 0) {
        int sms = 0, per_sm = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaFuncSetAttribute(grad_gate_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kBytes) !=
                cudaSuccess ||
            cudaFuncSetAttribute(grad_gate_kernel<D>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, grad_gate_kernel<D>, 32 * S::WARPS, S::kBytes) !=
                cudaSuccess ||
            per_sm < 1)
            return 0;
        n = sms * per_sm;
        resident[dev].store(n, std::memory_order_release);
    }
    const int64_t per = (int64_t)S::WARPS * S::UPW, need = (2 * B + per - 1) / per;
    return need < n ? need : n;
}

template <int D>
bool launch_d(const GradDenseArgs& a, int64_t blocks, cudaStream_t s) {
    using S = GradLanes<D>;
    grad_gate_kernel<D><<<(unsigned)blocks, 32 * S::WARPS, S::kBytes, s>>>(a);
    if (cudaGetLastError() != cudaSuccess) return false;
    if (!a.dlogP) return true;
    const double* part = reinterpret_cast<const double*>(reinterpret_cast<const float2*>(a.lws) +
                                                         blocks * S::WARPS * S::UPW * S::kSlice);
    grad_sum_kernel<<<4 * S::N, 256, 0, s>>>(part, blocks, 4 * S::N, a.dnoise);
    return cudaGetLastError() == cudaSuccess;
}

template <int D>
constexpr int64_t workspace_d() {
    using S = GradLanes<D>;
    return 2 * (int64_t)S::WARPS * S::UPW * S::kSlice + 2 * 4 * S::N;
}

}  // namespace

int64_t grad_gate_blocks(int d, int64_t B) {
    switch (d) {
        case 3: return blocks_d<3>(B);
        case 5: return blocks_d<5>(B);
        case 7: return blocks_d<7>(B);
        case 9: return blocks_d<9>(B);
        case 11: return blocks_d<11>(B);
    }
    return 0;
}

int64_t grad_gate_workspace_floats(int d) {
    switch (d) {
        case 3: return workspace_d<3>();
        case 5: return workspace_d<5>();
        case 7: return workspace_d<7>();
        case 9: return workspace_d<9>();
        case 11: return workspace_d<11>();
    }
    return 0;
}

bool launch_grad_gate(int d, const GradDenseArgs& a, int64_t blocks, cudaStream_t s) {
    switch (d) {
        case 3: return launch_d<3>(a, blocks, s);
        case 5: return launch_d<5>(a, blocks, s);
        case 7: return launch_d<7>(a, blocks, s);
        case 9: return launch_d<9>(a, blocks, s);
        case 11: return launch_d<11>(a, blocks, s);
    }
    return false;
}

}  // namespace mld
