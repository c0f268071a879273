// Untruncated decode by the column transfer (mld_gate.cuh): d = 3, 5, 7 with
// one thread per (syndrome, l_Z), d = 9, 11, 13 with the state spread over 16,
// 32 or 64 lanes. All four classes, the decision and the check of the noise
// in one launch; a second one over ties at d <= 9.
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "mld_exact_impl.cuh"
#include "mld_gate.cuh"
#include "mld_gate.h"
#include "mld_internal.h"

namespace mld {
namespace {

using namespace gate;

constexpr int kInvalid = 1 << MLD_ERR_INVALID_ARG;
constexpr int kNumeric = 1 << MLD_ERR_NUMERIC;

// Row of processing step j of column c: rising in even columns, falling in
// odd ones.
__host__ __device__ constexpr int row_of(int d, int c, int j) { return (c & 1) ? d - 1 - j : j; }

__device__ __forceinline__ bool valid_row(float4 v) {
    const float sum = (v.x + v.y) + (v.z + v.w);
    return v.x >= 0.f && v.y >= 0.f && v.z >= 0.f && v.w >= 0.f && fabsf(sum - 1.f) <= 1e-6f;   // NaN fails
}
__device__ __forceinline__ bool valid_rate(float p) { return p >= 0.f && p <= 1.f; }

// Representative bit of (column c, step j, k = 0 control / 1 flip) as a mask
// over syndrome bits: row of the destabiliser table.
__device__ __forceinline__ const uint64_t* mask_row(const uint64_t* dmask, int d, int words, int c, int j, int k) {
    const int r = row_of(d, c, j);
    const int z = (k ^ r ^ 1) & 1;                    // even rows: flip = x part, control = z part
    return dmask + ((size_t)(r * d + c) * 2 + z) * words;
}

// Classes within this of the best are a tie: four times the largest difference
// seen between two kernels' FP32 roundings of one ln Z (2.5e-6 at d = 9).
constexpr double kTie = 1e-5;

__host__ __device__ inline ExactArgs exact_args(const GateArgs& a) {
    ExactArgs e;
    e.dmask = a.dmask;
    e.noise = a.noise;
    e.syn = a.syn;
    e.logP = a.logP;
    e.status = a.status;
    e.B = a.B;
    e.noise_mode = a.noise_mode;
    return e;
}

// The decision among four values held by two threads (l = 2 lZ + lX); equal
// values and all -inf go to the lowest class. Bit 7 marks a tie.
__device__ __forceinline__ int best_of_pair(double l0, double l1, int lz, unsigned mask) {
    const int mine = l1 > l0 ? 1 : 0;
    const double v = mine ? l1 : l0, w = mine ? l0 : l1;
    const double ov = __shfl_xor_sync(mask, v, 1), ow = __shfl_xor_sync(mask, w, 1);
    const int omine = __shfl_xor_sync(mask, mine, 1);
    const bool other = lz == 0 ? ov > v : !(v > ov);
    const double best = other ? ov : v, second = other ? fmax(v, ow) : fmax(w, ov);
    const int at = other ? 2 * (lz ^ 1) + omine : 2 * lz + mine;
    return at | (best - second < kTie ? 0x80 : 0);      // -inf - -inf compares false
}

// ---------------------------------------------------------------- d <= 7 ----
// A thread holds the whole state (2^d floats: 8, 32, 128 registers), so no
// column exchanges anything; the two threads of a syndrome (l_Z = 0, 1) share
// its representative bits. Position 0 is the pair's. Bound: FP32 pipe (two
// operations an entry and gate).

template <int D>
struct ThreadShape {
    static constexpr int N = D * D;
    static constexpr int NB = D - 1;
    static constexpr int NT = 128;
    static constexpr int PAIRS = (D + 1) / 2;           // column pairs: even column low half, odd high half
};

template <int NB>
__device__ __forceinline__ float2 finish(float2 (&S)[1 << NB], const float4* w, int (&e)[2]) {
    // last column from its second row on: halves are l_X = 0, 1; w[0] odd row
    // (control toggled by l_X), w[1] even row (flip toggled, new bit 0). The
    // classes part here (one may pay a rate in every row), so each is rescaled
    // by itself between the row pairs.
    gate_bit<NB, 0>(S, w[0]);
    const float4 v = w[1];
    float2 out[1 << (NB - 2)];
#pragma unroll
    for (int k = 0; k < (1 << (NB - 2)); ++k) {
        float2 acc = make_float2(0.f, 0.f);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = h ^ (NB > 2 ? k & 1 : 0);
            const float a = c ? v.y : v.x, b = c ? v.w : v.z;
            acc = fma2(make_float2(a, b), S[4 * k + h], acc);
            acc = fma2(make_float2(b, a), S[4 * k + 2 + h], acc);
        }
        out[k] = acc;
    }
    if constexpr (NB == 2) {
        return out[0];
    } else {
        float2 m = out[0];
#pragma unroll
        for (int k = 1; k < (1 << (NB - 2)); ++k) m = make_float2(fmaxf(m.x, out[k].x), fmaxf(m.y, out[k].y));
        const float2 sc = make_float2(rescale<>(__float_as_uint(m.x), e[0]), rescale<>(__float_as_uint(m.y), e[1]));
#pragma unroll
        for (int k = 0; k < (1 << (NB - 2)); ++k) out[k] = mul2(sc, out[k]);
        return finish<NB - 2>(out, w + 2, e);
    }
}

template <int D, bool DEPOL, bool TIES>
__device__ __forceinline__ void thread_body(const GateArgs& a, const float4* table) {
    using S = ThreadShape<D>;
    constexpr int FPW = exact::LayoutOf<D>::lay.floats_per_warp;
    __shared__ float4 tie_ws[TIES ? S::NT / 32 * FPW / 4 : 1];
    __shared__ float4 tab[DEPOL ? 1 : S::N * 4];                 // [c][j][e]: weights [flip][ctrl] under e
    __shared__ uint64_t masks[S::PAIRS * 2 * D * 2];             // [c][j][k]
    const int tid = threadIdx.x;
    if (!DEPOL) {
        bool ok = true;
        for (int i = tid; i < S::N; i += S::NT) {
            const int c = i / D, j = i % D, r = row_of(D, c, j);
            const float4 p = table[r * D + c];
            ok = ok && valid_row(p);
            const float4 v = flip_ctrl(p, (r & 1) == 0);
            for (uint32_t e = 0; e < 4; ++e) tab[4 * i + e] = permuted(v, e);
        }
        if (!ok && a.status && blockIdx.x == 0) atomicOr(a.status, kInvalid);
    }
    for (int i = tid; i < S::PAIRS * 2 * D * 2; i += S::NT) {
        const int c = i / (2 * D), j = (i / 2) % D, k = i & 1;
        masks[i] = c < D ? *mask_row(a.dmask, D, 1, c, j, k) : 0;
    }
    __syncthreads();

    const int lz = tid & 1;
    const int64_t step = (int64_t)gridDim.x * (S::NT / 2);
    for (int64_t b0 = (int64_t)blockIdx.x * (S::NT / 2) + (tid >> 5) * 16; b0 < a.B; b0 += step) {
        const int64_t b = b0 + ((tid & 31) >> 1);
        const bool live = b < a.B;
        const int64_t bb = live ? b : a.B - 1;
        const uint64_t s = a.syn[bb];
        float p0 = 0.f, p1 = 0.f;
        if (DEPOL) {
            const float p = a.noise[bb];
            if (!valid_rate(p) && a.status) atomicOr(a.status, kInvalid);
            p0 = 1.f - p;
            p1 = p * (1.f / 3.f);
        }
        // representative bits, two columns to a word: each thread of the pair
        // forms one of the two and they exchange them
        uint32_t W[S::PAIRS];
#pragma unroll
        for (int i = 0; i < S::PAIRS; ++i) {
            const uint64_t* mk = masks + (2 * i + lz) * 2 * D;
            uint32_t w = 0;
#pragma unroll
            for (int k = 0; k < 2 * D; ++k) w |= (uint32_t)(__popcll(s & mk[k]) & 1) << k;
            const uint32_t o = __shfl_xor_sync(0xffffffffu, w, 1);
            W[i] = lz ? (o | (w << 16)) : (w | (o << 16));
            // Z on row 0: control of the first step of even columns and of the last of odd ones
            W[i] ^= lz ? (1u | (1u << (16 + 2 * (D - 1)))) : 0u;
        }
        const auto weight = [&](int c, int j, uint32_t word) {
            const uint32_t e = (word >> (2 * j)) & 3;
            if (DEPOL) return make_float4(e == 0 ? p0 : p1, e == 1 ? p0 : p1, e == 2 ? p0 : p1, e == 3 ? p0 : p1);
            return tab[(c * D + j) * 4 + e];
        };
        float2 P[1 << S::NB];
        int e2 = -kTop;
        {
            const float4 v = weight(0, 0, W[0]);                 // row 0: old bit 0; o = old bit of row 1
            const float2 top = dup(top_scale());
            const float2 ext[2] = {mul2(top, make_float2(v.x, v.z)), mul2(top, make_float2(v.y, v.w))};
            const auto w = [&](int T) { return weight(0, T + 1, W[0]); };
            Grow<S::NB, 0, decltype(w)>::odd(P, ext, w);
        }
        float sc = rescale<>(__float_as_uint(max_of(P)), e2);
#pragma unroll 1
        for (int i = 0; 2 * i + 1 < D - 1; ++i) {
            {
                const int c = 2 * i + 1;                         // falling: steps 0..D-2 on bits D-2..0, then the pair
                const uint32_t word = W[0] >> 16;
                float4 v = weight(c, 0, word);
                v = make_float4(v.x * sc, v.y * sc, v.z * sc, v.w * sc);
                gate_bit<S::NB, S::NB - 1>(P, v);
                const auto w = [&](int T) { return weight(c, D - 2 - T, word); };
                if constexpr (S::NB >= 2) gates_down<S::NB, S::NB - 2>(P, w);
                gate_pair<S::NB>(P, weight(c, D - 1, word));
                sc = rescale<>(__float_as_uint(max_of(P)), e2);
            }
#pragma unroll
            for (int k = 0; k + 1 < S::PAIRS; ++k) W[k] = W[k + 1];
            if (2 * i + 2 < D - 1) {
                const int c = 2 * i + 2;                         // rising: the pair, then bits 0..D-2
                float4 v = weight(c, 0, W[0]);
                v = make_float4(v.x * sc, v.y * sc, v.z * sc, v.w * sc);
                gate_pair<S::NB>(P, v);
                const auto w = [&](int T) { return weight(c, T + 1, W[0]); };
                gates_up<S::NB, 0>(P, w);
                sc = rescale<>(__float_as_uint(max_of(P)), e2);
            }
        }
        // last column, both l_X at once: X on the column flips row 0's new bit,
        // so its two values are the two classes
        float4 wl[D];
#pragma unroll
        for (int j = 0; j < D; ++j) wl[j] = weight(D - 1, j, W[0]);
        wl[0] = make_float4(wl[0].x * sc, wl[0].y * sc, wl[0].z * sc, wl[0].w * sc);
        gate_pair<S::NB>(P, wl[0]);
        int e[2] = {e2, e2};
        const float2 z = finish<S::NB>(P, wl + 1, e);
        const double l0 = ln_scaled(z.x, e[0]), l1 = ln_scaled(z.y, e[1]);
        const int best = best_of_pair(l0, l1, lz, 0xffffffffu);
        if (live) {
            if ((!(z.x < INFINITY) || !(z.y < INFINITY)) && a.status) atomicOr(a.status, kNumeric);
            const bool mark = TIES && a.mark_ties && lz == 0 && (best & 0x80);
            a.logP[b * 4 + 2 * lz] = mark ? (double)NAN : l0;
            a.logP[b * 4 + 2 * lz + 1] = l1;
            if (a.argmax && lz == 0) a.argmax[b] = (uint8_t)(best & 3);
        }
        if constexpr (TIES) {
            if (!a.mark_ties) {
                unsigned marked = __ballot_sync(0xffffffffu, live && lz == 0 && (best & 0x80));
                while (marked) {
                    const int l = __ffs(marked) - 1;
                    marked &= marked - 1;
                    exact::decide_tie<D, MLD_FP32>(exact_args(a), a.argmax,
                                                   reinterpret_cast<float*>(tie_ws) + (size_t)(tid >> 5) * FPW,
                                                   b0 + (l >> 1), tid & 31);
                    __syncwarp();
                }
            }
        }
    }
}

// ---------------------------------------------------------------- d >= 9 ----

template <int D>
struct LaneShape {
    static constexpr int N = D * D;
    static constexpr int M = (D - 1) / 2;               // index bits, lane bits
    static constexpr int LANES = 1 << M;                // threads of a unit (syndrome, l_Z)
    static constexpr int TS = 2 * LANES;                // threads of a syndrome
    static constexpr int WORDS = (N - 1 + 63) / 64;
    static constexpr int STRIDE = LANES + 1;            // float2 units: rows and columns both conflict-free
    static constexpr int XCH = LANES * STRIDE;          // float2 of one unit's exchange buffer
    // d = 9: several syndromes share a block and its tables (weights under all
    // four representatives, masks in step order); above, one block is one
    // syndrome and the table is kept compact so that 10 (d = 11) and 3
    // (d = 13) blocks fit an SM's shared memory
    static constexpr bool WARP = D == 9;
    static constexpr int SLOTS = 8;                     // syndromes whose logarithms are taken together
};

template <int D, bool DEPOL>
size_t lane_smem(int syndromes_per_block) {
    using S = LaneShape<D>;
    size_t bytes = (size_t)syndromes_per_block * (2 * S::XCH * sizeof(float2) + S::SLOTS * 4 * 8 + 64);
    if (!DEPOL) bytes += (size_t)S::N * 16 * (S::WARP ? 4 : 1);
    if (S::WARP) bytes += (size_t)D * 2 * D * S::WORDS * 8;
    return bytes;
}

// Last column on the register side, from its second step on: q0, q1 are the
// states of l_X = 0, 1 over index bits 0..T (and T+1, the odd position summed
// after the even one below it). Weights of l_X = 1: flip toggled in even rows,
// control in odd ones.
template <int M, int T, class W>
struct Shrink {
    static constexpr int J = M - 1 - T;
    static constexpr bool kEven = (J & 1) == 0;
    static __device__ __forceinline__ void run(float2* q0, float2* q1, const W& w) {
        const float4 v = w(J);
        if constexpr (kEven) {
#pragma unroll
            for (int lx = 0; lx < 2; ++lx) {
                float2* q = lx ? q1 : q0;
                const float4 u = lx ? make_float4(v.z, v.w, v.x, v.y) : v;
                float2 out[1 << T];
#pragma unroll
                for (int k = 0; k < (1 << T); ++k) {
                    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int c = h ^ (T > 0 ? (k >> (T > 0 ? T - 1 : 0)) & 1 : 0);
                        const float2 A = T == 0 ? (c ? make_float2(u.y, u.x) : make_float2(u.x, u.y)) : dup(c ? u.y : u.x);
                        const float2 B = T == 0 ? (c ? make_float2(u.w, u.z) : make_float2(u.z, u.w)) : dup(c ? u.w : u.z);
                        acc = fma2(A, q[(h << (T + 1)) | k], acc);
                        acc = fma2(B, q[(h << (T + 1)) | (1 << T) | k], acc);
                    }
                    out[k] = acc;
                }
#pragma unroll
                for (int k = 0; k < (1 << T); ++k) q[k] = out[k];
            }
        } else {
            gate_bit<T + 1, T>(*reinterpret_cast<float2(*)[2 << T]>(q0), v);
            gate_bit<T + 1, T>(*reinterpret_cast<float2(*)[2 << T]>(q1), make_float4(v.y, v.x, v.w, v.z));
        }
        if constexpr (T > 0) Shrink<M, T - 1, W>::run(q0, q1, w);
    }
};

template <int D>
__device__ __forceinline__ void unit_sync(int lz) {
    if constexpr (LaneShape<D>::LANES == 64)
        asm volatile("bar.sync %0, 64;" ::"r"(1 + lz) : "memory");
    else
        __syncwarp();
}
template <int D>
__device__ __forceinline__ void group_sync() {
    if constexpr (LaneShape<D>::WARP)
        __syncwarp();
    else
        __syncthreads();
}

template <int D, bool DEPOL>
__device__ __forceinline__ void lane_body(const GateArgs& a, const float4* table) {
    using S = LaneShape<D>;
    constexpr int M = S::M;
    extern __shared__ float4 smem[];
    const int tid = threadIdx.x, nt = blockDim.x;
    const int groups = nt / S::TS, g = tid / S::TS, gt = tid % S::TS;
    float4* tab = smem;                                           // [c][j] (x 4 representatives at d = 9)
    uint64_t* masks = reinterpret_cast<uint64_t*>(tab + (DEPOL ? 0 : S::N * (S::WARP ? 4 : 1)));
    float2* xch0 = reinterpret_cast<float2*>(masks + (S::WARP ? D * 2 * D * S::WORDS : 0));
    float* slots0 = reinterpret_cast<float*>(xch0 + (size_t)groups * 2 * S::XCH);
    if (!DEPOL) {
        bool ok = true;
        for (int i = tid; i < S::N; i += nt) {
            const int c = i / D, j = i % D, r = row_of(D, c, j);
            const float4 p = table[r * D + c];
            ok = ok && valid_row(p);
            const float4 v = flip_ctrl(p, (r & 1) == 0);
            if (S::WARP)
                for (uint32_t e = 0; e < 4; ++e) tab[4 * i + e] = permuted(v, e);
            else
                tab[i] = v;
        }
        if (!ok && a.status && blockIdx.x == 0) atomicOr(a.status, kInvalid);
    }
    if (S::WARP)
        for (int i = tid; i < D * 2 * D; i += nt) {
            const uint64_t* mk = mask_row(a.dmask, D, S::WORDS, i / (2 * D), (i / 2) % D, i & 1);
            for (int w = 0; w < S::WORDS; ++w) masks[i * S::WORDS + w] = mk[w];
        }
    __syncthreads();

    float2* xch = xch0 + (size_t)g * 2 * S::XCH;
    float* slot_z = slots0 + g * (S::SLOTS * 8 + 16);             // [slot][class]
    int* slot_e = reinterpret_cast<int*>(slot_z + S::SLOTS * 4);
    float* pair_x = slot_z + S::SLOTS * 8;                        // [lz][..]: what the two warps of a unit exchange
    const int lane = gt % S::LANES, lz = gt / S::LANES;
    float2* X = xch + lz * S::XCH;
    const int wl = tid & 31;                                      // lane of the warp
    const int64_t ng = (int64_t)gridDim.x * groups, gid = (int64_t)blockIdx.x * groups + g;
    const int64_t lo = gid * a.B / ng, hi = (gid + 1) * a.B / ng;
    // lane bits as representative toggles: row t of the other side at index bit t
    const auto lb = [&](int t) { return (uint32_t)(lane >> t) & 1u; };

    for (int64_t b = lo; b < hi; ++b) {
        uint64_t s[S::WORDS];
#pragma unroll
        for (int w = 0; w < S::WORDS; ++w) s[w] = a.syn[b * S::WORDS + w];
        float p0 = 0.f, p1 = 0.f;
        if (DEPOL) {
            const float p = a.noise[b];
            if (!valid_rate(p) && a.status) atomicOr(a.status, kInvalid);
            p0 = 1.f - p;
            p1 = p * (1.f / 3.f);
        }
        // representative bits: lane L forms bit L (step L/2, control or flip)
        // of column c, a ballot makes the word, lane c keeps it
        uint32_t words = 0;
        {
            const int L = wl < 2 * D ? wl : 0;
#pragma unroll
            for (int c = 0; c < D; ++c) {
                const uint64_t* mk = S::WARP ? masks + (c * 2 * D + L) * S::WORDS
                                             : mask_row(a.dmask, D, S::WORDS, c, L >> 1, L & 1);
                uint64_t x = s[0] & mk[0];
#pragma unroll
                for (int w = 1; w < S::WORDS; ++w) x ^= s[w] & mk[w];
                const uint32_t word = __ballot_sync(0xffffffffu, wl < 2 * D && (__popcll(x) & 1));
                if (wl == c) words = word;
            }
        }
        const auto column_word = [&](int c) {
            // Z on row 0: control of the first step of even columns, of the last of odd ones
            const uint32_t w = __shfl_sync(0xffffffffu, words, c);
            return w ^ (lz ? ((c & 1) ? 1u << (2 * (D - 1)) : 1u) : 0u);
        };
        const auto weight = [&](int c, int j, uint32_t word, uint32_t toggle) {
            const uint32_t e = ((word >> (2 * j)) & 3) ^ toggle;
            if (DEPOL) return make_float4(e == 0 ? p0 : p1, e == 1 ? p0 : p1, e == 2 ? p0 : p1, e == 3 ? p0 : p1);
            return S::WARP ? tab[(c * D + j) * 4 + e] : permuted(tab[c * D + j], e);
        };
        float2 P[1 << M];
        int e2 = -kTop;
        {
            // column 0: the lane's own positions 0..M-1 (position p at lane bit
            // M-1-p) one by one, then M and the register side
            const uint32_t word = column_word(0);
            float u0 = 0.f, u1 = 0.f, v = top_scale();
            uint32_t prev = 0;
#pragma unroll
            for (int p = 0; p < M; ++p) {
                const uint32_t bit = lb(M - 1 - p);
                const float4 w = weight(0, p, word, (bit << 1) | prev);
                if ((p & 1) == 0) {
                    u0 = v * w.x;
                    u1 = v * w.y;
                } else {
                    v = fmaf(u0, w.x, u1 * w.z);
                }
                prev = bit;
            }
            const float4 w = weight(0, M, word, prev);
            const auto wo = [&](int T) { return weight(0, M + 1 + T, word, 0); };
            if constexpr ((M & 1) == 0) {
                const float2 ext[2] = {make_float2(v * w.x, v * w.z), make_float2(v * w.y, v * w.w)};
                Grow<M, 0, decltype(wo)>::odd(P, ext, wo);
            } else {
                const float2 cur[1] = {make_float2(fmaf(u0, w.x, u1 * w.z), fmaf(u0, w.z, u1 * w.x))};
                Grow<M, 0, decltype(wo)>::even(P, cur, wo);
            }
        }
#pragma unroll 1
        for (int c = 1; c < D - 1; ++c) {
            const uint32_t word = column_word(c);
            const auto wi = [&](int T) { return weight(c, M - 1 - T, word, 0); };
            gates_down<M, M - 1>(P, wi);
            gate_pair<M>(P, weight(c, M, word, lb(0)));
            // exchange the two sides; the largest entry goes along
            uint32_t mx = __float_as_uint(max_of(P));
            if constexpr (S::LANES == 16) {
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            } else {
                mx = __reduce_max_sync(0xffffffffu, mx);
            }
            if constexpr (S::LANES == 64)
                if (wl == 0) pair_x[lz * 8 + (lane >> 5)] = __uint_as_float(mx);
#pragma unroll
            for (int k = 0; k < (1 << M); ++k) X[lane * S::STRIDE + k] = P[k];
            unit_sync<D>(lz);
#pragma unroll
            for (int k = 0; k < (1 << M); ++k) P[k] = X[k * S::STRIDE + lane];
            if constexpr (S::LANES == 64)
                mx = max(__float_as_uint(pair_x[lz * 8]), __float_as_uint(pair_x[lz * 8 + 1]));
            unit_sync<D>(lz);
            const float sc = rescale<>(mx, e2);
            float4 v = weight(c, M + 1, word, 0);
            v = make_float4(v.x * sc, v.y * sc, v.z * sc, v.w * sc);
            gate_bit<M, 0>(P, v);
            const auto wo = [&](int T) { return weight(c, M + 1 + T, word, 0); };
            gates_up<M, 1>(P, wo);
        }
        // last column: row 0's new bit is 0, and X on the column (l_X = 1) flips
        // it, so the gate's two outputs are the two classes; even positions
        // drop out, each odd one is summed once the next row has used it
        const uint32_t word = column_word(D - 1);
        const auto wi = [&](int j) { return weight(D - 1, j, word, 0); };
        gate_bit<M, M - 1>(P, wi(0));
        Shrink<M, M - 2, decltype(wi)>::run(P, P + (1 << (M - 1)), wi);
        float v0, v1;
        if constexpr ((M & 1) == 0) {
            const float4 w = weight(D - 1, M, word, lb(0));
            const float2 *q0 = P, *q1 = P + (1 << (M - 1));
            v0 = fmaf(w.x, q0[0].x, w.z * q0[0].y) + fmaf(w.y, q0[1].x, w.w * q0[1].y);
            v1 = fmaf(w.z, q1[0].x, w.x * q1[0].y) + fmaf(w.w, q1[1].x, w.y * q1[1].y);
        } else {
            const float4 w = weight(D - 1, M, word, lb(0));       // control toggled by l_X
            const float2 q0 = P[0], q1 = P[1 << (M - 1)];
            const float x0 = fmaf(w.x, q0.x, w.z * q0.y), y0 = fmaf(w.z, q0.x, w.x * q0.y);
            const float x1 = fmaf(w.y, q1.x, w.w * q1.y), y1 = fmaf(w.w, q1.x, w.y * q1.y);
            const float4 u = weight(D - 1, M + 1, word, lb(1));
            const float ox0 = __shfl_xor_sync(0xffffffffu, x0, 1), oy0 = __shfl_xor_sync(0xffffffffu, y0, 1);
            const float ox1 = __shfl_xor_sync(0xffffffffu, x1, 1), oy1 = __shfl_xor_sync(0xffffffffu, y1, 1);
            v0 = fmaf(u.x, x0, u.z * ox0) + fmaf(u.y, y0, u.w * oy0);
            v1 = fmaf(u.z, x1, u.x * ox1) + fmaf(u.w, y1, u.y * oy1);
        }
        // the classes have parted on the register side (one may have paid a
        // rate in every row): each is rescaled by itself
        int e_0 = e2, e_1 = e2;
        {
            uint32_t m0 = __float_as_uint(v0), m1 = __float_as_uint(v1);
            if constexpr (S::LANES == 16) {
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) {
                    m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, o));
                    m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, o));
                }
            } else {
                m0 = __reduce_max_sync(0xffffffffu, m0);
                m1 = __reduce_max_sync(0xffffffffu, m1);
            }
            if constexpr (S::LANES == 64) {
                float* x = pair_x + lz * 8;
                if (wl == 0) {
                    x[(lane >> 5) * 2] = __uint_as_float(m0);
                    x[(lane >> 5) * 2 + 1] = __uint_as_float(m1);
                }
                unit_sync<D>(lz);
                m0 = __float_as_uint(fmaxf(x[0], x[2]));
                m1 = __float_as_uint(fmaxf(x[1], x[3]));
                unit_sync<D>(lz);
            }
            v0 *= rescale<>(m0, e_0);
            v1 *= rescale<>(m1, e_1);
        }
        // the lane side: valid where the even positions' lane bits are 0
#pragma unroll
        for (int t = M & 1; t < M; ++t) {
            const int j = M + 1 + t;
            const bool even = (j & 1) == 0;
            if (t == 5) {
                // d = 13: position 12 is the unit's warp bit; lanes 0 and 16 hold both values of position 11
                if ((wl & 15) == 0) {
                    pair_x[lz * 8 + (lane >> 5) * 4 + (wl >> 4) * 2] = v0;
                    pair_x[lz * 8 + (lane >> 5) * 4 + (wl >> 4) * 2 + 1] = v1;
                }
                unit_sync<D>(lz);
                const float* x = pair_x + lz * 8;
                const float4 w = weight(D - 1, j, word, 0);
                v0 = fmaf(w.x, x[0], w.z * x[4]) + fmaf(w.y, x[2], w.w * x[6]);
                v1 = fmaf(w.z, x[1], w.x * x[5]) + fmaf(w.w, x[3], w.y * x[7]);
                unit_sync<D>(lz);
            } else {
                const uint32_t tog = even ? lb(t - 1) ^ (t + 1 < M ? lb(t + 1) : 0u) : lb(t + 1);
                const float4 w = weight(D - 1, j, word, tog);
                const float o0 = __shfl_xor_sync(0xffffffffu, v0, 1 << t), o1 = __shfl_xor_sync(0xffffffffu, v1, 1 << t);
                v0 = fmaf(w.x, v0, w.z * o0);
                v1 = even ? fmaf(w.z, v1, w.x * o1) : fmaf(w.y, v1, w.w * o1);
                if (even) {
                    v0 += __shfl_xor_sync(0xffffffffu, v0, 1 << (t - 1));
                    v1 += __shfl_xor_sync(0xffffffffu, v1, 1 << (t - 1));
                }
            }
        }
        const int slot = (int)(b - lo) % S::SLOTS;
        if (lane == 0) {
            slot_z[slot * 4 + 2 * lz] = v0;
            slot_z[slot * 4 + 2 * lz + 1] = v1;
            slot_e[slot * 4 + 2 * lz] = e_0;
            slot_e[slot * 4 + 2 * lz + 1] = e_1;
        }
        // logarithms, decisions and stores of up to eight syndromes at a time:
        // one lane per (syndrome, class)
        if (slot == S::SLOTS - 1 || b == hi - 1) {
            group_sync<D>();
            if (gt < 32) {
                const bool live = (gt >> 2) <= slot;
                const float z = live ? slot_z[gt] : 1.f;
                const double l = ln_scaled(z, live ? slot_e[gt] : 0);
                if (!(z < INFINITY) && a.status) atomicOr(a.status, kNumeric);
                double best = l;
                int at = gt & 3;
#pragma unroll
                for (int o = 1; o < 4; o <<= 1) {
                    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
                    const int oa = __shfl_xor_sync(0xffffffffu, at, o);
                    if (ob > best || (ob == best && oa < at)) {
                        best = ob;
                        at = oa;
                    }
                }
                const unsigned near = __ballot_sync(0xffffffffu, best - l < kTie);      // -inf - -inf compares false
                const bool tie = a.mark_ties && __popc(near >> (gt & 28) & 15u) > 1;
                const int64_t b0 = b - slot;
                if (live) {
                    a.logP[b0 * 4 + gt] = tie && (gt & 3) == 0 ? (double)NAN : l;
                    if (a.argmax && (gt & 3) == 0) a.argmax[b0 + (gt >> 2)] = (uint8_t)at;
                }
            }
            group_sync<D>();
        }
    }
}

// ---------------------------------------------------------------- kernels ----

template <int D>
constexpr int kBlock = D <= 7 ? 128 : (D == 9 ? 256 : LaneShape<(D > 7 ? D : 9)>::TS);
template <int D>
constexpr int kBlocksPerSm = D == 3 || D == 5 ? 8 : (D == 7 ? 3 : (D == 9 ? 4 : (D == 11 ? 10 : 3)));

template <int D, bool DEPOL, bool TIES>
__device__ __forceinline__ void body(const GateArgs& a, const float4* table) {
    if constexpr (D <= 7)
        thread_body<D, DEPOL, TIES>(a, table);
    else
        lane_body<D, DEPOL>(a, table);
}

template <int D, bool DEPOL>
__global__ void __launch_bounds__(kBlock<D>, kBlocksPerSm<D>) gate_decode_kernel(GateArgs a) {
    body<D, DEPOL, true>(a, reinterpret_cast<const float4*>(a.noise));
}

template <int D>
__global__ void __launch_bounds__(kBlock<D>, kBlocksPerSm<D>)
gate_table_kernel(GateArgs a, const __grid_constant__ GateTable t) {
    body<D, false, false>(a, reinterpret_cast<const float4*>(&t.p[0][0]));
}

// Resident blocks per SM and the SM count, looked up once per device, kernel
// and block size (an occupancy query costs more host time than the launch).
constexpr int kMaxDevices = 64;

int sm_count(int dev) {
    static std::atomic<int> cache[kMaxDevices];
    int n = cache[dev].load(std::memory_order_relaxed);
    if (n == 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        cache[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

template <int D, bool DEPOL, bool TABLE>
bool launch_d(const GateArgs& a, const GateTable* table, int warps, cudaStream_t s) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return false;
    const int sms = sm_count(dev);
    if (sms < 1) return false;
    int threads = kBlock<D>;
    if (D == 9 && (warps == 1 || warps == 2 || warps == 4)) threads = 32 * warps;
    size_t smem = 0;
    int64_t per_block = 64;                               // syndromes a block decodes at a time
    if constexpr (D > 7) {
        per_block = threads / LaneShape<D>::TS;
        smem = lane_smem<D, DEPOL>((int)per_block);
    }
    static std::atomic<int> occupancy[kMaxDevices][4];
    const int shape = threads == 32 ? 1 : (threads == 64 && D == 9 ? 2 : (threads == 128 && D == 9 ? 3 : 0));
    int per_sm = occupancy[dev][shape].load(std::memory_order_acquire);
    const void* kern = TABLE ? reinterpret_cast<const void*>(gate_table_kernel<(D <= 11 ? D : 11)>)
                             : reinterpret_cast<const void*>(gate_decode_kernel<D, DEPOL>);
    if (per_sm == 0) {
        if (smem > 0 &&
            (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  smem > 48 * 1024 ? (int)smem : 48 * 1024) != cudaSuccess ||
             cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                  cudaSharedmemCarveoutMaxShared) != cudaSuccess))
            return false;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess || per_sm < 1)
            return false;
        occupancy[dev][shape].store(per_sm, std::memory_order_release);
    }
    int64_t blocks = (int64_t)sms * per_sm;
    const int64_t need = (a.B + per_block - 1) / per_block;
    if (blocks > need) blocks = need;
    if (blocks < 1) return false;
    if constexpr (TABLE)
        gate_table_kernel<D><<<(unsigned)blocks, threads, smem, s>>>(a, *table);
    else
        gate_decode_kernel<D, DEPOL><<<(unsigned)blocks, threads, smem, s>>>(a);
    return cudaGetLastError() == cudaSuccess;
}

template <int D>
bool dispatch(const GateArgs& a, const GateTable* table, int warps, cudaStream_t s) {
    if (table) {
        if constexpr (D <= 11) return launch_d<D, false, true>(a, table, warps, s);
        return false;
    }
    return a.noise_mode == MLD_NOISE_DEPOL ? launch_d<D, true, false>(a, nullptr, warps, s)
                                           : launch_d<D, false, false>(a, nullptr, warps, s);
}

}  // namespace

bool gate_supported(int d) { return d >= 3 && d <= 13 && (d & 1); }

double gate_flops_per_syndrome(int d) {
    // three flops an entry and gate: columns 1..d-2 per l_Z in full; the first
    // column grows to the whole state and the last shrinks from it (once for
    // both l_X its first gate, then two states of a quarter and less): about
    // one full gate each way
    const double gate = 3.0 * (double)(1 << d);
    return 2.0 * gate * ((double)d * (d - 2) + 3.0);
}

// Where ties are decided at d <= 7: inside the kernel for single shots (a second
// launch takes 3 us more of some 23, and a tie among them 15 to 30 us either
// way), by the second launch above, where the rest of a warp's sixteen syndromes
// would wait for each tie (65,536 x 4 shots at d = 7, p = 0.02..0.18: 329 us
// inside, 266 by the pass; 64 at d = 5, p = 0.10: 52 and 33; start 35).
constexpr int64_t kTiesInside = 2;

bool launch_gate(int d, const GateArgs& args, const GateTable* table, int warps, cudaStream_t s) {
    GateArgs a = args;
    a.mark_ties = !table && (d == 9 || (d < 9 && a.B > kTiesInside));
    bool ok = false;
    switch (d) {
        case 3: ok = dispatch<3>(a, table, warps, s); break;
        case 5: ok = dispatch<5>(a, table, warps, s); break;
        case 7: ok = dispatch<7>(a, table, warps, s); break;
        case 9: ok = dispatch<9>(a, table, warps, s); break;
        case 11: ok = dispatch<11>(a, table, warps, s); break;
        case 13: ok = dispatch<13>(a, table, warps, s); break;
    }
    return ok && (!a.mark_ties || launch_decide_ties(d, exact_args(a), a.argmax, a.precision, s));
}

}  // namespace mld
