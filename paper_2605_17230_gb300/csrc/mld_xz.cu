// Independent X/Z (and bit-flip) noise, exact at every d (Sec. 3.1.3's
// problem): Pr(E) factors into x and z parts, so Z_(lX,lZ) = ZX_lX ZZ_lZ, and
// each part's coset sum is a planar random-bond Ising partition function.
// Swept column by column its boundary state is one bit per plaquette of the
// part's type, h = (d-1)/2 bits: 256 entries at d = 17, 4,096 at d = 25. Every
// term is a product of probabilities, so nothing cancels at any rate, where a
// Kac-Ward determinant (a signed sum) loses ln Z at low rates. For h <= 12 the
// transfer is also the smaller computation: 0.5 MFLOP a syndrome at d = 17 against 6.0 executed by a banded
// elimination of the 2|E| x 2|E| matrix, without its chain of pivots.
//
// The z part: Z-type plaquettes, at the odd row positions of a corner column.
// A qubit in an odd row replaces bit k by the next column's (flip
// probabilities f), a qubit in an even row weights the parity of the two bits
// beside it (g). One gate takes an even row and the odd row after it:
//     new[n] = sum_o f[o ^ n] g[prev ^ o] old[o],  prev = the bit before, new
// (rows rising in even columns, falling in odd ones), and the last even row of
// a column joins the first of the next. The x part is the z part of the patch
// turned by a quarter. Both ends are free: all-ones before the first column,
// a plain sum after the last. l_Z (l_X) is the string on row 0: it toggles
// that row's qubits, one unit per (part, sector).
//
// FP64 accuracy at FP32 rates: for h >= 7 an entry is a pair of FP32 numbers
// (19 FP32 operations for an output a x + b y, against two of the FP64 pipe at
// 1/64 of the rate). A qubit's two weights are stored as 1 and the odds, the
// larger probability going to one FP64 product a part: as p and 1 - p, a
// gate's most likely weight (1 - f)(1 - g) was rounded to 2^-48, under uniform
// rates the same way in every gate (largest error of ln Z over eight syndromes
// at p = 0.10, d = 25: 1.7e-12, with the odds 3.4e-13; complex FP64 elimination
// 1.1e-13 of the leading class and up to 1 of the others).
//
// Range: a pair has FP32's exponents. A unit watches its smallest entry at
// every rescaling; where one lies so low that the subnormals lost since the
// last may show, or where a rate is below 2^-33, the syndrome is marked and a
// second pass decodes it in FP64 (rescaled alike, entries 2^1880 apart). At
// d = 25 that is every syndrome from about p = 3e-3 down, at d = 17 from 1e-4.
//
// Bound: the FP32 pipe (62% busy at d = 25: two warps a scheduler, all the
// registers hold). Measured on GB300: d = 25, 700 syndromes 2.9 ms (all of
// them in the FP64 pass as well 17; banded elimination 125.8); d = 17, 1,024
// syndromes 0.20 ms (42; 2 us of it the second launch, which finds no mark);
// d = 9, 1,024 syndromes 0.10 ms (4.9).
// Registers hold RB bits of the state, lanes the rest, and a column exchanges them once
// through shared memory. A column's program is the same in both directions:
// at its start register bit t holds the row pair j = RB-1-t in processing
// order and lane bit u the pair H-1-u, at its end t holds j = LB+t and u holds
// j = u, which seen from the next column, whose order is reversed, is the
// start again.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <type_traits>
#include <vector>

#include "mld_gate.cuh"
#include "mld_internal.h"
#include "mld_xz.cuh"
#include "mld_xz.h"

namespace mld {
namespace {

using namespace gate;
using namespace xz;

// h <= 6: a thread holds the whole state in FP64, columns unrolled in pairs.
// Above: 64 entries of twice FP32 (128 registers); 64 lanes a unit at d = 25.
template <int H, bool WIDE = false>
struct Shape {
    static constexpr bool kPairs = H > 6 && !WIDE;
    using T = std::conditional_t<kPairs, Twin, double>;
    static constexpr int H_ = H;
    static constexpr int RB = H <= 6 ? H : 6;
    static constexpr int LB = H - RB;
    static constexpr int D = 2 * H + 1;
    static constexpr int N = D * D;
    static constexpr int LANES = 1 << LB;
    static constexpr int MID = RB - LB;                  // bits that stay in registers
    static constexpr int WORDS = (N - 1 + 63) / 64;
    static constexpr int NI = (N + 31) / 32 * 32;        // representative bits of a part, padded
    static constexpr int BW = NI / 32 + 1;
    static constexpr int NT = 4 * LANES > 128 ? 4 * LANES : 128;
    // exchange buffer of a unit, in vectors of VB bytes: [slot][row][column],
    // row stride LANES + 1; the units' regions are offset so that the lanes of
    // one access phase hit distinct banks
    static constexpr int VBYTES = (int)sizeof(T) << MID;
    static constexpr int VB = VBYTES >= 16 ? 16 : VBYTES;
    static constexpr int SLOTS = VBYTES / VB;
    static constexpr int STRIDE = LANES + 1;
    static constexpr int REGION0 = SLOTS * LANES * STRIDE;
    static constexpr int PHASE = 128 / VB;
    static constexpr int REGION =
        LB == 0 ? 0 : (LANES >= PHASE ? REGION0 : REGION0 + (LANES + PHASE - REGION0 % PHASE) % PHASE);
};

struct Args {
    const uint64_t* masks;     // [part][word][NI]: representative bits in processing order
    const uint64_t* xtype;     // [words]: X-type checks (bit-flip noise allows none of them)
    const float* px;
    const float* pz;           // nullptr: bit-flip noise
    const uint64_t* syn;
    double* logP;
    uint8_t* argmax;
    int* status;
    double* flops;
    int64_t B;
};

template <class S>
size_t shared_bytes(int units) {
    using T = typename S::T;
    constexpr int H = S::H_;
    size_t b = (size_t)2 * S::D * (H + 1) * 2 * sizeof(T) * 2;               // (p, 1 - p) per qubit of a gate
    b += (size_t)units * S::REGION * S::VB;
    b = (b + 15) & ~(size_t)15;
    b += (size_t)(units / 2) * 2 * S::BW * 4;                                // bits (at most units / 2 syndromes)
    b += (size_t)units * (sizeof(T) + 4) + units * 2 * sizeof(T) + 64;       // results, two warps' shares
    b += (S::NT / 32) * 2 * sizeof(double) + units * 4;                      // products of the larger probabilities, low
    return b;
}

// qubit of column c, processing step j of a part
template <int D>
__host__ __device__ __forceinline__ int qubit_of(int part, int c, int j) {
    const int r = (c & 1) ? D - 1 - j : j;
    return part == 0 ? (D - 1 - c) * D + r : r * D + c;
}

// A rate below this leaves products of three weights no room in a pair.
constexpr float kPairRate = 1.1641532182693481e-10f;    // 2^-33
__device__ __forceinline__ float small_rate(float p) { return p > 0.5f ? 1.f - p : p; }
// In logP[b][0]: a syndrome for the FP64 pass.
__device__ __forceinline__ bool is_marked(double l) { return l != l; }

// WIDE: the FP64 pass over the syndromes that the pairs marked.
template <int H, bool WIDE>
__global__ void __launch_bounds__(Shape<H>::NT) xz_kernel(Args a) {
    using S = Shape<H, WIDE>;
    using T = typename S::T;
    constexpr int D = S::D, RB = S::RB, LB = S::LB;
    using Scale = typename ScaleOf<T>::type;
    constexpr int R = 1 << RB;
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x;
    const int nu = a.pz ? 4 : 2;                          // units of a syndrome: (part, sector)
    const int per = nu * S::LANES;                        // threads of a syndrome
    const int sb = S::NT / per;                           // syndromes a block decodes at a time
    const int units = S::NT / S::LANES;
    if constexpr (WIDE) {                                 // nothing to do, as a rule
        bool any = false;
        for (int64_t c = blockIdx.x; c * sb < a.B; c += gridDim.x)
            any = any || (tid < sb && c * sb + tid < a.B && is_marked(a.logP[4 * (c * sb + tid)]));
        if (!__syncthreads_or(any)) return;
    }
    // [part][c][k]: f pair of the odd row, g pair of the even row before it;
    // k = H: the last even row's g
    T* tab = reinterpret_cast<T*>(smem);
    unsigned char* xch = smem + (size_t)2 * D * (H + 1) * 4 * sizeof(T);
    size_t off = (size_t)2 * D * (H + 1) * 4 * sizeof(T) + (size_t)units * S::REGION * S::VB;
    off = (off + 15) & ~(size_t)15;
    T* res_z = reinterpret_cast<T*>(smem + off);          // [unit]
    T* share = res_z + units;                             // [unit][2]
    int* res_e = reinterpret_cast<int*>(share + 2 * units);
    double* larger = reinterpret_cast<double*>(res_e + units);               // [warp][part] (units: a multiple of 4)
    int* low = reinterpret_cast<int*>(larger + S::NT / 32 * 2);              // [unit]: an entry left the range
    uint32_t* bits = reinterpret_cast<uint32_t*>(low + units);

    bool ok = true, rare = false;
    double prod[2] = {1.0, 1.0};
    for (int i = tid; i < nu / 2 * D * (H + 1); i += S::NT) {
        const int part = i / (D * (H + 1)), c = i / (H + 1) % D, k = i % (H + 1);
        const float* p = part ? a.pz : a.px;
        const float g = p[qubit_of<D>(part, c, 2 * k)];
        const float f = k < H ? p[qubit_of<D>(part, c, 2 * k + 1)] : 0.5f;
        ok = ok && g > 0.f && g < 1.f && f > 0.f && f < 1.f;                 // NaN fails
        double top = odds_of(tab + 4 * i + 2, g), f_top = odds_of(tab + 4 * i, f);
        rare = rare || !(small_rate(g) >= kPairRate) || !(small_rate(f) >= kPairRate);
        if (k < H) top *= f_top;
        if (part) prod[1] *= top;
        else prod[0] *= top;
    }
    if (!ok && blockIdx.x == 0) atomicOr(a.status, 1 << MLD_ERR_INVALID_ARG);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        prod[0] *= __shfl_xor_sync(0xffffffffu, prod[0], o);
        prod[1] *= __shfl_xor_sync(0xffffffffu, prod[1], o);
    }
    if ((tid & 31) == 0) {
        larger[tid >> 5 << 1] = prod[0];
        larger[(tid >> 5 << 1) + 1] = prod[1];
    }
    const int64_t nchunks = (a.B + sb - 1) / sb;
    if (__syncthreads_or(rare) && S::kPairs) {
        for (int64_t c = blockIdx.x; c < nchunks; c += gridDim.x)
            if (tid < sb && c * sb + tid < a.B) a.logP[4 * (c * sb + tid)] = NAN;
        return;
    }
    const int unit = tid / S::LANES, lane = tid % S::LANES;
    const int sub = unit / nu, part = unit % nu >> 1, sector = unit & 1;
    const T* ptab = tab + (size_t)part * D * (H + 1) * 4;
    int64_t done = 0;
    for (int64_t chunk = blockIdx.x; chunk < nchunks; chunk += gridDim.x) {
        const int64_t b0 = chunk * sb;
        const int live = (int)(a.B - b0 < sb ? a.B - b0 : sb);
        bool mine = true;                                 // this thread's syndrome is to be written
        if constexpr (WIDE) {
            mine = tid < live && is_marked(a.logP[4 * (b0 + tid)]);
            if (!__syncthreads_or(mine)) continue;
        }
        done += live;
        if (LB > 0 && lane == 0) low[unit] = 0;
        // representative bits: 32 at a time, a lane each, collected by a ballot
        {
            const int wl = tid & 31, nr = nu / 2 * (S::NI / 32);
            for (int i = tid >> 5; i < live * nr; i += S::NT / 32) {
                const int s = i / nr, rr = i % nr, pp = rr / (S::NI / 32), blk = rr % (S::NI / 32);
                const uint64_t* syn = a.syn + (b0 + s) * S::WORDS;
                const uint64_t* mk = a.masks + (size_t)pp * S::WORDS * S::NI + blk * 32 + wl;
                uint64_t x = 0;
#pragma unroll
                for (int w = 0; w < S::WORDS; ++w) x ^= syn[w] & mk[(size_t)w * S::NI];
                const uint32_t word = __ballot_sync(0xffffffffu, __popcll(x) & 1);
                if (wl == 0) bits[(s * 2 + pp) * S::BW + blk] = word;
            }
        }
        __syncthreads();
        const uint32_t* ubits = bits + ((sub < live ? sub : 0) * 2 + part) * S::BW;
        // bits of column c (bit j = processing step j), the string on row 0
        // toggled in
        const auto column_word = [&](int c) {
            const int i = c * D;
            const uint32_t w = __funnelshift_r(ubits[i >> 5], ubits[(i >> 5) + 1], i & 31);
            return w ^ ((uint32_t)sector << ((c & 1) ? D - 1 : 0));
        };
        T v[R];
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = Range<T>::start();
        int e2 = -Range<T>::top;
        T l0 = make<T>(1.0), l1 = l0;                         // last even row of the previous column
        Scale sc = 1;                                     // rescaling not yet applied
        // weights of gate k: g[prev ^ o] with prev toggled in where a lane holds it
        const auto gate_weights = [&](int c, int k, uint32_t word, uint32_t toggle) {
            const T* t = ptab + (c * (H + 1) + k) * 4;
            const uint32_t e = (word >> (2 * k)) ^ toggle;
            const T f0 = (e & 2) ? t[0] : t[1], f1 = (e & 2) ? t[1] : t[0];
            const T g0 = (e & 1) ? t[2] : t[3], g1 = (e & 1) ? t[3] : t[2];
            return Weights<T>{times(f0, g0), times(f1, g0), times(f0, g1), times(f1, g1)};
        };
        const auto first_weights = [&](int c, uint32_t word) {
            Weights<T> w = gate_weights(c, 0, word, 0);
            const T a0 = scaled(l0, sc), a1 = scaled(l1, sc);
            return Weights<T>{times(w.c00, a0), times(w.c10, a0), times(w.c01, a1), times(w.c11, a1)};
        };
        const auto last_row = [&](int c, uint32_t word) {
            const T* t = ptab + (c * (H + 1) + H) * 4 + 2;
            const bool e = word >> (2 * H) & 1;
            l0 = e ? t[0] : t[1];
            l1 = e ? t[1] : t[0];
        };
        if constexpr (LB == 0) {
            // bit t is row pair t; rising and falling columns alternate
#pragma unroll 1
            for (int c = 0; c < D; c += 2) {
                uint32_t word = column_word(c);
                gate_on<RB, 0, -1>(v, first_weights(c, word));
                const auto up = [&](int t) { return gate_weights(c, t, word, 0); };
                if constexpr (H > 1) gates_rising<RB, 1, RB>(v, up);
                last_row(c, word);
                sc = Range<T>::rescale(max_bits(v), e2);
                if (c + 1 < D) {
                    word = column_word(c + 1);
                    gate_on<RB, RB - 1, -1>(v, first_weights(c + 1, word));
                    const auto down = [&](int t) { return gate_weights(c + 1, RB - 1 - t, word, 0); };
                    if constexpr (H > 1) gates_falling<RB, RB - 2>(v, down);
                    last_row(c + 1, word);
                    sc = Range<T>::rescale(max_bits(v), e2);
                }
            }
        } else {
            // One gate body (1,300 instructions) for all row pairs: unrolled
            // over the twelve of d = 25 it is 230 KB of code and fetching it
            // takes as long again (8.3 ms against 4.2 for 1,024 syndromes).
            unsigned char* X = xch + (size_t)unit * S::REGION * S::VB;
#pragma unroll 1
            for (int c = 0; c < D; ++c) {
                const uint32_t word = column_word(c);
#pragma unroll 1
                for (int j = 0; j < H; ++j) {
                    bool no_prev = j == 0;
                    uint32_t toggle = 0;
                    if (j == RB) {
                        uint32_t mx = max_bits(v);
                        if (min_bits(v) < Range<T>::low) low[unit] = 1;
                        if constexpr (S::LANES >= 32) {
                            mx = __reduce_max_sync(0xffffffffu, mx);
                        } else {
#pragma unroll
                            for (int o = S::LANES / 2; o > 0; o >>= 1)
                                mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                        }
                        if constexpr (S::LANES > 32)
                            if ((tid & 31) == 0) reinterpret_cast<uint32_t*>(share + 2 * unit)[lane >> 5] = mx;
                        exchange_store<S>(X, v, lane);
                        unit_sync<S::LANES>(unit);
                        exchange_load<S>(X, v, lane);
                        if constexpr (S::LANES > 32) {
                            const uint32_t* m = reinterpret_cast<const uint32_t*>(share + 2 * unit);
                            mx = max(m[0], m[1]);
                        }
                        unit_sync<S::LANES>(unit);
                        sc = Range<T>::rescale(mx, e2);
                        if constexpr (S::MID == 0) {
                            no_prev = true;              // the pair before went to the lanes
                            toggle = (uint32_t)(lane >> (LB - 1)) & 1u;
                        }
                    }
                    Weights<T> w = j == 0 ? first_weights(c, word) : gate_weights(c, j, word, toggle);
                    if (j == RB) {
                        w = Weights<T>{scaled(w.c00, sc), scaled(w.c10, sc), scaled(w.c01, sc), scaled(w.c11, sc)};
                        sc = 1;
                    }
                    const T wa[2][2] = {{w.c00, w.c10}, {no_prev ? w.c00 : w.c01, no_prev ? w.c10 : w.c11}};
                    const T wb[2][2] = {{w.c11, w.c01}, {no_prev ? w.c11 : w.c10, no_prev ? w.c01 : w.c00}};
                    gate_and_rotate<RB>(v, wa, wb);
                }
                // register bit t is now row pair t of the next column
#pragma unroll
                for (int i = 0; i < R; ++i)
                    if (i < reversed<RB>(i)) {
                        const T x = v[i];
                        v[i] = v[reversed<RB>(i)];
                        v[reversed<RB>(i)] = x;
                    }
                last_row(c, word);
            }
        }
        // the last even row of the last column weights row pair H-1 = register bit RB-1
        T z;
        {
            if (LB > 0 && min_bits(v) < Range<T>::low) low[unit] = 1;
            T s0 = v[0], s1 = v[R / 2];
#pragma unroll
            for (int i = 1; i < R / 2; ++i) {
                s0 = plus(s0, v[i]);
                s1 = plus(s1, v[R / 2 + i]);
            }
            z = scaled(dot(l0, s0, l1, s1), sc);
#pragma unroll
            for (int o = 1; o < S::LANES && o < 32; o <<= 1) z = plus(z, shuffled(z, o));
            if constexpr (S::LANES > 32) {
                if ((tid & 31) == 0) share[2 * unit + (lane >> 5)] = z;
                unit_sync<S::LANES>(unit);
                z = plus(share[2 * unit], share[2 * unit + 1]);
            }
        }
        if (lane == 0) {
            res_z[unit] = z;
            res_e[unit] = e2;
        }
        __syncthreads();
        bool out = false;                                 // of the range
        if (LB > 0 && tid < live && mine)
            for (int s = 0; s < nu; ++s) out = out || low[tid * nu + s];
        if (out && S::kPairs) {
            a.logP[4 * (b0 + tid)] = NAN;
        } else if (tid < live && mine) {
            double larger_m[2] = {1.0, 1.0};              // m 2^e
            int larger_e[2] = {0, 0};
            for (int p = 0; p < nu / 2; ++p) {
                for (int w = 0; w < S::NT / 32; ++w) larger_m[p] *= larger[2 * w + p];
                larger_m[p] = mantissa(larger_m[p], larger_e[p]);
            }
            const int64_t b = b0 + tid;
            double lx[2], lz[2];
            bool bad = out;
            for (int s = 0; s < 2; ++s) {
                const double zx = value_of(res_z[tid * nu + s]);
                bad = bad || !(zx > 0.0) || !(zx < INFINITY);
                lx[s] = log_of(zx, larger_m[0], larger_e[0] + res_e[tid * nu + s]);
                if (nu == 4) {
                    const double zz = value_of(res_z[tid * nu + 2 + s]);
                    bad = bad || !(zz > 0.0) || !(zz < INFINITY);
                    lz[s] = log_of(zz, larger_m[1], larger_e[1] + res_e[tid * nu + 2 + s]);
                }
            }
            if (nu == 2) {
                // no z flips: only the identity's class, and only if no X-type check fired
                uint64_t any = 0;
                for (int w = 0; w < S::WORDS; ++w) any |= a.syn[b * S::WORDS + w] & a.xtype[w];
                lz[0] = any ? -INFINITY : 0.0;
                lz[1] = -INFINITY;
            }
            if (bad) atomicOr(a.status, 1 << MLD_ERR_NUMERIC);
            int best = 0;
            double l[4];
            for (int k = 0; k < 4; ++k) {
                l[k] = lx[k & 1] + lz[k >> 1];
                a.logP[4 * b + k] = l[k];
                if (l[k] > l[best]) best = k;
            }
            if (a.argmax) a.argmax[b] = (uint8_t)best;
        }
        __syncthreads();
    }
    // three flops an entry and gate, one an entry for the last row and sum
    if (tid == 0 && done > 0)
        atomicAdd(a.flops, (double)done * nu * (double)(1 << H) * (3.0 * D * H + 1.0));
}

constexpr int kMaxDevices = 64;

template <int H, bool WIDE>
mld_status launch_pass(const Args& a, cudaStream_t s) {
    using S = Shape<H, WIDE>;
    const auto kernel = xz_kernel<H, WIDE>;
    const int units = S::NT / S::LANES;
    const size_t smem = shared_bytes<S>(units);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return MLD_ERR_CUDA;
    static std::atomic<int> resident[kMaxDevices];         // blocks the device holds at once
    int n = resident[dev].load(std::memory_order_acquire);
    if (n == 0) {
        int sms = 0, per_sm = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)std::max(smem, (size_t)48 * 1024)) != cudaSuccess ||
            cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, S::NT, smem) != cudaSuccess)
            return MLD_ERR_CUDA;
        if (per_sm < 1) return MLD_ERR_UNSUPPORTED;
        n = sms * per_sm;
        resident[dev].store(n, std::memory_order_release);
    }
    const int sb = S::NT / ((a.pz ? 4 : 2) * S::LANES);
    int64_t blocks = (a.B + sb - 1) / sb;
    if (blocks > n) blocks = n;
    kernel<<<(unsigned)blocks, S::NT, smem, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? MLD_OK : MLD_ERR_CUDA;
}

template <int H>
mld_status launch_h(const Args& a, cudaStream_t s) {
    const mld_status st = launch_pass<H, false>(a, s);
    if constexpr (Shape<H>::kPairs) {
        if (st == MLD_OK) return launch_pass<H, true>(a, s);
    }
    return st;
}

mld_status launch(int d, const Args& a, cudaStream_t s) {
    switch ((d - 1) / 2) {
        case 1: return launch_h<1>(a, s);
        case 2: return launch_h<2>(a, s);
        case 3: return launch_h<3>(a, s);
        case 4: return launch_h<4>(a, s);
        case 5: return launch_h<5>(a, s);
        case 6: return launch_h<6>(a, s);
        case 7: return launch_h<7>(a, s);
        case 8: return launch_h<8>(a, s);
        case 9: return launch_h<9>(a, s);
        case 10: return launch_h<10>(a, s);
        case 11: return launch_h<11>(a, s);
        case 12: return launch_h<12>(a, s);
    }
    return MLD_ERR_UNSUPPORTED;
}

std::mutex g_xz_mutex;

// Device tables of a code, made on first use: the representative masks in
// processing order ([part][word][NI]), the X-type checks, and the counter of
// executed flops.
mld_status ensure_xz(mld_code* C) {
    std::lock_guard<std::mutex> lock(g_xz_mutex);
    if (C->d_xz) return MLD_OK;
    const int d = C->d, n = C->n, W = C->words, NI = (n + 31) / 32 * 32;
    std::vector<uint64_t> h((size_t)2 * W * NI + W + 1, 0);
    for (int part = 0; part < 2; ++part)
        for (int c = 0; c < d; ++c)
            for (int j = 0; j < d; ++j) {
                const int r = (c & 1) ? d - 1 - j : j;
                const int q = part == 0 ? (d - 1 - c) * d + r : r * d + c;
                for (int w = 0; w < W; ++w)
                    h[((size_t)part * W + w) * NI + c * d + j] = C->dmask[((size_t)q * 2 + part) * W + w];
            }
    for (int k = 0; k < C->m; ++k)
        if (C->stab_type[k] == 0) h[(size_t)2 * W * NI + k / 64] |= 1ULL << (k % 64);
    void* dev = nullptr;
    if (cudaMalloc(&dev, h.size() * 8) != cudaSuccess) return MLD_ERR_NOMEM;
    if (cudaMemcpy(dev, h.data(), h.size() * 8, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaFree(dev);
        return MLD_ERR_CUDA;
    }
    C->xz_masks = (size_t)2 * W * NI;
    C->d_xz = static_cast<uint64_t*>(dev);
    return MLD_OK;
}

}  // namespace

mld_status decode_xz_fp64(mld_code* C, const float* px, const float* pz, const uint64_t* syn, int64_t B, double* logP,
                          uint8_t* argmax, cudaStream_t s) {
    const mld_status st = ensure_xz(C);
    if (st != MLD_OK) return st;
    Args a;
    a.masks = C->d_xz;
    a.xtype = C->d_xz + C->xz_masks;
    a.px = px;
    a.pz = pz;
    a.syn = syn;
    a.logP = logP;
    a.argmax = argmax;
    a.status = C->d_status;
    a.flops = reinterpret_cast<double*>(C->d_xz + C->xz_masks + C->words);
    a.B = B;
    return launch(C->d, a, s);
}

mld_status xz_fp64_flops(mld_code* C, double* out) {
    *out = 0.0;
    if (!C->d_xz) return MLD_OK;
    uint64_t* cnt = C->d_xz + C->xz_masks + C->words;
    if (cudaMemcpy(out, cnt, sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess) return MLD_ERR_CUDA;
    if (cudaMemset(cnt, 0, sizeof(double)) != cudaSuccess) return MLD_ERR_CUDA;
    return MLD_OK;
}

}  // namespace mld

