// Rank-adaptive boundary-MPS sweep for truncating chi on sm_103a.
//
// Sec. 3.2.1: after each column's MPO is applied, the boundary MPS is brought
// to left-canonical form (QR, left to right) and compressed right to left by
// SVDs that keep the largest singular values, at most chi of them. Here the
// kept count at every cut is k = min(chi, #{sigma_j > cutoff * sigma_1}): the
// Schmidt spectra of these boundary states fall by seven orders of magnitude
// within the first ~20 values at p ~ 0.1 (kept bonds average 3..6 at d = 17
// and 25, p = 0.12), so a fixed bond of 32..128 would carry values below FP32
// resolution through every later product. Bonds are therefore runtime values
// per unit and every product, QR and Jacobi sweep runs on the actual shapes.
//
// Both factorisations are rank-revealing: Householder QR with column
// pivoting stops once every remaining column norm is at most cutoff times the
// largest one, so a QR of the left sweep keeps only the numerically
// significant rows of R (the carry, and with it the next site's row count,
// follows the numerical rank), and the SVD of a bond matrix T is taken from
// its pivoted triangle R by one-sided Jacobi on R^T (Drmac and Veselic's
// preconditioning: the rows of a pivoted R are nearly orthogonal, so few
// sweeps settle) over r' columns instead of all of T.
//
// One warp sweeps one (syndrome, l_Z) unit (both l_X classes: the X_L string
// sits on column d-1, columns 0..d-2 are swept once and the last column once
// per l_X from the state they leave); warps are persistent and take units
// from a device queue. The matrices are small (tens of rows), so a warp per
// unit keeps every step warp-synchronous and many units resident per SM. In
// batches that leave warps idle a unit has a team of two or four: the others
// take their share of the loops over more than 32 columns (MPO products,
// reflections, applications of Q), which are the heavy units' steps.
// Each site step lays its buffers out from its actual shapes in the warp's
// shared-memory arena: the incoming carry at one end, the outgoing carry at
// the other (ends alternate from step to step, so a carry is never moved),
// the work buffers in between. A step whose buffers do not fit keeps its
// carries and the site in the unit's global spill arena; the blocks that its
// factorisations work on (M; T; X and W) come on chip all the same, one after
// the other, where they fit. The MPS and the column's
// Householder reflectors are stored compactly in the unit's global slice
// (written once and read back once per column). A unit whose shapes exceed
// the slice's capacities goes to an overflow list that the fixed-shape kernel
// (same truncation rule) decodes afterwards.
//
// Every sum keeps one order whatever the layout, so the results have the same
// bits on chip and spilled, at any arena size: the cutoff (1e-7 by default)
// lies at FP32's rounding floor, where another order of summation would keep
// other components (a cutoff 10% off moves posteriors by 4e-5).
//
// Bound: instruction fetch under load (16 warps an SM at different places of
// a 78 KB program; 0.3 instructions a clock and SM), the latency of the
// heaviest unit's chain in small batches (a unit takes up to six times the
// mean, most of it in the few per cent of steps that spill). Hence loops are
// not unrolled beyond loading four rows ahead of their stores, copies run
// over flattened indices, arg-max and maximum are integer reductions, and
// small batches get larger arenas and teams. Measured on GB300: d = 17,
// chi = 32, 2,048 syndromes 78 ms (91 with the units in the caller's order, 178
// with loops unrolled by the compiler, spilled steps walking global columns),
// 8,192 syndromes 208 ms (237, 449); d = 25,
// chi = 64, 515 syndromes 114 ms (130 without teams; 321); d = 17, p = 0.17, 32
// syndromes 65 ms (89 without teams), one easy syndrome at d = 19 23.0 (24.1).
//
// Matrices on chip are column-major with odd leading dimensions (lanes walking
// one column each hit distinct banks), in the spill arena row-major (the lanes
// read whole lines).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "mld_internal.h"
#include "mld_trunc.h"

namespace mld {
namespace trunc {

constexpr int kWarpsPerBlock = 4;         // one, two or four units
constexpr int kMaxSweeps = 40;
constexpr float kTol = 1.0e-5f;           // pair orthogonality threshold (as the fixed-shape kernel)
constexpr float kNoise = 1.0e-8f;         // rotations moving less than this of the block are skipped
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}
// of values >= 0, whose bits order as unsigned integers
__device__ __forceinline__ float warp_max(float v) {
    return __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(v)));
}

// frexpf's exponent of x >= 0 (the library call only for zero and subnormals).
__device__ __forceinline__ int exponent_of(float x) {
    const int e = (int)(__float_as_uint(x) >> 23);
    if (e > 0 && e < 255) return e - 126;
    int ex = 0;
    frexpf(x, &ex);
    return ex;
}
// log2 of the lanes per column: the largest power of two G <= 32 with cols G <= 32.
__device__ __forceinline__ int group_shift(int cols) {
    return cols <= 1 ? 5 : (cols > 32 ? 0 : __clz(cols - 1) - 27);
}

__device__ __forceinline__ int imin(int a, int b) { return a < b ? a : b; }

// Exact quotient e / d for 0 <= e < 2^20 and 1 <= d <= 2^10 by one multiply:
// (e + 1/2) / d lies at least 1/(2d) from an integer, far beyond the float
// rounding of the product.
struct FDiv {
    int d;
    float inv;
    __device__ explicit FDiv(int d_) : d(d_), inv(1.f / (float)d_) {}
    __device__ int q(int e) const { return __float2int_rz(((float)e + 0.5f) * inv); }
};

// Odd leading dimension: the columns of a matrix walked by one lane each then
// fall into distinct shared-memory banks.
__device__ __forceinline__ int odd(int k) { return k | 1; }

// Rows of a column that are loaded ahead of the arithmetic and the stores on
// them: row by row each load would wait for the store before it (they might
// alias).
constexpr int kAhead = 4;

// A pointer into shared memory as a 32-bit index: loads and stores through it
// are shared-memory instructions with 32-bit addresses. A float* that may point
// to either memory costs 64-bit address arithmetic for every element, more
// instructions than the arithmetic itself.
struct Sh {
    int o;
    __device__ __forceinline__ float& operator[](int i) const {
        extern __shared__ __align__(16) unsigned char smem_raw[];
        return reinterpret_cast<float*>(smem_raw)[o + i];
    }
    __device__ __forceinline__ float& operator*() const { return (*this)[0]; }
    __device__ __forceinline__ Sh operator+(int i) const { return Sh{o + i}; }
    __device__ __forceinline__ Sh& operator+=(int i) { o += i; return *this; }
    __device__ __forceinline__ Sh& operator++() { ++o; return *this; }
};
__device__ __forceinline__ Sh shared_of(const float* p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    return Sh{(int)(p - reinterpret_cast<const float*>(smem_raw))};
}
// Row stride of a matrix on chip: 1.
template <class P>
constexpr bool kChip = std::is_same_v<P, Sh>;
// With one warp a unit and sixteen units an SM the second copy of each loop
// costs more (instruction fetch) than its addresses: one copy there.
template <int T>
using ChipPtr = std::conditional_t<(T > 1), Sh, float*>;

// A unit's team is T warps (T = 1, 2, 4). Warp 0 runs the sweep; the others wait
// at the team's barrier for a loop over columns or entries that is worth
// sharing, run their part of it and meet warp 0 there again. Each
// column or entry is computed by one lane or lane group as warp 0 alone would,
// so the bits do not depend on T.
enum JobKind { kQuit, kApply, kNorms, kUpdate, kApplyQ, kScale };
struct Job {
    int kind;
    int chip;                             // which matrices are on chip
    float part[4];                        // maxima of the warps' parts
    const float *C, *A, *wq, *V0, *tau0, *V1, *tau1;
    float *M, *nrm;
    int K, N, rs, cs, j, ncolA, Dl, Dr, ldC, pam, par, bp, i, rsplit, nr0, nr1, split, vrs, vcs;
    float f;
};

// The barrier of this thread's team (0 is the block's).
template <int T>
__device__ __forceinline__ void team_barrier() {
    __syncwarp();
    static_assert(kWarpsPerBlock == 4, "two teams of two warps or one of four");
    if (T == 4 || threadIdx.x < 64) asm volatile("barrier.sync 1, %0;" ::"n"(32 * T) : "memory");
    else asm volatile("barrier.sync 2, %0;" ::"n"(32 * T) : "memory");
}

// Elements lane, lane + 32, ... (step apart), four loads ahead of their stores.
__device__ __forceinline__ void copy_floats(float* dst, const float* src, int n, int first, int step) {
    int e = first;
#pragma unroll 1
    for (; e + 3 * step < n; e += 4 * step) {
        float x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = src[e + u * step];
#pragma unroll
        for (int u = 0; u < 4; ++u) dst[e + u * step] = x[u];
    }
#pragma unroll 1
    for (; e < n; e += step) dst[e] = src[e];
}

// Column norms and the identity permutation: columns of warp w of nw.
template <class P>
__device__ __forceinline__ void column_norms(P M, int K, int rs_, int cs, int N, float* nrm, int w, int nw) {
    const int rs = kChip<P> ? 1 : rs_;
#pragma unroll 1
    for (int c = 32 * w + (threadIdx.x & 31); c < N; c += 32 * nw) {
        const P col = M + c * cs;
        float s = 0.f;
        int r = 0;
#pragma unroll 1
        for (; r + kAhead <= K; r += kAhead) {
            float x[kAhead];
#pragma unroll
            for (int u = 0; u < kAhead; ++u) x[u] = col[(r + u) * rs];
#pragma unroll
            for (int u = 0; u < kAhead; ++u) s = fmaf(x[u], x[u], s);
        }
#pragma unroll 1
        for (; r < K; ++r) s = fmaf(col[r * rs], col[r * rs], s);
        nrm[c] = sqrtf(s);
    }
}

// H_j on columns j+1 .. N-1 and their norms below row j: a group of G
// lanes per column (G the largest power of two with (N-1-j) G <= 32),
// the rows dealt round-robin over the group, the dot product and the
// norm summed across it by shuffles. Columns of warp w of nw.
template <class P>
__device__ __forceinline__ void reflect_columns(P M, int K, int rs_, int cs, int N, float* nrm, int j, float tj,
                                                int w_, int nw) {
    const int lane = threadIdx.x & 31, rs = kChip<P> ? 1 : rs_;
    const P vj = M + j * cs;
    const int rem = N - 1 - j, sh = group_shift(rem), G = 1 << sh, gs = rs << sh;
    const int groups = 32 >> sh, grp = lane >> sh, g = lane & (G - 1);
#pragma unroll 1
    for (int base = j + 1 + w_ * groups; base < N; base += nw * groups) {
        const int cc = base + grp;
        const bool act = cc < N;
        const P col = M + (act ? cc : j) * cs;
        const int rows = (K - j - 1 - g + G - 1) >> sh;       // this lane's rows j+1+g, +G, ..
        const P v0 = vj + (j + 1 + g) * rs;
        const P x0p = col + (j + 1 + g) * rs;
        float w = 0.f;
        if (act && tj != 0.f) {
            if (g == 0) w = col[j * rs];
            P vp = v0, xp = x0p;
            int m = rows;
#pragma unroll 1
            for (; m >= kAhead; m -= kAhead) {
                float v[kAhead], x[kAhead];
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    v[u] = vp[u * gs];
                    x[u] = xp[u * gs];
                }
#pragma unroll
                for (int u = 0; u < kAhead; ++u) w = fmaf(v[u], x[u], w);
                vp += kAhead * gs;
                xp += kAhead * gs;
            }
#pragma unroll 1
            for (; m > 0; --m, vp += gs, xp += gs) w = fmaf(*vp, *xp, w);
        }
#pragma unroll 1
        for (int o = G >> 1; o > 0; o >>= 1) w += __shfl_xor_sync(kFull, w, o);
        float s = 0.f;
        if (act) {
            if (tj != 0.f) {
                w *= tj;
                if (g == 0) col[j * rs] -= w;
            }
            P vp = v0, xp = x0p;
            int m = rows;
#pragma unroll 1
            for (; m >= kAhead; m -= kAhead) {
                float v[kAhead], x[kAhead];
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    v[u] = vp[u * gs];
                    x[u] = xp[u * gs];
                }
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    if (tj != 0.f) x[u] = fmaf(-v[u], w, x[u]);
                    xp[u * gs] = x[u];
                    s = fmaf(x[u], x[u], s);
                }
                vp += kAhead * gs;
                xp += kAhead * gs;
            }
#pragma unroll 1
            for (; m > 0; --m, vp += gs, xp += gs) {
                const float x = tj != 0.f ? fmaf(-*vp, w, *xp) : *xp;
                *xp = x;
                s = fmaf(x, x, s);
            }
        }
#pragma unroll 1
        for (int o = G >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
        if (act && g == 0) nrm[cc] = sqrtf(s);
    }
}
template <int T, class P>
__device__ __noinline__ void reflect_columns_team(P M, int K, int rs, int cs, int N, float* nrm, int j, float tj,
                                                  int w, int nw) {
    reflect_columns(M, K, rs, cs, N, nrm, j, tj, w, nw);
}

// Householder QR with column pivoting, in place, of a K x N matrix (element
// (r, c) at r rs + c cs). Step j swaps the column of largest remaining
// norm into place, forms its reflector (R on and above the diagonal, the tail
// below it with v_j[j] = 1 implied, tau[j]) and applies it to the later
// columns; piv[j] is the original index of the column now at j. It stops once
// every remaining column norm is at most thr_rel times the largest initial
// one (or after min(K, N, maxr) steps) and returns the step count r. The
// reflector is formed across the warp's lanes; the later columns are updated
// one per lane (their row loops run serially, with no cross-lane reduction).
// The reflector norm is taken of the column scaled by a power of two near its
// maximum (a column far below the matrix's largest entries would lose its
// squares to underflow).
template <int T, class P>
__device__ __noinline__ int qrcp(float* Mg, int K, int rs_, int cs, int N, float* tau, int* piv, float* nrm,
                                 float thr_rel, int maxr, unsigned long long* fl, Job* job) {
    const int lane = threadIdx.x & 31, rs = kChip<P> ? 1 : rs_;
    P M;
    if constexpr (kChip<P>) M = shared_of(Mg);
    else M = Mg;
    const bool many = T > 1 && N > 32;
    if (many) {
        if (lane == 0) {
            job->kind = kNorms;
            job->chip = kChip<P>; job->M = Mg; job->K = K; job->rs = rs; job->cs = cs; job->N = N; job->nrm = nrm;
        }
        team_barrier<T>();
    }
    column_norms(M, K, rs, cs, N, nrm, 0, many ? T : 1);
#pragma unroll 1
    for (int c = lane; c < N; c += 32) piv[c] = c;
    if (many) team_barrier<T>();
    __syncwarp();
    float thr = 0.f;
#pragma unroll 1
    for (int c = lane; c < N; c += 32) thr = fmaxf(thr, nrm[c]);
    thr = thr_rel * warp_max(thr);
    const int steps = imin(imin(K, N), maxr);
    int r = 0;
    unsigned long long flops = 0;
#pragma unroll 1
    for (int j = 0; j < steps; ++j) {
        float best = -1.f;
        int p = j;
#pragma unroll 1
        for (int c = j + lane; c < N; c += 32) {
            const float v = nrm[c];
            if (v > best) { best = v; p = c; }
        }
        // largest norm, lowest index: the bits of floats >= 0 (and of -1) order as integers
        const int top = __reduce_max_sync(kFull, __float_as_int(best));
        p = __reduce_min_sync(kFull, __float_as_int(best) == top ? p : 0x7fffffff);
        best = __int_as_float(top);
        if (!(best > thr && best > 0.f)) break;
        r = j + 1;
        const P vj = M + j * cs;
        if (p != j) {
            const P cp = M + p * cs;
#pragma unroll 1
            for (int rr = lane; rr < K; rr += 32) {
                const float t = vj[rr * rs];
                vj[rr * rs] = cp[rr * rs];
                cp[rr * rs] = t;
            }
            if (lane == 0) {
                const float tn = nrm[j]; nrm[j] = nrm[p]; nrm[p] = tn;
                const int ti = piv[j]; piv[j] = piv[p]; piv[p] = ti;
            }
            __syncwarp();
        }
        float mx = 0.f;
#pragma unroll 1
        for (int rr = j + 1 + lane; rr < K; rr += 32) mx = fmaxf(mx, fabsf(vj[rr * rs]));
        mx = warp_max(mx);
        const float x0 = vj[j * rs];
        int ex = exponent_of(fmaxf(mx, fabsf(x0)));
        ex = ex < -125 ? -125 : (ex > 126 ? 126 : ex);
        const float sc = pow2f(-ex), isc = pow2f(ex);
        float ss = 0.f;
#pragma unroll 1
        for (int rr = j + 1 + lane; rr < K; rr += 32) { const float x = vj[rr * rs] * sc; ss = fmaf(x, x, ss); }
        ss = warp_sum(ss);
        float tj = 0.f, beta = x0, scal = 0.f;
        if (mx > 0.f) {
            const float x0s = x0 * sc;
            const float betas = -copysignf(sqrtf(fmaf(x0s, x0s, ss)), x0s);
            tj = (betas - x0s) / betas;
            scal = 1.f / (x0s - betas);
            beta = betas * isc;
        }
        __syncwarp();
        if (tj != 0.f) {
#pragma unroll 1
            for (int rr = j + 1 + lane; rr < K; rr += 32) vj[rr * rs] = (vj[rr * rs] * sc) * scal;
        }
        if (lane == 0) { vj[j * rs] = beta; tau[j] = tj; }
        __syncwarp();
        // H_j on the later columns and their norms
        const bool wide = T > 1 && N - 1 - j > 32;
        if (wide) {
            if (lane == 0) {
                job->kind = kUpdate;
                job->chip = kChip<P>; job->M = Mg; job->K = K; job->rs = rs; job->cs = cs; job->N = N; job->nrm = nrm;
                job->j = j; job->f = tj;
            }
            team_barrier<T>();
        }
        if (wide) {
            reflect_columns_team<T, P>(M, K, rs, cs, N, nrm, j, tj, 0, T);
            team_barrier<T>();
        } else {
            reflect_columns(M, K, rs, cs, N, nrm, j, tj, 0, 1);
        }
        __syncwarp();
        flops += 3ULL * (K - j) + 6ULL * (K - j) * (N - 1 - j);
    }
    if (lane == 0) *fl += flops;
    return r;
}

// Y <- Q Y for the columns of Y (element (r, c) at r yrs + c ycs), Q =
// H_0 ... H_{nr-1} with reflectors V (strides vrs, vcs,
// v_j below row j) and tau. Columns n < split use set 0 (V0, tau0, nr0), the
// others set 1. A group of G lanes per column (G the largest power of two
// with ncols G <= 32), the rows dealt round-robin over the group and each
// reflector's dot product summed across it by shuffles. Columns of warp w_ of
// nw.
template <class PV, class PY>
__device__ __noinline__ void apply_q(PV V0, const float* tau0, int nr0, PV V1,
                                     const float* tau1, int nr1, int split, int vrs_, int vcs, int K, PY Y,
                                     int yrs_, int ycs, int ncols, int w_, int nw) {
    const int lane = threadIdx.x & 31, vrs = kChip<PY> ? 1 : vrs_, yrs = kChip<PY> ? 1 : yrs_;
    const int sh = group_shift(ncols), G = 1 << sh, gv = vrs << sh, gy = yrs << sh;
    const int groups = 32 >> sh, grp = lane >> sh, g = lane & (G - 1);
    const int nrmax = nr0 > nr1 ? nr0 : nr1;
#pragma unroll 1
    for (int base = w_ * groups; base < ncols; base += nw * groups) {
        const int n = base + grp;
        const bool act = n < ncols;
        const bool s1 = n >= split;
        const PV Vs = s1 ? V1 : V0;
        const float* ts = s1 ? tau1 : tau0;
        const int nr = act ? (s1 ? nr1 : nr0) : 0;
        const PY y = Y + (act ? n : 0) * ycs;
        // every lane runs nrmax steps so that the group shuffles stay uniform;
        // lane g owns the rows r = g (mod G) in every step, so no lane reads
        // another's writes (v_j[j] = 1 is implied)
#pragma unroll 1
        for (int j = nrmax - 1; j >= 0; --j) {
            const bool on = j < nr && ts[j] != 0.f;
            const int r0 = j + ((g - j) & (G - 1));
            const PV v0 = Vs + j * vcs + r0 * vrs;
            const PY y0 = y + r0 * yrs;
            const int rows = (K - r0 + G - 1) >> sh;
            const bool diag = r0 == j;                    // the first of this lane's rows is row j
            float w = 0.f;
            if (on) {
                PV vp = v0;
                PY yp = y0;
                int m = rows;
                if (diag && m > 0) {
                    w = fmaf(1.f, *yp, w);
                    vp += gv;
                    yp += gy;
                    --m;
                }
#pragma unroll 1
                for (; m >= kAhead; m -= kAhead) {
                    float u[kAhead], x[kAhead];
#pragma unroll
                    for (int k = 0; k < kAhead; ++k) {
                        u[k] = vp[k * gv];
                        x[k] = yp[k * gy];
                    }
#pragma unroll
                    for (int k = 0; k < kAhead; ++k) w = fmaf(u[k], x[k], w);
                    vp += kAhead * gv;
                    yp += kAhead * gy;
                }
#pragma unroll 1
                for (; m > 0; --m, vp += gv, yp += gy) w = fmaf(*vp, *yp, w);
            }
#pragma unroll 1
            for (int o = G >> 1; o > 0; o >>= 1) w += __shfl_xor_sync(kFull, w, o);
            if (on) {
                w *= ts[j];
                PV vp = v0;
                PY yp = y0;
                int m = rows;
                if (diag && m > 0) {
                    *yp = fmaf(-1.f, w, *yp);
                    vp += gv;
                    yp += gy;
                    --m;
                }
#pragma unroll 1
                for (; m >= kAhead; m -= kAhead) {
                    float u[kAhead], x[kAhead];
#pragma unroll
                    for (int k = 0; k < kAhead; ++k) {
                        u[k] = vp[k * gv];
                        x[k] = yp[k * gy];
                    }
#pragma unroll
                    for (int k = 0; k < kAhead; ++k) yp[k * gy] = fmaf(-u[k], w, x[k]);
                    vp += kAhead * gv;
                    yp += kAhead * gy;
                }
#pragma unroll 1
                for (; m > 0; --m, vp += gv, yp += gy) *yp = fmaf(-*vp, w, *yp);
            }
        }
    }
    __syncwarp();
}

// apply_q where the matrices are: bit 0 of `chip`, Y on chip (and V's row
// stride 1); bit 1, V too.
template <int T>
__device__ __forceinline__ void apply_q_at(int chip, const float* V0, const float* tau0, int nr0, const float* V1,
                                           const float* tau1, int nr1, int split, int vrs, int vcs, int K, float* Y,
                                           int yrs, int ycs, int ncols, int w, int nw) {
    if (T > 1 && chip == 3)
        apply_q<Sh, Sh>(shared_of(V0), tau0, nr0, shared_of(V1), tau1, nr1, split, 1, vcs, K, shared_of(Y), 1, ycs,
                        ncols, w, nw);
    else if (T > 1 && chip == 1)
        apply_q<const float*, Sh>(V0, tau0, nr0, V1, tau1, nr1, split, 1, vcs, K, shared_of(Y), 1, ycs, ncols, w, nw);
    else
        apply_q<const float*, float*>(V0, tau0, nr0, V1, tau1, nr1, split, vrs, vcs, K, Y, yrs, ycs, ncols, w, nw);
}
template <int T>
__device__ __forceinline__ void apply_q_team(int chip, const float* V0, const float* tau0, int nr0, const float* V1,
                                             const float* tau1, int nr1, int split, int vrs, int vcs, int K, float* Y,
                                             int yrs, int ycs, int ncols, unsigned long long* fl, Job* job) {
    const int lane = threadIdx.x & 31;
    const bool wide = T > 1 && ncols > 32;
    if (wide) {
        if (lane == 0) {
            job->kind = kApplyQ;
            job->chip = chip;
            job->V0 = V0; job->tau0 = tau0; job->nr0 = nr0; job->V1 = V1; job->tau1 = tau1; job->nr1 = nr1;
            job->split = split; job->vrs = vrs; job->vcs = vcs; job->K = K; job->M = Y; job->rs = yrs;
            job->cs = ycs; job->N = ncols;
        }
        team_barrier<T>();
    }
    apply_q_at<T>(chip, V0, tau0, nr0, V1, tau1, nr1, split, vrs, vcs, K, Y, yrs, ycs, ncols, 0, wide ? T : 1);
    if (wide) team_barrier<T>();
    if (lane == 0) {
        // sum_j 4 (K - j) over nr reflectors, per column
        const unsigned long long f0 = 2ULL * nr0 * (2 * K - nr0 + 1), f1 = 2ULL * nr1 * (2 * K - nr1 + 1);
        const int c0 = split < ncols ? split : ncols;
        *fl += f0 * c0 + f1 * (ncols - c0);
    }
    __syncwarp();
}

// M^{b'}[kappa][col] = sum_a w(a, a', beta(kappa), b') sum_l C[kappa][a Dl + l] A[l][col]
// (qubit (i-1, c)), the entries of warp w_ of nw; returns this lane's largest
// modulus. Four columns of one row at a time: one load of C for four products,
// and four chains to overlap.
template <class P, class PC>
__device__ __forceinline__ float mpo_apply(const Job& a, PC C, PC A, P M, int w_, int nw) {
    const float* wq = a.wq;
    const int K = a.K, ncol = a.N, rsM = kChip<P> ? 1 : a.rs, csM = a.cs, ncolA = a.ncolA, Dl = a.Dl, Dr = a.Dr, ldC = a.ldC,
              pam = a.pam, par = a.par, bp = a.bp, i = a.i, rsplit = a.rsplit;
    const int quads = (ncol + 3) >> 2;
    const FDiv dK(K);
    float mx = 0.f;
#pragma unroll 1
    for (int e = 32 * w_ + (threadIdx.x & 31); e < K * quads; e += 32 * nw) {
        const int quad = dK.q(e), kap = e - quad * K, col = quad << 2;
        const int beta = (i == 0 || kap < rsplit) ? 0 : 1;
        const int c1 = imin(col + 1, ncol - 1) - col, c2 = imin(col + 2, ncol - 1) - col,
                  c3 = imin(col + 3, ncol - 1) - col;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int al = 0; al < pam; ++al) {
            PC crow = C + (al * Dl) * ldC + kap;
            PC arow = A + col;
            float x[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
            for (int l = 0; l < Dl; ++l, crow += ldC, arow += ncolA) {
                const float cv = *crow;
                x[0] = fmaf(cv, arow[0], x[0]);
                x[1] = fmaf(cv, arow[c1], x[1]);
                x[2] = fmaf(cv, arow[c2], x[2]);
                x[3] = fmaf(cv, arow[c3], x[3]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float w = 1.f;
                if (i > 0) {
                    const int ab = (col + u >= Dr ? 1 : 0) ^ beta, ub = al ^ bp;
                    w = par == 0 ? wq[ub + 2 * ab] : wq[ab + 2 * ub];
                }
                acc[u] = fmaf(w, x[u], acc[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (col + u < ncol) {
                M[(col + u) * csM + kap * rsM] = acc[u];
                mx = fmaxf(mx, fabsf(acc[u]));
            }
    }
    return mx;
}
template <int T>
__device__ __noinline__ float mpo_apply_team(const Job* a, int w, int nw) {
    return a->chip ? mpo_apply<Sh, Sh>(*a, shared_of(a->C), shared_of(a->A), shared_of(a->M), w, nw)
                   : mpo_apply<float*, const float*>(*a, a->C, a->A, a->M, w, nw);
}

__device__ __forceinline__ void scale_floats(float* M, int n, float f, int first, int step) {
    int e = first;
#pragma unroll 1
    for (; e + 3 * step < n; e += 4 * step) {
        float x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = M[e + u * step];
#pragma unroll
        for (int u = 0; u < 4; ++u) M[e + u * step] = x[u] * f;
    }
#pragma unroll 1
    for (; e < n; e += step) M[e] *= f;
}

// Warp w's side of a team until the team's unit queue is empty.
template <int T>
__device__ __forceinline__ void serve(Job& job, int w) {
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (;;) {
        team_barrier<T>();
        const int kind = job.kind;
        if (kind == kQuit) return;
        if (kind == kApply) {
            const float mx = warp_max(mpo_apply_team<T>(&job, w, T));
            if (lane == 0) job.part[w] = mx;
        } else if (kind == kNorms) {
            if (job.chip) column_norms(shared_of(job.M), job.K, 1, job.cs, job.N, job.nrm, w, T);
            else column_norms(job.M, job.K, job.rs, job.cs, job.N, job.nrm, w, T);
        } else if (kind == kUpdate) {
            if (job.chip)
                reflect_columns_team<T, Sh>(shared_of(job.M), job.K, 1, job.cs, job.N, job.nrm, job.j, job.f, w, T);
            else
                reflect_columns_team<T, float*>(job.M, job.K, job.rs, job.cs, job.N, job.nrm, job.j, job.f, w, T);
        } else if (kind == kApplyQ) {
            apply_q_at<T>(job.chip, job.V0, job.tau0, job.nr0, job.V1, job.tau1, job.nr1, job.split, job.vrs, job.vcs,
                          job.K, job.M, job.rs, job.cs, job.N, w, T);
        } else {
            scale_floats(job.M, job.N, job.f, 32 * w + lane, 32 * T);
        }
        team_barrier<T>();
    }
}

// Plane rotation of every G-th row (stride gs) of two columns.
template <class P>
__device__ __forceinline__ void rotate_columns(P xp, P xq, int rows, int gs, float cs, float sn) {
#pragma unroll 1
    for (; rows >= kAhead; rows -= kAhead) {
        float va[kAhead], vb[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            va[u] = xp[u * gs];
            vb[u] = xq[u * gs];
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const float a = va[u], b = vb[u];
            xp[u * gs] = cs * a - sn * b;
            xq[u * gs] = sn * a + cs * b;
        }
        xp += kAhead * gs;
        xq += kAhead * gs;
    }
#pragma unroll 1
    for (; rows > 0; --rows, xp += gs, xq += gs) {
        const float a = *xp, b = *xq;
        *xp = cs * a - sn * b;
        *xq = sn * a + cs * b;
    }
}

// One-sided Jacobi (Hestenes) on the n columns (length L, element (r, c) at
// r xrs + c xcs) of X, accumulating the rotations into W (n x n, strides wrs,
// wcs, starts at I). Parallel tournament order: each round rotates n/2
// disjoint pairs, one group of G lanes per pair (G a power of two). A pair is
// rotated when it is not orthogonal to kTol and the rotation moves more than
// kNoise of the block's Frobenius norm (below that it is FP32 rounding noise,
// which rotations regenerate). Rotation parameters: Rutishauser's formulas in
// FP32. Returns false when kMaxSweeps sweeps did not settle. (The entries of
// X lie in one block of L n floats, those of W in one of n n: both layouts
// are dense.)
template <class P>
__device__ __forceinline__ bool jacobi(P X, int L, int xrs_, int xcs, int n, P W, int wrs_, int wcs,
                                    unsigned long long* fl) {
    const int lane = threadIdx.x & 31, xrs = kChip<P> ? 1 : xrs_, wrs = kChip<P> ? 1 : wrs_;
    float f2 = 0.f;
    const FDiv dL(L);
#pragma unroll 1
    for (int e = lane; e < L * n; e += 32) {
        const int c = dL.q(e);
        const float x = X[(e - c * L) * xrs + c * xcs];
        f2 = fmaf(x, x, f2);
    }
    const float fro = sqrtf(warp_sum(f2));
#pragma unroll 1
    for (int e = lane; e < n * n; e += 32) W[e] = 0.f;
    __syncwarp();
#pragma unroll 1
    for (int e = lane; e < n; e += 32) W[e * (n + 1)] = 1.f;
    __syncwarp();
    const int nvp = n + (n & 1), npairs = nvp >> 1;
    const int sh = group_shift(npairs), G = 1 << sh;
    const int groups = 32 >> sh, grp = lane >> sh, g = lane & (G - 1);
    const int xgs = xrs << sh, wgs = wrs << sh, rows = (L - g + G - 1) >> sh, wrows = (n - g + G - 1) >> sh;
    int ev = 0, rt = 0;                        // pair evaluations and rotations by this group leader
    bool ok = n < 2;
#pragma unroll 1
    for (int sweep = 0; sweep < kMaxSweeps && !ok; ++sweep) {
        int rotated = 0;
#pragma unroll 1
        for (int round = 0; round < nvp - 1; ++round) {
#pragma unroll 1
            for (int base = 0; base < npairs; base += groups) {
                const int k = base + grp;
                int p = -1, q = -1;
                if (k < npairs) {
                    if (k == 0) { p = round; q = nvp - 1; }
                    else {
                        p = round + k;
                        if (p >= nvp - 1) p -= nvp - 1;
                        q = round - k;
                        if (q < 0) q += nvp - 1;
                    }
                    if (p >= n || q >= n) p = q = -1;
                }
                float al = 0.f, be = 0.f, ga = 0.f;
                if (p >= 0) {
                    P xp = X + p * xcs + g * xrs, xq = X + q * xcs + g * xrs;
                    int m = rows;
#pragma unroll 1
                    for (; m >= kAhead; m -= kAhead) {
                        float va[kAhead], vb[kAhead];
#pragma unroll
                        for (int u = 0; u < kAhead; ++u) {
                            va[u] = xp[u * xgs];
                            vb[u] = xq[u * xgs];
                        }
#pragma unroll
                        for (int u = 0; u < kAhead; ++u) {
                            al = fmaf(va[u], va[u], al); be = fmaf(vb[u], vb[u], be); ga = fmaf(va[u], vb[u], ga);
                        }
                        xp += kAhead * xgs;
                        xq += kAhead * xgs;
                    }
#pragma unroll 1
                    for (; m > 0; --m, xp += xgs, xq += xgs) {
                        const float a = *xp, b = *xq;
                        al = fmaf(a, a, al); be = fmaf(b, b, be); ga = fmaf(a, b, ga);
                    }
                }
#pragma unroll 1
                for (int o = G >> 1; o > 0; o >>= 1) {
                    al += __shfl_xor_sync(kFull, al, o);
                    be += __shfl_xor_sync(kFull, be, o);
                    ga += __shfl_xor_sync(kFull, ga, o);
                }
                if (p >= 0 && g == 0) ++ev;
                if (p >= 0 && ga != 0.f && fabsf(ga) > kTol * sqrtf(al) * sqrtf(be) &&
                    fabsf(ga) > kNoise * sqrtf(fmaxf(al, be)) * fro) {
                    const float zeta = (be - al) / (2.f * ga);
                    const float az = fabsf(zeta);
                    const float t = copysignf(1.f, zeta) / (az + (az < 1e18f ? sqrtf(fmaf(az, az, 1.f)) : az));
                    const float cs = 1.f / sqrtf(fmaf(t, t, 1.f)), sn = cs * t;
#pragma unroll 1
                    for (int h = 0; h < 2; ++h) {         // X, then W
                        const P blk = h ? W + g * wrs : X + g * xrs;
                        const int cst = h ? wcs : xcs;
                        rotate_columns(blk + p * cst, blk + q * cst, h ? wrows : rows, h ? wgs : xgs, cs, sn);
                    }
                    rotated = 1;
                    if (g == 0) ++rt;
                }
                __syncwarp();
            }
        }
        ok = !__any_sync(kFull, rotated);
    }
    // flops: 6L per evaluation, 6(L + n) per rotation, from the group leaders
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ev += __shfl_xor_sync(kFull, ev, o);
        rt += __shfl_xor_sync(kFull, rt, o);
    }
    if (lane == 0) *fl += 6ULL * L * ev + 6ULL * (L + n) * rt + 2ULL * L * n;
    __syncwarp();
    return ok;
}

template <class P>
__device__ __noinline__ bool jacobi_call(P X, int L, int xrs, int xcs, int n, P W, int wrs, int wcs,
                                         unsigned long long* fl) {
    return jacobi<P>(X, L, xrs, xcs, n, W, wrs, wcs, fl);
}

// Per-unit state in shared memory beside the arena.
struct Small {
    float wcol[kMaxD * 4];
    uint64_t syn[kMaxSynWords];
    int Dold[kMaxD + 2], Dnew[kMaxD + 2], Dkeep[kMaxD + 2];
    int Kr[kMaxD + 2], R0[kMaxD + 2], R1[kMaxD + 2];   // left sweep: rows, kept rank of each beta block
    int Qoff[2 * kMaxD + 4];             // reflector store offset of each site's beta blocks (this column)
    int Moff[2][kMaxD + 2];              // site offsets in the two MPS buffers
    unsigned long long fl;               // executed flops of the current unit (lane 0 adds)
};

// Placement of one site step's buffers in an arena of `cap` floats: the
// incoming carry stays at its end (bottom or top), the work buffers follow
// it, the outgoing carry goes to the other end.
struct Placement {
    float* base;
    int cap;
    const float* in;
    float* work;
    bool out_top;
    int outsz;
};

// ---------------------------------------------------------------- the unit
template <int T>
struct Unit {
    const TruncArgs& a;
    Small& S;
    Job* job;             // the team's (T > 1)
    float* arena;         // on-chip arena (a.arena floats)
    float* mps0;          // global MPS buffers (0 and 1)
    float* mps1;
    float* qst;           // global reflector store
    float* spill;         // global spill arena (a.caps.spill floats)
    int64_t b;            // syndrome
    int lz;               // class l_Z of this unit
    int e2;               // accumulated power-of-two exponent
    bool zero, bad, ovf, timeout;
    // where the carry is: arena, start, size, at the top of the arena or not
    float* cbase;
    float* cptr;
    int csize;
    int cld;              // leading dimension (rows) of the carry
    bool ctop;

    __device__ int present(int i, int j) const { return plaquette_is_check(a.d, i, j) ? 2 : 1; }

    // Lay out a step with the current carry, an outgoing carry of at most
    // `out` floats and `work` floats of buffers; the spill arena when the
    // on-chip one is too small (the carry is copied there first).
    __device__ int capof(const float* base) const { return base == arena ? a.arena : (int)a.caps.spill; }
    __device__ bool place(int out, int work, Placement& P) {
        const int lane = threadIdx.x & 31;
        // the carry's footprint: from its start to its end of the arena
        const int foot = ctop ? capof(cbase) - (int)(cptr - cbase) : csize;
        int need = foot + out + work;
        float* base = cbase;
        int cap = capof(cbase);
        if (need > cap || (cbase != arena && csize + out + work <= a.arena)) {
            need = csize + out + work;
            if (need <= a.arena) { base = arena; cap = a.arena; }
            else if (need <= a.caps.spill) {
                base = spill;
                cap = (int)a.caps.spill;
                if (lane == 0) atomicAdd(a.bond_hist, 1ULL);   // bin 0: steps run in the spill arena
            } else { ovf = true; return false; }
            if (base != cbase) {
                copy_floats(base, cptr, csize, lane, 32);
            } else {                           // same arena, carry moved to its bottom
                // (only when it sits at the top with room to spare below it)
#pragma unroll 1
                for (int e = lane; e < csize; e += 32) {
                    const float v = cptr[e];
                    __syncwarp();
                    base[e] = v;
                }
            }
            __syncwarp();
            cbase = base;
            cptr = base;
            ctop = false;
        }
        P.base = base;
        P.cap = cap;
        P.in = cptr;
        if (!ctop) {
            P.work = base + csize;
            P.out_top = true;
        } else {
            P.work = base + out;
            P.out_top = false;
        }
        P.outsz = out;
        return true;
    }
    // the outgoing carry: at the top of the reserved region or at the bottom
    __device__ float* out_ptr(const Placement& P) const { return P.out_top ? P.base + P.cap - P.outsz : P.base; }
    __device__ void carry_is(const Placement& P, float* ptr, int size, int ld) {
        cbase = P.base;
        cptr = ptr;
        csize = size;
        cld = ld;
        ctop = P.out_top;
    }

    // factor weights of column c's qubits: wcol[r][u + 2v] = p_q[E_q xor X^u Z^v]
    __device__ void column_weights(int c, int lx) {
        const int d = a.d, lane = threadIdx.x & 31;
#pragma unroll 1
        for (int r = lane; r < d; r += 32) {
            const int q = r * d + c;
            const uint64_t* mk = a.dmask + (size_t)q * 2 * a.words;
            int x = 0, z = 0;
#pragma unroll 1
            for (int w = 0; w < a.words; ++w) {
                x ^= __popcll(S.syn[w] & mk[w]) & 1;
                z ^= __popcll(S.syn[w] & mk[a.words + w]) & 1;
            }
            if (lz && r == 0) z ^= 1;                 // Z_L on row 0
            if (lx && c == d - 1) x ^= 1;             // X_L on column d-1
            float row[4];
            if (a.noise_mode == MLD_NOISE_TABLE) {
                const float4 v = *reinterpret_cast<const float4*>(a.noise + 4 * (size_t)q);
                row[0] = v.x; row[1] = v.y; row[2] = v.z; row[3] = v.w;
            } else {
                const float p = a.noise[b];
                row[0] = 1.f - p; row[1] = row[2] = row[3] = p * (1.f / 3.f);
            }
#pragma unroll 1
            for (int uv = 0; uv < 4; ++uv) {
                const int xx = x ^ (uv & 1), zz = z ^ (uv >> 1);
                S.wcol[4 * r + uv] = row[(!xx && !zz) ? 0 : (xx && !zz) ? 1 : (xx && zz) ? 2 : 3];
            }
        }
    }

    // Column c: MPO apply + pivoted QR sweep left to right, then the SVD sweep
    // right to left, MPS buffer sb -> db.
    __device__ void sweep_column(int c, int lx, int sb, int db) {
        const int d = a.d, lane = threadIdx.x & 31;
        const float* src = sb ? mps1 : mps0;
        float* dst = db ? mps1 : mps0;
        column_weights(c, lx);
        // the carry before site 0 is [1], at the bottom of the on-chip arena
        cbase = arena;
        cptr = arena;
        csize = 1;
        cld = 1;
        ctop = false;
        if (lane == 0) arena[0] = 1.f;
        __syncwarp();
        // ------------------------------------------------------ left sweep
        // The carry's rows are (beta_{i-1}, j): block 0's r0 rows, then block
        // 1's; rsplit = r0 of the previous site (beta = 0 below it).
        int K = 1, rsplit = 1, qo = 0;
#pragma unroll 1
        for (int i = 0; i <= d; ++i) {
            if (K > a.caps.max_rows) { ovf = true; return; }
            const int pam = i == 0 ? 1 : present(i - 1, c);
            const int pa = present(i, c), pb = present(i, c + 1);
            const int Dl = S.Dold[i], Dr = S.Dold[i + 1];
            const int ncolA = pa * Dr;
            const int ncol = i < d ? ncolA : 1;
            const int rmax = imin(K, ncol);
            const int ldM = odd(K);
            const int ldo = pb * rmax;            // rows reserved in the outgoing carry
            // work: A | M (one beta block at a time) | tau, nrm, piv, ipiv (ncol each)
            const int sA = Dl * ncolA, sM = ldM * ncol;
            Placement P;
            if (!place(ldo * ncol, sA + sM + 4 * ncol, P)) return;
            const float* C = P.in;
            const int ldC = cld;
            float* A = P.work;
            // a spilled step's carries and site stay in the spill arena; the
            // block that the QR works on comes on chip all the same if it fits
            const bool hot = P.base == arena || sM + 4 * ncol <= a.arena;
            float* M = P.base == arena || !hot ? A + sA : arena;
            float* tau = M + sM;
            float* nrm = tau + ncol;
            int* piv = reinterpret_cast<int*>(nrm + ncol);
            int* ipiv = piv + ncol;
            float* Co = out_ptr(P);
            // stage the old site (Dl x ncolA, row-major as stored)
            const float* Ag = src + S.Moff[sb][i];
            copy_floats(A, Ag, sA, lane, 32);
            __syncwarp();
            // on chip the rows of a column lie together (odd stride between
            // columns: lanes walking one column each hit distinct banks); in the
            // spill arena the columns of a row (lanes read whole lines)
            const int rsM = hot ? 1 : ncol, csM = hot ? ldM : 1;
            const int par = (i - 1 + c) & 1;
            const float* wq = S.wcol + 4 * (i - 1);
            const FDiv dK(K);
            int rb[2] = {0, 0};
            int E = 0;                            // common exponent of the site's blocks
            bool any = false;
#pragma unroll 1
            for (int bp = 0; bp < pb; ++bp) {
                // (at i = d alpha_d is summed into the single column)
                float mx = 0.f;
                const bool wide = T > 1 && K * ncol > 512;
                if (i < d) {
                    Job m;
                    m.kind = kApply;
                    m.chip = P.base == arena;
                    m.C = C; m.A = A; m.wq = wq; m.M = M; m.K = K; m.N = ncol; m.rs = rsM; m.cs = csM;
                    m.ncolA = ncolA; m.Dl = Dl; m.Dr = Dr; m.ldC = ldC; m.pam = pam; m.par = par; m.bp = bp;
                    m.i = i; m.rsplit = rsplit;
                    if (wide) {
                        if (lane == 0) *job = m;
                        team_barrier<T>();
                        mx = mpo_apply_team<T>(job, 0, T);
                        team_barrier<T>();
#pragma unroll
                        for (int w = 1; w < T; ++w) mx = fmaxf(mx, job->part[w]);
                    } else {
                        mx = mpo_apply<float*, const float*>(m, C, A, M, 0, 1);
                    }
                } else
#pragma unroll 1
                for (int kap = lane; kap < K; kap += 32) {
                    // the last site: its alpha is summed into the single column
                    const int beta = kap < rsplit ? 0 : 1;
                    float acc = 0.f;
#pragma unroll 1
                    for (int t = 0; t < pa * pam; ++t) {
                        const int ap = pam == 2 ? t >> 1 : t, al = pam == 2 ? t & 1 : 0;
                        const float* crow = C + (al * Dl) * ldC + kap;
                        float x = 0.f;
#pragma unroll 1
                        for (int l = 0; l < Dl; ++l) x = fmaf(crow[l * ldC], A[l * ncolA + ap], x);
                        const int ab = ap ^ beta, ub = al ^ bp;
                        acc = fmaf(par == 0 ? wq[ub + 2 * ab] : wq[ab + 2 * ub], x, acc);
                    }
                    M[kap * rsM] = acc;
                    mx = fmaxf(mx, fabsf(acc));
                }
                if (lane == 0) S.fl += 2ULL * K * ncolA * pam * (Dl + 1);
                mx = warp_max(mx);
                if (!(mx < INFINITY)) { bad = true; return; }
                if (mx == 0.f) continue;          // this block is zero: no rows
                // power-of-two scaling of the block (exact), exponent kept
                const int ex = exponent_of(mx);
                if (ex > 126 || ex < -125) { bad = true; return; }
                const float sc = pow2f(-ex);
                if (T > 1 && sM > 512) {
                    if (lane == 0) { job->kind = kScale; job->M = M; job->N = sM; job->f = sc; }
                    team_barrier<T>();
                    scale_floats(M, sM, sc, lane, 32 * T);
                    team_barrier<T>();
                } else {
                    __syncwarp();
                    scale_floats(M, sM, sc, lane, 32);
                }
                __syncwarp();
                // rank-revealing QR M^{b'} = Q [R; R22] P^T, R22 dropped
                const int r = hot ? qrcp<T, ChipPtr<T>>(M, K, rsM, csM, ncol, tau, piv, nrm, a.cutoff, rmax, &S.fl, job)
                                  : qrcp<T, float*>(M, K, rsM, csM, ncol, tau, piv, nrm, a.cutoff, rmax, &S.fl, job);
                rb[bp] = r;
                // reflectors (leading dimension K) and taus to the store
                const int qsz = K * r + r;
                if (qo + qsz > a.caps.q) { ovf = true; return; }
                float* Q = qst + qo;
#pragma unroll 1
                for (int e = lane; e < K * r; e += 32) {
                    const int j = dK.q(e);
                    Q[e] = M[j * csM + (e - j * K) * rsM];
                }
#pragma unroll 1
                for (int j = lane; j < r; j += 32) Q[K * r + j] = tau[j];
#pragma unroll 1
                for (int j = lane; j < ncol; j += 32) ipiv[piv[j]] = j;
                __syncwarp();
                // the block's carry rows: R[j][position of col] (upper trapezoid),
                // on the site's common power-of-two scale
                int rel = 0;
                if (!any) E = ex;
                else if (ex > E) {                // rescale the rows already written
#pragma unroll 1
                    for (int col = 0; col < ncol; ++col)
#pragma unroll 1
                        for (int row = lane; row < rb[0]; row += 32)
                            Co[col * ldo + row] = ldexpf(Co[col * ldo + row], E - ex);
                    E = ex;
                } else rel = ex - E;
                any = true;
                const int row0 = bp == 0 ? 0 : rb[0];
                if (r > 0) {
                    const FDiv dr(r);
                    const float fac = rel >= -126 ? pow2f(rel) : 0.f;
#pragma unroll 1
                    for (int e = lane; e < ncol * r; e += 32) {
                        const int col = dr.q(e), j = e - col * r, jp = ipiv[col];
                        float v = 0.f;
                        if (j <= jp) {
                            const float m = M[jp * csM + j * rsM];
                            v = rel >= -126 ? m * fac : ldexpf(m, rel);
                        }
                        Co[col * ldo + row0 + j] = v;
                    }
                }
                if (lane == 0) S.Qoff[2 * i + bp] = qo;
                qo += qsz;
                __syncwarp();
            }
            if (!any) { zero = true; return; }
            e2 += E;
            if (lane == 0) { S.Kr[i] = K; S.R0[i] = rb[0]; S.R1[i] = rb[1]; }
            __syncwarp();
            carry_is(P, Co, ldo * ncol, ldo);
            K = rb[0] + rb[1];
            rsplit = rb[0];
        }
        // ----------------------------------------------------- right sweep
        int Sr = 1, mo = 0;
#pragma unroll 1
        for (int i = d; i >= 0; --i) {
            const int pb = present(i, c + 1);
            const int Ki = S.Kr[i], r0 = S.R0[i], r1 = S.R1[i];
            const int N = pb * Sr;
            const int mn = imin(Ki, N);
            const int ldT = odd(Ki);
            const int kcap = imin(mn, a.chi);
            // work: T (Ki x N) | X (N x mn) | W (mn x mn) | tau, nrm, piv (N) | sig, perm (mn)
            const int sT = ldT * N, sX = N * mn, sW = mn * mn;
            Placement P;
            if (!place(i == 0 ? 0 : ldT * kcap, sT + sX + sW + 3 * N + 2 * mn, P)) return;
            const float* G = P.in;
            const int ldG = cld;                  // rows (b', j): r0 + r1 of them
            // spilled: T on chip if it fits, later X and W (their sizes follow the
            // rank), the vectors at the arena's end
            const bool chip = P.base == arena;
            const int small = 3 * N + 2 * mn;
            const int room = chip ? 0 : a.arena - small;
            const bool t_on = chip || sT <= room;
            bool t_in = t_on;                     // (its reflectors, later)
            float* Tm = chip || !t_on ? P.work : arena;
            float* X = P.work + sT;
            float* W = X + sX;
            float* tau = chip || room < 0 ? W + sW : arena + room;
            float* nrm = tau + N;
            int* piv = reinterpret_cast<int*>(nrm + N);
            float* sig = reinterpret_cast<float*>(piv + N);
            int* perm = reinterpret_cast<int*>(sig + mn);
            // T^{b'} = Q^{b'} [G^{b'}; 0]: block b' of G is rows [b' r0, b' r0 + r_b')
            const int rsT = t_on ? 1 : N, csT = t_on ? ldT : 1;       // layouts as in the left sweep
            const FDiv dKi(Ki);
#pragma unroll 1
            for (int e = lane; e < N * Ki; e += 32) {
                const int n = dKi.q(e), kap = e - n * Ki;
                const int bp = n >= Sr ? 1 : 0, s = n - bp * Sr;
                const int rr = bp ? r1 : r0, off = bp ? r0 : 0;
                Tm[n * csT + kap * rsT] = kap < rr ? G[s * ldG + off + kap] : 0.f;
            }
            __syncwarp();
            {
                const float* Q0 = qst + S.Qoff[2 * i];
                const float* Q1 = qst + S.Qoff[2 * i + 1];
                apply_q_team<T>(t_on ? 1 : 0, Q0, Q0 + Ki * r0, r0, Q1, Q1 + Ki * r1, r1, Sr, 1, Ki, Ki, Tm, rsT, csT, N, &S.fl, job);
                __syncwarp();
            }
            if (i == 0) {                         // Ki = 1: the orthogonality centre is the site
                if (mo + N > a.caps.mps) { ovf = true; return; }
                float* site = dst + mo;
#pragma unroll 1
                for (int e = lane; e < N; e += 32) site[e] = Tm[e * csT];
                if (lane == 0) { S.Dnew[0] = 1; S.Moff[db][0] = mo; }
                __syncwarp();
                break;
            }
            // T P = Q_T [R; R22], R22 dropped; Jacobi on X = R^T (N x r')
            const int rp = t_on ? qrcp<T, ChipPtr<T>>(Tm, Ki, rsT, csT, N, tau, piv, nrm, a.cutoff, mn, &S.fl, job)
                                : qrcp<T, float*>(Tm, Ki, rsT, csT, N, tau, piv, nrm, a.cutoff, mn, &S.fl, job);
            if (rp == 0) { zero = true; return; }
            const int need = (N + rp) * rp;
            bool x_on = chip;
            int used = 0;                         // of the arena, by a spilled step
            if (!chip && need <= room) {
                used = t_on && sT + need <= room ? sT : 0;
                if (t_on && used == 0) {          // T (from here on its reflectors) makes way
                    copy_floats(P.work, Tm, sT, lane, 32);
                    Tm = P.work;
                    t_in = false;
                    __syncwarp();
                }
                x_on = true;
                X = arena + used;
                W = X + N * rp;
                used += need;
            }
            const int rsX = x_on ? 1 : rp, csX = x_on ? N : 1, rsW = x_on ? 1 : rp, csW = x_on ? rp : 1;
            const FDiv dN(N);
#pragma unroll 1
            for (int e = lane; e < rp * N; e += 32) {
                const int j = dN.q(e), n = e - j * N;
                X[n * rsX + j * csX] = j <= n ? Tm[n * csT + j * rsT] : 0.f;
            }
            __syncwarp();
            bool settled;
            if constexpr (T > 1)
                settled = x_on ? jacobi_call<Sh>(shared_of(X), N, 1, csX, rp, shared_of(W), 1, csW, &S.fl)
                               : jacobi_call<float*>(X, N, rsX, csX, rp, W, rsW, csW, &S.fl);
            else
                settled = jacobi<float*>(X, N, rsX, csX, rp, W, rsW, csW, &S.fl);
            if (!settled) timeout = true;
            // R = W Sigma U'^T: right vectors of T = P U', left = Q_T [W; 0];
            // keep k = min(chi, #{sigma > cutoff sigma_max}) largest
            float smax = 0.f;
#pragma unroll 1
            for (int j = lane; j < rp; j += 32) {
                float s2 = 0.f;
#pragma unroll 1
                for (int rr = 0; rr < N; ++rr) s2 = fmaf(X[j * csX + rr * rsX], X[j * csX + rr * rsX], s2);
                sig[j] = sqrtf(s2);
                smax = fmaxf(smax, sig[j]);
            }
            smax = warp_max(smax);
            __syncwarp();
            int kept = 0;
#pragma unroll 1
            for (int j = lane; j < rp; j += 32) kept += (sig[j] > a.cutoff * smax && sig[j] > 0.f);
#pragma unroll 1
            for (int o = 16; o > 0; o >>= 1) kept += __shfl_xor_sync(kFull, kept, o);
            const int k = imin(kept, a.chi);
            if (k == 0) { zero = true; return; }
            if (k > a.caps.max_bond || mo + k * N > a.caps.mps) { ovf = true; return; }
#pragma unroll 1
            for (int j = lane; j < rp; j += 32) {
                const float sj = sig[j];
                int rank = 0;
#pragma unroll 1
                for (int m = 0; m < rp; ++m) rank += (sig[m] > sj) || (sig[m] == sj && m < j);
                if (rank < k) perm[rank] = j;
            }
            __syncwarp();
            float* site = dst + mo;
            // (the reciprocals take the place of the norms and taus in nrm: N >= k entries, free by now)
#pragma unroll 1
            for (int l = lane; l < k; l += 32) nrm[l] = 1.f / sig[perm[l]];
            __syncwarp();
#pragma unroll 1
            for (int e = lane; e < k * N; e += 32) {
                const int l = dN.q(e), n = e - l * N;
                site[l * N + piv[n]] = X[perm[l] * csX + n * rsX] * nrm[l];
            }
            // (a spilled step's new carry: formed on chip where there is room, then copied)
            float* Go = out_ptr(P);
            const bool stage = !chip && x_on && used + k * ldT <= room;
            float* Gn = stage ? arena + used : Go;
#pragma unroll 1
            for (int e = lane; e < k * Ki; e += 32) {
                const int l = dKi.q(e), kap = e - l * Ki;
                Gn[l * ldT + kap] = kap < rp ? W[perm[l] * csW + kap * rsW] * sig[perm[l]] : 0.f;
            }
            if (lane == 0) {
                S.Dnew[i] = k;
                S.Moff[db][i] = mo;
                atomicAdd(a.bond_hist + (k < 64 ? k : 64), 1ULL);
            }
            __syncwarp();
            apply_q_team<T>((chip || stage) ? (t_in ? 3 : rsT == 1 ? 1 : 0) : 0, Tm, tau, rp, Tm, tau, rp, k, rsT, csT, Ki,
                            Gn, 1, ldT, k, &S.fl, job);
            __syncwarp();
            if (stage) {
                copy_floats(Go, Gn, k * ldT, lane, 32);
                __syncwarp();
            }
            carry_is(P, Go, ldT * kcap, ldT);
            mo += k * N;
            Sr = k;
        }
#pragma unroll 1
        for (int i = lane; i <= d; i += 32) S.Dold[i] = S.Dnew[i];
        if (lane == 0) S.Dold[d + 1] = 1;
        __syncwarp();
    }

    // Contraction of the MPS (buffer db) with all-ones vectors -> ln Z (FP64)
    __device__ double contract(int db) {
        const int d = a.d, lane = threadIdx.x & 31;
        float* v = arena;                 // bonds of at most 128 (the large capacities)
        float* vn = arena + 128;
        if (lane == 0) v[0] = 1.f;
        __syncwarp();
#pragma unroll 1
        for (int i = 0; i <= d; ++i) {
            const int Dl = S.Dold[i], Dr = S.Dold[i + 1];
            const int p = present(i, d);                            // corner column d
            const float* site = (db ? mps1 : mps0) + S.Moff[db][i];
#pragma unroll 1
            for (int s = lane; s < Dr; s += 32) {
                float acc = 0.f;
#pragma unroll 1
                for (int l = 0; l < Dl; ++l)
#pragma unroll 1
                    for (int bb = 0; bb < p; ++bb) acc = fmaf(v[l], site[l * p * Dr + bb * Dr + s], acc);
                vn[s] = acc;
            }
            __syncwarp();
            float* t = v; v = vn; vn = t;
        }
        const float z = v[0];
        __syncwarp();
        if (!(z == z)) bad = true;
        return z > 0.f ? log((double)z) + (double)e2 * 0.69314718055994530942 : -INFINITY;
    }

    __device__ void run(int64_t unit) {
        const int d = a.d, lane = threadIdx.x & 31;
        b = unit >> 1;
        lz = (int)(unit & 1);
        e2 = 0;
        zero = bad = ovf = timeout = false;
#pragma unroll 1
        for (int w = lane; w < a.words; w += 32) S.syn[w] = a.syn[b * a.words + w];
        // all-ones product state over corner column 0 (site i: 1 x p x 1 at 2i)
#pragma unroll 1
        for (int i = lane; i <= d; i += 32) {
            mps0[2 * i] = 1.f;
            mps0[2 * i + 1] = 1.f;
            S.Dold[i] = 1;
            S.Moff[0][i] = 2 * i;
        }
        if (lane == 0) { S.Dold[d + 1] = 1; S.fl = 0ULL; }
        __syncwarp();
        // passes: columns 0..d-2 (l_X = 0), then column d-1 once per l_X from
        // the state after column d-2 (kept in buffer sb, its bonds in Dkeep)
        double out[2] = {-INFINITY, -INFINITY};
        int sb = 0, e2p = 0;
#pragma unroll 1
        for (int pass = 0; pass < d + 1; ++pass) {
            const int c = pass < d - 1 ? pass : d - 1;
            const int lx = pass == d ? 1 : 0;
            if (pass == d - 1) {                  // keep the state for the second last-column pass
                e2p = e2;
#pragma unroll 1
                for (int i = lane; i <= d + 1; i += 32) S.Dkeep[i] = S.Dold[i];
                __syncwarp();
            } else if (pass == d) {
                e2 = e2p;
                zero = false;
#pragma unroll 1
                for (int i = lane; i <= d + 1; i += 32) S.Dold[i] = S.Dkeep[i];
                __syncwarp();
            }
            sweep_column(c, lx, sb, sb ^ 1);
            __syncwarp();
            if (bad || ovf) break;
            if (pass < d - 1) {
                if (zero) break;                  // every class of this unit vanishes
                sb ^= 1;
            } else if (!zero) {
                out[pass - (d - 1)] = contract(sb ^ 1);
            }
        }
        if (lane == 0) {
            if (ovf) {
                if (a.ovf_list) {
                    const int slot = atomicAdd(a.ovf_count, 1);
                    a.ovf_list[slot] = (int64_t)unit;
                } else {
                    atomicOr(a.status, 1 << MLD_ERR_UNSUPPORTED);
                }
            } else {
                a.logP[b * 4 + 2 * lz] = out[0];
                a.logP[b * 4 + 2 * lz + 1] = out[1];
            }
            if (bad) atomicOr(a.status, 1 << MLD_ERR_NUMERIC);
            if (timeout) atomicOr(a.status, 1 << MLD_ERR_TIMEOUT);
            atomicAdd(a.flops, (double)S.fl);
        }
        __syncwarp();
    }
};

// Shared memory of one unit: Small, then the team's job (T > 1), then the
// arena (16-byte aligned).
template <int T>
__host__ __device__ constexpr size_t small_bytes() {
    return ((sizeof(Small) + 15) & ~size_t(15)) + (T > 1 ? (sizeof(Job) + 15) & ~size_t(15) : 0);
}
template <int T>
__host__ __device__ constexpr size_t unit_bytes(int arena) {
    return small_bytes<T>() + (((size_t)arena * sizeof(float) + 15) & ~size_t(15));
}

template <int T>
__global__ void __launch_bounds__(32 * kWarpsPerBlock, 4) trunc_kernel(TruncArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, team = warp / T;
    unsigned char* mine = smem_raw + (size_t)team * unit_bytes<T>(a.arena);
    Small& S = *reinterpret_cast<Small*>(mine);
    Job* job = T > 1 ? reinterpret_cast<Job*>(mine + ((sizeof(Small) + 15) & ~size_t(15))) : nullptr;
    if constexpr (T > 1) {
        if (warp % T) {
            serve<T>(*job, warp % T);
            return;
        }
    }
    float* arena = reinterpret_cast<float*>(mine + small_bytes<T>());
    const int64_t slot = (int64_t)blockIdx.x * (kWarpsPerBlock / T) + team;
    float* base = a.ws + slot * a.caps.slice();
    const unsigned long long units = a.in_list ? (unsigned long long)*a.in_count : 2ULL * (unsigned long long)a.B;
#pragma unroll 1
    for (;;) {
        unsigned long long idx = 0;
        if (lane == 0) idx = atomicAdd(a.next_unit, 1ULL);
        idx = __shfl_sync(kFull, idx, 0);
        if (idx >= units) break;
        Unit<T> u{a, S, job, arena, base, base + a.caps.mps, base + 2 * a.caps.mps,
                  base + 2 * a.caps.mps + a.caps.q};
        u.run(a.in_list ? a.in_list[idx]
                        : a.order ? 2 * a.order[idx >> 1] + (int64_t)(idx & 1) : (int64_t)idx);
    }
    if constexpr (T > 1) {
        if (lane == 0) job->kind = kQuit;
        team_barrier<T>();
    }
}

// Syndromes by weight, heaviest first. A unit's time follows the ranks of its
// boundary states, which follow the syndrome's weight; a queue that hands out
// the long units first has no long one left to start when the others are done.
// One block: a pass to count the weights, one to place the syndromes.
constexpr int kOrderThreads = 1024, kOrderBins = kMaxD * kMaxD;
__device__ __forceinline__ int syndrome_weight(const uint64_t* s, int words) {
    int w = 0;
    for (int i = 0; i < words; ++i) w += __popcll(s[i]);
    return w < kOrderBins ? w : kOrderBins - 1;     // (bits past the last check are the caller's)
}
__global__ void __launch_bounds__(kOrderThreads) order_kernel(const uint64_t* syn, int64_t B, int words,
                                                              int64_t* order) {
    __shared__ unsigned bin[kOrderBins];
    for (int i = threadIdx.x; i < kOrderBins; i += kOrderThreads) bin[i] = 0;
    __syncthreads();
    for (int64_t b = threadIdx.x; b < B; b += kOrderThreads) atomicAdd(&bin[syndrome_weight(syn + b * words, words)], 1u);
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned at = 0;
        for (int i = kOrderBins - 1; i >= 0; --i) {
            const unsigned n = bin[i];
            bin[i] = at;
            at += n;
        }
    }
    __syncthreads();
    for (int64_t b = threadIdx.x; b < B; b += kOrderThreads)
        order[atomicAdd(&bin[syndrome_weight(syn + b * words, words)], 1u)] = b;
}

// Warps of a unit's team: the SM's sixteen, shared by the units its arenas
// leave room for.
constexpr int team_of(int arena) { return arena >= kTruncArenas[2] ? 4 : (arena >= kTruncArenas[1] ? 2 : 1); }

template <int T>
bool allow() {
    // (the largest arena of the team size, so that threads launching with
    // different arenas do not undo each other's)
    return cudaFuncSetAttribute(trunc_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(kWarpsPerBlock / T * unit_bytes<T>(kTruncArenas[T / 2]))) == cudaSuccess;
}
template <int T>
int resident(size_t bytes) {
    int n = 0;
    if (!allow<T>() || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, trunc_kernel<T>, 32 * kWarpsPerBlock,
                                                                     bytes) != cudaSuccess)
        return 0;
    return n;
}

}  // namespace trunc

int trunc_units_per_block(int arena) { return trunc::kWarpsPerBlock / trunc::team_of(arena); }

size_t trunc_smem_bytes(int arena) {
    switch (trunc::team_of(arena)) {
        case 4: return trunc::unit_bytes<4>(arena);
        case 2: return 2 * trunc::unit_bytes<2>(arena);
    }
    return 4 * trunc::unit_bytes<1>(arena);
}

int trunc_blocks_per_sm(int arena) {
    const size_t bytes = trunc_smem_bytes(arena);
    switch (trunc::team_of(arena)) {
        case 4: return trunc::resident<4>(bytes);
        case 2: return trunc::resident<2>(bytes);
    }
    return trunc::resident<1>(bytes);
}

bool launch_order(const uint64_t* syn, int64_t B, int words, int64_t* order, cudaStream_t s) {
    trunc::order_kernel<<<1, trunc::kOrderThreads, 0, s>>>(syn, B, words, order);
    return cudaGetLastError() == cudaSuccess;
}

bool launch_trunc(const TruncArgs& a, int blocks, cudaStream_t s) {
    const size_t bytes = trunc_smem_bytes(a.arena);
    const int threads = 32 * trunc::kWarpsPerBlock;
    switch (trunc::team_of(a.arena)) {
        case 4:
            if (!trunc::allow<4>()) return false;
            trunc::trunc_kernel<4><<<blocks, threads, bytes, s>>>(a);
            break;
        case 2:
            if (!trunc::allow<2>()) return false;
            trunc::trunc_kernel<2><<<blocks, threads, bytes, s>>>(a);
            break;
        default:
            if (!trunc::allow<1>()) return false;
            trunc::trunc_kernel<1><<<blocks, threads, bytes, s>>>(a);
    }
    return cudaGetLastError() == cudaSuccess;
}

}  // namespace mld
