// Launcher of the rank-adaptive truncated sweep.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mld {

// Capacities of one unit's shapes and global slice (floats). The first pass
// over all units runs on every resident team with the smallest that hold
// chi (bond 48, 64 or 128: 2.25, 4.5 or 17.8 MB per unit); units that exceed
// them are decoded by a second pass with the large ones, a unit per SM.
struct TruncCaps {
    int max_bond;        // kept bond per cut
    int max_rows;        // carry rows
    int64_t mps;         // one boundary MPS, compact
    int64_t q;           // one column's reflectors and taus, compact
    int64_t spill;       // a site's work buffers when they do not fit on chip
    __host__ __device__ int64_t slice() const { return 2 * mps + q + spill; }
};
constexpr TruncCaps kTruncSmall{48, 192, 128 * 1024, 256 * 1024, 64 * 1024};
constexpr TruncCaps kTruncMid{64, 256, 256 * 1024, 512 * 1024, 128 * 1024};
constexpr TruncCaps kTruncLarge{128, 512, 1024 * 1024, 2048 * 1024, 384 * 1024};

// On-chip work arena of a unit (floats): 16, 8 or 4 units share an SM's sixteen
// warps, in teams of 1, 2 or 4. Batches that leave an SM at most 8 or 4 units
// get the larger ones: their time is the heaviest unit's, whose large steps
// then stay on chip and are shared by its team (d = 25, chi = 64, 515 syndromes:
// 114 ms with 8 units, 137 with 4; d = 17, p = 0.17, 128 syndromes: 100 ms with
// 4, 149 with 8 and 181 with 16 single warps; under load more units are faster:
// d = 17, 2,048 syndromes 91 ms with 16, 121 with 8).
constexpr int kTruncArenas[3] = {3072, 6500, 13500};
constexpr int trunc_arena(int64_t units, int sms) {
    return kTruncArenas[units <= 4 * (int64_t)sms ? 2 : (units <= 8 * (int64_t)sms ? 1 : 0)];
}

struct TruncArgs {
    const uint64_t* dmask;           // [n][2][words]
    const float* noise;              // [n][4] or [B]
    const uint64_t* syn;             // [B][words]
    double* logP;                    // [B][4]
    int* status;                     // status word (bits 1 << mld_status)
    int64_t B;
    int d, n, words, noise_mode;
    int chi;                         // cap on every new bond
    float cutoff;                    // keep sigma_k > cutoff * sigma_1 (relative)
    int arena;                       // on-chip work arena per unit (floats)
    TruncCaps caps;                  // shape and slice capacities of this pass
    float* ws;                       // per-unit global slices of caps.slice() floats
    unsigned long long* next_unit;   // work queue head (zeroed before the launch)
    const int64_t* order;            // the order to take the syndromes in (nullptr: as they come)
    const int64_t* in_list;          // units to decode (nullptr: all 2B units)
    const int* in_count;             // number of entries of in_list
    int64_t* ovf_list;               // units whose shapes exceed the capacities
    int* ovf_count;                  // (zeroed before the launch)
    double* flops;                   // executed flop counter (added to)
    unsigned long long* bond_hist;   // [65]: kept bonds k of every truncating cut (k >= 64 in the last bin)
};

// Units per block, dynamic shared memory per block for an arena of
// `arena` floats per unit, resident blocks per SM (0 on error), and the launch.
int trunc_units_per_block(int arena);
size_t trunc_smem_bytes(int arena);
int trunc_blocks_per_sm(int arena);
bool launch_trunc(const TruncArgs& a, int blocks, cudaStream_t s);

// order[B]: the syndromes by weight, heaviest first (B < 2^32).
bool launch_order(const uint64_t* syn, int64_t B, int words, int64_t* order, cudaStream_t s);

}  // namespace mld
