// Launcher of the untruncated column transfer (d = 3..13).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mld {

struct GateArgs {
    const uint64_t* dmask;     // [n][2][words]
    const float* noise;        // [n][4] (I, X, Y, Z) or [B] depolarizing p
    const uint64_t* syn;       // [B][words]
    double* logP;              // [B][4]
    uint8_t* argmax;           // [B] or nullptr
    int* status;               // status word (bits 1 << mld_status), or nullptr
    int64_t B;
    int noise_mode;
    int precision;             // of the sweep that decides ties
    bool mark_ties;            // for a second launch; set by launch_gate
};

constexpr int kGateMaxTableQubits = 121;

// A noise table passed by value (the detector picture composes its
// mechanisms on the host: nothing is allocated or copied).
struct GateTable {
    float p[kGateMaxTableQubits][4];
};

// Distances with a kernel, its counted flops per syndrome (four classes), and
// the launch: ln Z, the decision and the noise check in one kernel,
// asynchronous on s; with a noise table or rates in memory, ties at d <= 9 are
// decided by the boundary-MPS sweep (a second launch, but for single shots at
// d <= 7). warps: warps per block at d = 9 (0: default). table: the noise table
// by value in place of a.noise (d <= 11), else nullptr.
bool gate_supported(int d);
double gate_flops_per_syndrome(int d);
bool launch_gate(int d, const GateArgs& a, const GateTable* table, int warps, cudaStream_t s);

}  // namespace mld
