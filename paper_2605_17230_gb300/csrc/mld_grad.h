// Launchers of the adjoint of untruncated sweeps, d = 3..13.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mld {

struct GradDenseArgs {
    const uint64_t* dmask;     // [n][2][words]
    const float* noise;        // [n][4] (I, X, Y, Z)
    const uint64_t* syn;       // [B][words]
    const double* dlogP;       // [B][4] or nullptr
    double* logP;              // [B][4] or nullptr
    double* dnoise;            // [n][4], accumulated
    float* lws;                // workspace: blocks x grad_dense_workspace_floats (or grad_gate_...)
    int* status;               // status word (bits 1 << mld_status)
    int64_t B;
    int words;
};

// d = 13: resident blocks the launch uses on a device with `sms` SMs, and the floats
// of global workspace each needs (the left states of one unit and the
// block's partial gradient sums).
int64_t grad_dense_blocks(int d, int sms, int64_t B);
int64_t grad_dense_workspace_floats(int d);
bool launch_grad_dense(int d, const GradDenseArgs& a, int64_t blocks, cudaStream_t s);

// The same by the column transfer, d = 3..11 (it checks the noise itself).
int64_t grad_gate_blocks(int d, int64_t B);
int64_t grad_gate_workspace_floats(int d);
bool launch_grad_gate(int d, const GradDenseArgs& a, int64_t blocks, cudaStream_t s);

}  // namespace mld
