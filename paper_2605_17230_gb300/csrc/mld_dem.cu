// Code-capacity detector error models (Sec. 3.2.2): independent mechanisms,
// each one Pauli on one qubit. A qubit's mechanisms compose by Pauli product
// into its Pauli distribution (a contraction local to the qubit), and summing
// the network's detector parities out leaves the generator picture's column
// transfer with that table: the same Z_l(s), over a boundary of d bits where
// the open detectors' partial parities and both logical parities take d + 4.
// (Measured at d = 9, 65,536 syndromes: a dense sweep over the d + 4 parities
// 8.7 ms.)
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "mld_checks.h"
#include "mld_dem.h"
#include "mld_gate.h"
#include "mld_internal.h"

extern "C" mld_status mld_decode_dem(const mld_code* Cc, const int32_t* mech_qubit, const int32_t* mech_pauli,
                                     const double* mech_p, int32_t n_mech, const uint64_t* syndromes, int64_t B,
                                     double* logP, uint8_t* argmax, void* stream) {
    using namespace mld;
    NvtxRange trace("mld_decode_dem");
    mld_code* C = const_cast<mld_code*>(Cc);
    if (!C || n_mech < 0 || B < 0) return MLD_ERR_INVALID_ARG;
    if (n_mech > 0 && (!mech_qubit || !mech_pauli || !mech_p)) return MLD_ERR_INVALID_ARG;
    if (C->n > kGateMaxTableQubits) return MLD_ERR_UNSUPPORTED;
    const int d = C->d, n = C->n;
    // each qubit's Pauli distribution: independent mechanisms compose by Pauli product
    std::vector<double> dist((size_t)n * 4, 0.0);
    for (int q = 0; q < n; ++q) dist[(size_t)q * 4] = 1.0;
    for (int32_t m = 0; m < n_mech; ++m) {
        const int q = mech_qubit[m], e = mech_pauli[m];
        const double p = mech_p[m];
        if (q < 0 || q >= n || e < 1 || e > 3 || !(p >= 0.0 && p <= 1.0)) return MLD_ERR_INVALID_ARG;
        double* r = &dist[(size_t)q * 4];
        const double o[4] = {r[0], r[1], r[2], r[3]};
        for (int k = 0; k < 4; ++k) r[k] = (1.0 - p) * o[k] + p * o[k ^ e];
    }
    if (B == 0) return MLD_OK;
    if (!syndromes || !logP) return MLD_ERR_INVALID_ARG;
    mld_status st = ensure_code_device(C);
    if (st != MLD_OK) return st;
    GateTable table = {};
    for (int q = 0; q < n; ++q)
        for (int k = 0; k < 4; ++k)                  // Pauli code x + 2z -> I, X, Y, Z
            table.p[q][k] = (float)dist[(size_t)q * 4 + (k < 2 ? k : 5 - k)];
    GateArgs a;
    a.dmask = C->d_dmask;
    a.noise = nullptr;
    a.syn = syndromes;
    a.logP = logP;
    a.argmax = argmax;
    a.status = nullptr;                              // the mechanisms were checked above
    a.B = B;
    a.noise_mode = MLD_NOISE_TABLE;
    a.precision = MLD_FP32;
    return launch_gate(d, a, &table, 0, reinterpret_cast<cudaStream_t>(stream)) ? MLD_OK : MLD_ERR_CUDA;
}
