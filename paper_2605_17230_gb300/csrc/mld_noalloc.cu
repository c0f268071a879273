// Decoding entry point that allocates no device memory.
//
// Some callers cannot allocate device memory: a real-time decoding loop that
// must not stall on the implicit device-wide synchronisation of cudaMalloc,
// or a process whose device memory is already fully reserved by another
// framework's caching allocator. mld_decode allocates its code tables and
// status word on first use; this variant instead keeps that scratch in one
// file-scope __device__ array of fixed size, which every GPU that loads the
// library holds until the process exits. The caller still passes inputs and
// outputs in its own device memory.
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <vector>

#include "mld_checks.h"
#include "mld_gate.h"
#include "mld_internal.h"

namespace {

// Scratch layout: [0, 256) status word, [256, ...) per-qubit destabiliser
// masks of the code, n * 2 * syn_words uint64 (enough for d <= 11).
constexpr size_t kNoAllocBytes = 16384;
constexpr size_t kStatusSlot = 256;
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

std::mutex g_setup_mutex;
void* g_scratch_ptr[kMaxDevices] = {};
// FNV-1a hash of the destabiliser tables last written to each device's
// scratch array (0: none yet), so that consecutive calls for one code skip
// the upload; calls are serialised by the caller, as the array is shared
uint64_t g_tables_written[kMaxDevices] = {};

uint64_t table_hash(const std::vector<uint64_t>& t) {
    uint64_t h = 1469598103934665603ULL;
    for (uint64_t w : t)
        for (int k = 0; k < 8; ++k) {
            h ^= (w >> (8 * k)) & 0xffu;
            h *= 1099511628211ULL;
        }
    return h | 1ULL;                 // never 0
}

// Device address of the scratch array for the current device. In host code
// the array's name is only a host-side stand-in, so the address is looked up
// once per device (with that device current) and cached.
mld_status scratch_address(unsigned char** out, int* device) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return MLD_ERR_CUDA;
    *device = dev;
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return MLD_ERR_CUDA;
        g_scratch_ptr[dev] = p;
    }
    *out = static_cast<unsigned char*>(g_scratch_ptr[dev]);
    return MLD_OK;
}

}  // namespace

extern "C" mld_status mld_decode_noalloc(const mld_code* C, const float* noise, int noise_mode,
                                         const uint64_t* syndromes, int64_t B, int chi, int precision,
                                         double* logP, uint8_t* argmax, void* stream, int check_status) {
    mld::NvtxRange trace("mld_decode_noalloc");
    if (!C || B < 0 || chi < 1) return MLD_ERR_INVALID_ARG;
    if (noise_mode != MLD_NOISE_TABLE && noise_mode != MLD_NOISE_DEPOL) return MLD_ERR_INVALID_ARG;
    if (precision != MLD_FP32 && precision != MLD_MIXED_BF16 && precision != MLD_MIXED_TF32)
        return MLD_ERR_INVALID_ARG;
    if (B == 0) return MLD_OK;
    if (!noise || !syndromes || !logP) return MLD_ERR_INVALID_ARG;
    if (noise_mode == MLD_NOISE_TABLE && (reinterpret_cast<uintptr_t>(noise) & 15)) return MLD_ERR_INVALID_ARG;
    // only the untruncated FP32 sweep of the distances with a specialised
    // kernel, and only codes whose tables fit in the scratch array
    const size_t table_bytes = C->dmask.size() * sizeof(uint64_t);
    if (precision != MLD_FP32 || C->d > 11 || !mld::gate_supported(C->d) ||
        mld::make_plan(C->d, chi).svd_sites != 0 || kStatusSlot + table_bytes > kNoAllocBytes)
        return MLD_ERR_UNSUPPORTED;
    unsigned char* scratch = nullptr;
    int device = 0;
    mld_status st = scratch_address(&scratch, &device);
    if (st != MLD_OK) return st;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    // the status word starts at zero in every call; the tables are uploaded
    // only when the array holds another code's (the previous call's code is
    // remembered per device)
    if (cudaMemsetAsync(scratch, 0, sizeof(int), s) != cudaSuccess) return MLD_ERR_CUDA;
    const uint64_t tables = table_hash(C->dmask);
    {
        std::lock_guard<std::mutex> lock(g_setup_mutex);
        if (g_tables_written[device] != tables) {
            if (cudaMemcpyAsync(scratch + kStatusSlot, C->dmask.data(), table_bytes, cudaMemcpyHostToDevice, s) !=
                cudaSuccess)
                return MLD_ERR_CUDA;
            g_tables_written[device] = tables;
        }
    }
    mld::GateArgs ga;
    ga.dmask = reinterpret_cast<const uint64_t*>(scratch + kStatusSlot);
    ga.noise = noise;
    ga.syn = syndromes;
    ga.logP = logP;
    ga.argmax = argmax;
    ga.status = reinterpret_cast<int*>(scratch);
    ga.B = B;
    ga.noise_mode = noise_mode;
    ga.precision = precision;
    if (!mld::launch_gate(C->d, ga, nullptr, 0, s)) return MLD_ERR_CUDA;
    if (!check_status) return MLD_OK;
    int h = 0;
    if (cudaMemcpyAsync(&h, scratch, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return MLD_ERR_CUDA;
    if (h & (1 << MLD_ERR_INVALID_ARG)) return MLD_ERR_INVALID_ARG;
    if (h & (1 << MLD_ERR_NUMERIC)) return MLD_ERR_NUMERIC;
    if (h & (1 << MLD_ERR_TIMEOUT)) return MLD_ERR_TIMEOUT;
    return MLD_OK;
}
