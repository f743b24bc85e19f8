// Exhaustive potentials, forces and VJPs as a tensor-core contraction (contract.cu).
#pragma once

#include "mbm_internal.h"

enum : int { MBM_CONTRACT_PHI = 0, MBM_CONTRACT_FORCES = 1, MBM_CONTRACT_VJP = 2 };

// Smallest N that goes to the contraction: its chain of small kernels costs 0.2
// ms. Potentials: the pair-table sweep of N = 1 000 takes 0.21 ms, of 2 500 1.72
// (contraction 0.90). Gradients: the gather form of N = 64 takes 0.12 ms (0.19),
// of 100 0.30 (0.19); VJP 0.31 against 0.25.
constexpr int64_t kContractMinPhi = 1280;
constexpr int64_t kContractMinForces = 96;

// Scratch of a potential or force solve of N particles (0: not a contraction).
size_t mbm_contract_bytes(int64_t N, bool forces);

// What the caller's triple sweep needs to solve again on the device if *gate is set.
struct MbmGate {
    const int* gate = nullptr;
    unsigned long long* counter = nullptr;  // zeroed
    const float4* xh = nullptr;             // packed points
    const float4* xl = nullptr;
    void* room = nullptr;                   // scratch that is free by then
    size_t room_bytes = 0;
};

// Enqueue the solve (FP32-bulk accuracy); *done = false if the scratch does not
// fit the budget or the device and nothing was enqueued. The caller enqueues
// its triple sweep behind it, run by the kernels only if *gate is set (out is
// then zeroed). sign multiplies the gradient; g: VJP only.
mbm_status mbm_contract(mbm_ctx* ctx, const double* X, int64_t N, const double* g, int what,
                        double sign, double* out, cudaStream_t s, bool* done, MbmGate* gate);

// The same in FP64 (contract64.cu), potentials and forces.
struct MbmGate64 {
    const int* gate = nullptr;
    unsigned long long* counter = nullptr;  // zeroed
    const double4_32a* x4 = nullptr;        // packed points
};
// (FP64: the sweep of N = 300 takes 1.3 ms and the contraction 0.4; forces of
// N = 100 took 3 ms in gather form and take 0.5.)
constexpr int64_t kContract64MinPhi = 192;
constexpr int64_t kContract64MinForces = 96;
// Scratch of a potential or force solve of N particles (0: not a contraction).
size_t mbm_contract64_bytes(int64_t N, bool forces);
mbm_status mbm_contract64(mbm_ctx* ctx, const double* X, int64_t N, int what, double sign,
                          double* out, cudaStream_t s, bool* done, MbmGate64* gate);
