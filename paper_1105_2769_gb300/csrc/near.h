// Near pairs and the triples that hold one (near.cu).
#pragma once

#include "mbm_internal.h"

// tau[i]: r^2 (FP32, pair_d2_hilo) of particle i's third-nearest neighbour. A
// pair is near if r^2 <= max(tau_i, tau_j): both members see the same answer.
constexpr int kNearK = 3;
constexpr int kNearMax = 16;  // list capacity per particle; more sets the overflow word

size_t mbm_near_bytes(int64_t N);

struct MbmNear {
    float* tau = nullptr;
    int2* pairs = nullptr;      // i < j, ordered by i, then j
    int* count = nullptr;       // their number on the device (0 after an overflow)
    // What two packed points at r^2 <= min_d2 are: coincident if X holds them equal,
    // else too close for their packed form, which sets *overflow. Without X:
    // coincident if r^2 = 0.
    const double* X = nullptr;
    float min_d2 = 0.f;
    unsigned long long* excess = nullptr;  // zeroed word for the count, or NULL
    // Pairs far closer than the usual third neighbour are near too (raises tau).
    bool groups = false;
};

// Thresholds and the ordered list of near pairs, in `mem` (mbm_near_bytes).
// Sets *overflow if the list does not fit or a pair is too close (in/out->X,
// min_d2), MBM_FLAG_COINCIDENT on equal points, which are left out.
cudaError_t launch_near_list(const float4* xh, const float4* xl, int64_t N, void* mem,
                             int* overflow, int* flags, MbmNear* out, cudaStream_t s);

enum : int { MBM_NEAR_PHI = 0, MBM_NEAR_GRAD = 1 };

// Adds the triples with at least one near pair: potentials to out[N], or
// sign * w_t grad phi to out[3 N] (w_t = g_a + g_b + g_c, 1 without g).
// Nothing if *gate is set. out_lo: carries of FP64 potentials. X64: NULL = FP32 terms from xh/xl, else FP64 from these points.
cudaError_t launch_near_triples(const float4* xh, const float4* xl, const double4_32a* X64,
                                int64_t N, const MbmNear& near, const double* g, int what,
                                double sign, double* out, double* out_lo, int num_sms,
                                const int* gate, cudaStream_t s);

// The test itself, on the device.
__device__ __forceinline__ bool mbm_is_near(float s, float tau_a, float tau_b) {
    return s <= fmaxf(tau_a, tau_b);
}
