// The frame that the contractions work in (frame.cu): points are multiplied by a
// power of two 2^e such that max |x - x_0| falls in [2^10, 2^11), so that FP32
// quantities of the set (squared distances, r^-3, products of three edges) stay in
// range whatever unit the caller's coordinates are in. Powers of two change no
// digit: phi is homogeneous of degree -9, its gradient of degree -10. A VJP is linear
// in its weights, which are brought to [-2, 2] in the same way.
#pragma once

#include "mbm_internal.h"

struct MbmFrame {                // device words, zeroed by the caller
    unsigned long long extent;   // bits of max |x - x_0| over the coordinates (FP64)
    unsigned long long weight;   // bits of max |g|; 0 without weights
};

// Results, zeroed on the way in.
struct MbmOut {
    double* v;
    int64_t n;    // numbers
    int degree;   // 9 for potentials, 10 for gradients
    double* lo = nullptr;  // what the additions to v rounded off (NULL: not carried)
};

// The frame of X and the packed points in it: x4 = 2^e x (FP64), and xh + xl =
// 2^e (x - x_0) in two FP32 parts; gs = scaled weights (x4, and g with gs: NULL = not
// asked for). Sets MBM_FLAG_NONFINITE on points that are not finite, and *gate if the
// extent of finite points is not.
cudaError_t launch_frame(const double* X, int64_t N, const double* g, MbmFrame* frame, float4* xh,
                         float4* xl, double4_32a* x4, double* gs, const MbmOut& out, int* gate,
                         int* flags, cudaStream_t s);

// Out of the frame: out (with lo) times 2^(degree e) and the weights' unit. If *gate is set, zero
// instead, and the points packed as they are (x4, or xh and xl), for the sweep behind.
cudaError_t launch_unframe(const double* X, int64_t N, const MbmFrame* frame, float4* xh, float4* xl,
                           double4_32a* x4, const MbmOut& out, const int* gate, cudaStream_t s);
