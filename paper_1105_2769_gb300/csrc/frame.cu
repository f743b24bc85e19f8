// Points in the unit that the contractions work in, and results back from it.
// Two passes over the points, a few microseconds each: launches, not bytes.
#include <algorithm>

#include "frame.h"

namespace {

constexpr int kThreads = 256;

// x_0, or the origin where it is not finite.
__device__ __forceinline__ double origin(const double* X, int c) {
    const double x = X[c];
    return isfinite(x) ? x : 0.0;
}

__device__ __forceinline__ int frame_exponent(const MbmFrame* frame) {
    const double m = __longlong_as_double((long long)frame->extent);
    return m > 0.0 ? 10 - ilogb(m) : 0;
}

__device__ __forceinline__ int weight_exponent(const MbmFrame* frame) {
    const double m = __longlong_as_double((long long)frame->weight);
    return m > 0.0 ? ilogb(m) : 0;
}

// Non-negative doubles order as their bits do.
__device__ __forceinline__ void warp_max_into(unsigned long long* dst, double m) {
    for (int s = 16; s > 0; s >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, s));
    if ((threadIdx.x & 31) == 0 && m > 0.0)
        atomicMax(dst, (unsigned long long)__double_as_longlong(m));
}

__global__ void __launch_bounds__(kThreads)
extent_kernel(const double* __restrict__ X, int64_t N, const double* __restrict__ g,
              MbmFrame* __restrict__ frame, int* __restrict__ gate) {
    const double o[3] = {origin(X, 0), origin(X, 1), origin(X, 2)};
    double m = 0.0, w = 0.0;
    bool over = false;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double x = X[3 * i + c], d = fabs(x - o[c]);
            if (isfinite(d)) m = fmax(m, d);
            else over |= isfinite(x);
        }
        if (g && isfinite(g[i])) w = fmax(w, fabs(g[i]));
    }
    warp_max_into(&frame->extent, m);
    if (g) warp_max_into(&frame->weight, w);
    if (over) *gate = 1;
}

__device__ __forceinline__ void split(double x, float& h, float& l) {
    h = (float)x;
    l = (float)(x - (double)h);
}

__global__ void __launch_bounds__(kThreads)
frame_kernel(const double* __restrict__ X, int64_t N, const double* __restrict__ g,
             const MbmFrame* __restrict__ frame, float4* __restrict__ xh, float4* __restrict__ xl,
             double4_32a* __restrict__ x4, double* __restrict__ gs, MbmOut out,
             int* __restrict__ flags) {
    const int e = frame_exponent(frame), w = weight_exponent(frame);
    const double o[3] = {origin(X, 0), origin(X, 1), origin(X, 2)};
    const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = first; i < N; i += step) {
        double y[3];
        float h[3], l[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double x = X[3 * i + c];
            if (!isfinite(x)) atomicOr(flags, MBM_FLAG_NONFINITE);
            y[c] = scalbn(x, e);
            split(scalbn(x - o[c], e), h[c], l[c]);
        }
        xh[i] = make_float4(h[0], h[1], h[2], 0.f);
        xl[i] = make_float4(l[0], l[1], l[2], 0.f);
        if (x4) x4[i] = make_double4_32a(y[0], y[1], y[2], 0.0);
        if (gs) gs[i] = scalbn(g[i], -w);
    }
    for (int64_t i = first; i < out.n; i += step) {
        out.v[i] = 0.0;
        if (out.lo) out.lo[i] = 0.0;
    }
}

__global__ void __launch_bounds__(kThreads)
unframe_kernel(const double* __restrict__ X, int64_t N, const MbmFrame* __restrict__ frame,
               float4* __restrict__ xh, float4* __restrict__ xl, double4_32a* __restrict__ x4,
               MbmOut out, const int* __restrict__ gate) {
    const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    if (!*gate) {
        const int e = out.degree * frame_exponent(frame) + weight_exponent(frame);
        for (int64_t i = first; i < out.n; i += step)
            out.v[i] = scalbn(out.lo ? out.v[i] + out.lo[i] : out.v[i], e);
        return;
    }
    for (int64_t i = first; i < out.n; i += step) out.v[i] = 0.0;
    for (int64_t i = first; i < N; i += step) {
        const double x = X[3 * i], y = X[3 * i + 1], z = X[3 * i + 2];
        if (x4) {
            x4[i] = make_double4_32a(x, y, z, 0.0);
        } else {
            float h[3], l[3];
            split(x, h[0], l[0]);
            split(y, h[1], l[1]);
            split(z, h[2], l[2]);
            xh[i] = make_float4(h[0], h[1], h[2], 0.f);
            xl[i] = make_float4(l[0], l[1], l[2], 0.f);
        }
    }
}

unsigned blocks_of(int64_t n) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + kThreads - 1) / kThreads, 608));
}

}  // namespace

cudaError_t launch_frame(const double* X, int64_t N, const double* g, MbmFrame* frame, float4* xh,
                         float4* xl, double4_32a* x4, double* gs, const MbmOut& out, int* gate,
                         int* flags, cudaStream_t s) {
    extent_kernel<<<blocks_of(N), kThreads, 0, s>>>(X, N, g, frame, gate);
    frame_kernel<<<blocks_of(N), kThreads, 0, s>>>(X, N, g, frame, xh, xl, x4, gs, out, flags);
    return cudaGetLastError();
}

cudaError_t launch_unframe(const double* X, int64_t N, const MbmFrame* frame, float4* xh, float4* xl,
                           double4_32a* x4, const MbmOut& out, const int* gate, cudaStream_t s) {
    unframe_kernel<<<blocks_of(out.n), kThreads, 0, s>>>(X, N, frame, xh, xl, x4, out, gate);
    return cudaGetLastError();
}
