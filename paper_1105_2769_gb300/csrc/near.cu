// Near pairs, and the triples that hold one, term by term.
//
// The contraction (contract.cu) multiplies matrices of pair terms r^-3 whose
// largest entries are a few close pairs. Those carry most of every sum and set
// the scale that the others are cut against. So each particle's three nearest
// neighbours are taken out of the matrices, and the triples with at least one
// such pair (about 2 N of N^2 / 6 per particle) are summed directly here. What
// is left to the contraction is 4-14 % of a potential and smooth. (Two neighbours
// double the contraction's error, four cost a third more triples here.)
//
// A triple with several near pairs is met once from each of them and counts
// 1/2 or 1/3 each time.
#include <math.h>

#include "device_math.cuh"
#include "dfloat.cuh"
#include "near.h"
#include "sort_scan.h"
#include "tile_fp32.cuh"

namespace {

constexpr int kRowWarps = 8;

// What the pairs of particle i at r^2 <= min_d2 are (rare): MBM_FLAG_COINCIDENT, or
// too close for the packed points, which *overflow takes.
__device__ __noinline__ void sort_out_close(const float4* __restrict__ xh,
                                            const float4* __restrict__ xl, int N, int i, int lane,
                                            const double* __restrict__ X, float min_d2,
                                            int* __restrict__ overflow, int* __restrict__ flags) {
    for (int j = lane; j < N; j += 32) {
        const float s = pair_d2_hilo(xh[i], xl[i], xh[j], xl[j]);
        if (j == i || s > min_d2) continue;
        bool same = !(s > 0.f);
        if (X && s >= 0.f) {
            same = true;
            for (int c = 0; c < 3; ++c) same &= X[3 * (int64_t)i + c] == X[3 * (int64_t)j + c];
            if (!same) *overflow = 1;
        }
        if (same) atomicOr(flags, MBM_FLAG_COINCIDENT);
    }
}

// One warp per particle: the smallest r^2 of each lane, then of the warp.
__global__ void __launch_bounds__(kRowWarps * 32)
knn_kernel(const float4* __restrict__ xh, const float4* __restrict__ xl, int N,
           const double* __restrict__ X, float min_d2, float* __restrict__ tau,
           int* __restrict__ overflow, int* __restrict__ flags) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kRowWarps + (threadIdx.x >> 5);
    if (i >= N) return;
    const float4 ih = xh[i], il = xl[i];
    float t[kNearK];
#pragma unroll
    for (int k = 0; k < kNearK; ++k) t[k] = INFINITY;
    bool close = false;
    for (int j = lane; j < N; j += 32) {
        float s = pair_d2_hilo(ih, il, xh[j], xl[j]);
        if (j == i) continue;
        close |= !(s > min_d2);
        if (!(s > 0.f)) continue;
#pragma unroll
        for (int k = 0; k < kNearK; ++k) {  // insertion into the sorted list
            const float lo = fminf(s, t[k]);
            s = fmaxf(s, t[k]);
            t[k] = lo;
        }
    }
    if (__any_sync(0xffffffffu, close))
        sort_out_close(xh, xl, N, i, lane, X, min_d2, overflow, flags);
    float m = INFINITY;
    for (int k = 0; k < kNearK; ++k) {
        m = t[0];
        for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
        const unsigned holds = __ballot_sync(0xffffffffu, t[0] == m);
        if (lane == __ffs(holds) - 1) {  // one holder drops it
#pragma unroll
            for (int q = 0; q + 1 < kNearK; ++q) t[q] = t[q + 1];
            t[kNearK - 1] = INFINITY;
        }
    }
    if (lane == 0) tau[i] = m < INFINITY ? m : 0.f;
}

// Tight groups. A group of many points far closer than the rest leaves rows of the
// matrices with entries orders above the others', and fixed-point terms (contract64.cu)
// lose those orders in every product with such a row: FP64 forces of 8 000 particles
// beside 30 within 1e-3 of their spacing were off by 1.2e-12 of sum|grad phi|. So pairs
// closer than about a sixth of the usual third neighbour (half the particles have a
// nearer one) are near as well, if they are at most kGroupPairs per particle: ordinary
// sets have next to none.
constexpr int kGroupPairs = 4;

// cut = 2^-6 of the median of tau, to a power of two. One CTA.
__global__ void __launch_bounds__(1024)
group_cut_kernel(const float* __restrict__ tau, int N, float* __restrict__ cut,
                 unsigned long long* __restrict__ close) {
    __shared__ int hist[256];
    if (threadIdx.x < 256) hist[threadIdx.x] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < N; i += blockDim.x)
        atomicAdd(&hist[(__float_as_uint(tau[i]) >> 23) & 255], 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        int e = 0;
        for (int below = hist[0]; e < 254 && 2 * below < N; below += hist[e]) ++e;
        *cut = e > 6 ? __uint_as_float((unsigned)(e - 6) << 23) : 0.f;
        *close = 0;
    }
}

// The pairs that `cut` makes near, counted; then tau raised to it.
__global__ void __launch_bounds__(kRowWarps * 32)
group_count_kernel(const float4* __restrict__ xh, const float4* __restrict__ xl, int N,
                   const float* __restrict__ cut, unsigned long long* __restrict__ close) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kRowWarps + (threadIdx.x >> 5);
    if (i >= N) return;
    const float4 ih = xh[i], il = xl[i];
    const float c = *cut;
    int n = 0;
    for (int j = i + 1 + lane; j < N; j += 32) n += pair_d2_hilo(ih, il, xh[j], xl[j]) <= c;
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0 && n) atomicAdd(close, (unsigned long long)n);
}

__global__ void group_raise_kernel(float* __restrict__ tau, int N, const float* __restrict__ cut,
                                   const unsigned long long* __restrict__ close) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N && *close <= (unsigned long long)kGroupPairs * N) tau[i] = fmaxf(tau[i], *cut);
}

// Near pairs (i, j > i) of a particle: their number (pairs == NULL) or the pairs.
// The numbers are 32-bit and many ties can pass that (points on a few sites: N^2 / 4
// pairs), so what a particle holds beyond kNearMax is also added up in 64 bits
// (`excess`, rarely touched). The list fits only if the excess is at most its
// capacity, and then the 32-bit offsets cannot have wrapped: they are below
// kNearMax N + cap.
__device__ __forceinline__ bool list_overflows(const int* off, int N, int cap,
                                               const unsigned long long* excess) {
    return *excess > (unsigned long long)cap || off[N] > cap;
}

__global__ void __launch_bounds__(kRowWarps * 32)
pairs_kernel(const float4* __restrict__ xh, const float4* __restrict__ xl, int N,
             const float* __restrict__ tau, int* __restrict__ cnt, const int* __restrict__ off,
             int cap, unsigned long long* __restrict__ excess, int2* __restrict__ pairs) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kRowWarps + (threadIdx.x >> 5);
    if (i > N) return;
    if (i == N) {  // one past the end: makes the scan give the total
        if (!pairs && lane == 0) cnt[N] = 0;
        return;
    }
    if (pairs && list_overflows(off, N, cap, excess)) return;
    const float4 ih = xh[i], il = xl[i];
    const float ti = tau[i];
    int at = pairs ? off[i] : 0;
    for (int j0 = i + 1; j0 < N; j0 += 32) {
        const int j = j0 + lane;
        bool near = false;
        if (j < N) {
            const float s = pair_d2_hilo(ih, il, xh[j], xl[j]);
            near = s > 0.f && mbm_is_near(s, ti, tau[j]);
        }
        const unsigned m = __ballot_sync(0xffffffffu, near);
        if (pairs && near) pairs[at + __popc(m & ((1u << lane) - 1u))] = make_int2(i, j);
        at += __popc(m);
    }
    if (!pairs && lane == 0) {
        cnt[i] = at;
        if (at > kNearMax) atomicAdd(excess, (unsigned long long)(at - kNearMax));
    }
}

__global__ void total_kernel(const int* __restrict__ off, int N, int cap,
                             const unsigned long long* __restrict__ excess,
                             int* __restrict__ count, int* __restrict__ overflow) {
    const bool over = list_overflows(off, N, cap, excess);
    *count = over ? 0 : off[N];
    if (over) *overflow = 1;
}

// Unit vector, 1/r and r^-3 of a pair.
template <typename R>
struct Edge {
    R x, y, z, inv, rho;
};
// FP32 from hi/lo points: r^2 carries its rounding and 1/r is refined against
// both parts, so that the results are within an ulp of correctly rounded.
__device__ __forceinline__ Edge<float> edge32(float4 ph, float4 pl, float4 qh, float4 ql) {
    const float dx = (qh.x - ph.x) + (ql.x - pl.x);
    const float dy = (qh.y - ph.y) + (ql.y - pl.y);
    const float dz = (qh.z - ph.z) + (ql.z - pl.z);
    const float xx = __fmul_rn(dx, dx), yy = __fmul_rn(dy, dy), zz = __fmul_rn(dz, dz);
    float e = __fmaf_rn(dx, dx, -xx) + __fmaf_rn(dy, dy, -yy) + __fmaf_rn(dz, dz, -zz);
    const float a = __fadd_rn(xx, yy), at = __fsub_rn(a, xx);
    e += __fadd_rn(__fsub_rn(xx, __fsub_rn(a, at)), __fsub_rn(yy, at));
    const float s = __fadd_rn(a, zz), st = __fsub_rn(s, a);
    e += __fadd_rn(__fsub_rn(a, __fsub_rn(s, st)), __fsub_rn(zz, st));
    const float y0 = rsqrtf(s);
    const float p = __fmul_rn(y0, y0), pe = __fmaf_rn(y0, y0, -p);
    const float q = __fmul_rn(s, p), qe = __fmaf_rn(s, p, -q);
    const float res = __fsub_rn(__fsub_rn(1.0f, q), __fmaf_rn(e, p, __fmaf_rn(s, pe, qe)));
    const float dl = __fmul_rn(__fmul_rn(0.5f, y0), res);  // y = y0 + dl
    Edge<float> r;
    r.inv = __fadd_rn(y0, dl);
    r.x = __fmaf_rn(dx, dl, __fmul_rn(dx, y0));
    r.y = __fmaf_rn(dy, dl, __fmul_rn(dy, y0));
    r.z = __fmaf_rn(dz, dl, __fmul_rn(dz, y0));
    // y^3 = y0^3 + 3 y0^2 dl, with the rounding of y0^2
    r.rho = __fmaf_rn(p, y0, __fmaf_rn(pe, y0, __fmul_rn(__fmul_rn(3.0f, p), dl)));
    return r;
}
__device__ __forceinline__ Edge<double> edge64(double4_32a p, double4_32a q) {
    const double dx = q.x - p.x, dy = q.y - p.y, dz = q.z - p.z;
    const double s = dx * dx + dy * dy + dz * dz;
    const double y = rsqrt(s);
    return {dx * y, dy * y, dz * y, y, y * y * y};
}

// Edge vector, r^-2 and r^-3 to about 2^-40 for FP32 potentials: what the near
// triples lose is lost in the result, and they are few.
struct EdgeDf {
    df d[3], q, rho;
};
__device__ __forceinline__ EdgeDf edge_df(float4 ph, float4 pl, float4 qh, float4 ql) {
    EdgeDf r;
    r.d[0] = df_diff(qh.x, ql.x, ph.x, pl.x);
    r.d[1] = df_diff(qh.y, ql.y, ph.y, pl.y);
    r.d[2] = df_diff(qh.z, ql.z, ph.z, pl.z);
    const df y = df_rsqrt(df_dot(r.d, r.d));
    r.q = df_mul(y, y);
    r.rho = df_mul(r.q, y);
    return r;
}
// phi from three edges u = ab, a = ak, b = bk: with D the dot products of the edge
// vectors, cos cos cos = -(u.a)(u.b)(a.b) / (s_u s_a s_b).
__device__ __forceinline__ float phi_df(const EdgeDf& u, const EdgeDf& a, const EdgeDf& b) {
    const df d = df_mul(df_mul(df_dot(u.d, a.d), df_dot(u.d, b.d)), df_dot(a.d, b.d));
    const df t = df_mul(d, df_mul(u.q, df_mul(a.q, b.q)));
    const df n = df_add(df{1.0f, 0.0f}, df_mul(df{-3.0f, 0.0f}, t));
    const df f = df_mul(n, df_mul(u.rho, df_mul(a.rho, b.rho)));
    return f.h;
}

constexpr int kChunk = 32;      // near pairs staged at a time, one per lane in the sums
constexpr int kNearWarps = 4;   // 128 particles j per CTA

template <typename R>
struct NearPair {
    Edge<R> e;  // from i to j of the pair
    EdgeDf d;   // the same for FP32 potentials
    R w;        // g_i + g_j
    float ti, tj;
    int i, j;
};

// A CTA owns 128 particles k, one per lane, and every gridDim.y-th chunk of near
// pairs (a, b). k's share stays in registers; the shares of a and b are summed
// over the lanes through a transposed buffer, 32 pairs at a time. Bound by FP32
// instructions (FMA pipe 71 %, issue 82 %, 1.7 ms at N = 8 192) or, in FP64, by that
// pipe; FP32 gradients by the conversions of their sums to FP64 (pipe 82 %, 1.6 ms). Chunks of 32 pairs, not 64 or more: N = 700 has only 1 400 pairs for the
// whole chip.
template <typename R, bool Grad>
__global__ void __launch_bounds__(kNearWarps * 32)
near_kernel(const float4* __restrict__ xh, const float4* __restrict__ xl,
            const double4_32a* __restrict__ x64, int N, const float* __restrict__ tau,
            const int2* __restrict__ pairs, const int* __restrict__ count,
            const double* __restrict__ g, double sign, double* __restrict__ out,
            double* __restrict__ out_lo, const int* __restrict__ gate) {
    if (*gate) return;
    constexpr int kRow = Grad ? 6 : 1;   // shares of a and b
    constexpr int kCol = Grad ? 3 : 1;
    __shared__ NearPair<R> np[kChunk];
    __shared__ float4 ah[kChunk], al[kChunk], bh[kChunk], bl[kChunk];
    __shared__ R red[kNearWarps][32][33];
    __shared__ double rows[kRow][kNearWarps][kChunk];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.x * (kNearWarps * 32) + threadIdx.x;
    const bool kv = k < N;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 kh = kv ? xh[k] : z4, kl = kv ? xl[k] : z4;
    double4_32a kd = make_double4_32a(0, 0, 0, 0);
    if (sizeof(R) == 8 && kv) kd = x64[k];
    const float tk = kv ? tau[k] : 0.f;
    const R gk = g && kv ? (R)g[k] : (R)0;
    const int M = *count;
    double col[kCol];
#pragma unroll
    for (int d = 0; d < kCol; ++d) col[d] = 0.0;
    for (int p0 = blockIdx.y * kChunk; p0 < M; p0 += gridDim.y * kChunk) {
        const int cnt = min(kChunk, M - p0);
        __syncthreads();
        if (threadIdx.x < kChunk && (int)threadIdx.x < cnt) {
            const int2 ab = pairs[p0 + threadIdx.x];
            NearPair<R> q;
            q.i = ab.x;
            q.j = ab.y;
            q.ti = tau[ab.x];
            q.tj = tau[ab.y];
            q.w = g ? (R)(g[ab.x] + g[ab.y]) : (R)1;
            ah[threadIdx.x] = xh[ab.x];
            al[threadIdx.x] = xl[ab.x];
            bh[threadIdx.x] = xh[ab.y];
            bl[threadIdx.x] = xl[ab.y];
            if constexpr (sizeof(R) == 8) q.e = edge64(x64[ab.x], x64[ab.y]);
            else if constexpr (Grad) q.e = edge32(xh[ab.x], xl[ab.x], xh[ab.y], xl[ab.y]);
            else q.d = edge_df(xh[ab.x], xl[ab.x], xh[ab.y], xl[ab.y]);
            np[threadIdx.x] = q;
        }
        __syncthreads();
        R part[kCol], row[kRow];
#pragma unroll
        for (int d = 0; d < kCol; ++d) part[d] = 0;
        float low = 0.f;
        (void)low;
        for (int p = 0; p < kChunk; ++p) {
#pragma unroll
            for (int d = 0; d < kRow; ++d) row[d] = 0;
            if (p < cnt && kv) {
                const NearPair<R>& n = np[p];
                const float sa = pair_d2_hilo(ah[p], al[p], kh, kl);
                const float sb = pair_d2_hilo(bh[p], bl[p], kh, kl);
                if (k != n.i && k != n.j && sa > 0.f && sb > 0.f) {
                    const int hits = 1 + (int)mbm_is_near(sa, n.ti, tk) +
                                     (int)mbm_is_near(sb, n.tj, tk);
                    R w = hits == 1 ? (R)1 : hits == 2 ? (R)0.5 : (R)1 / (R)3;
                    if constexpr (sizeof(R) == 4 && !Grad) {
                        const float f = (float)w * phi_df(n.d, edge_df(ah[p], al[p], kh, kl),
                                                          edge_df(bh[p], bl[p], kh, kl));
                        // carried sums: see row_sum_exact
                        const float t = __fadd_rn(part[0], f), bb = __fsub_rn(t, part[0]);
                        low = __fadd_rn(low, __fadd_rn(__fsub_rn(part[0], __fsub_rn(t, bb)),
                                                       __fsub_rn(f, bb)));
                        part[0] = t;
                        row[0] = f;
                    } else {
                        Edge<R> a, b;
                        if constexpr (sizeof(R) == 8) {
                            a = edge64(x64[n.i], kd);
                            b = edge64(x64[n.j], kd);
                        } else {
                            a = edge32(ah[p], al[p], kh, kl);
                            b = edge32(bh[p], bl[p], kh, kl);
                        }
                        const R ux = n.e.x, uy = n.e.y, uz = n.e.z;
                        const R p1 = ux * a.x + uy * a.y + uz * a.z;
                        const R p2 = ux * b.x + uy * b.y + uz * b.z;
                        const R p3 = a.x * b.x + a.y * b.y + a.z * b.z;
                        const R rr = n.e.rho * a.rho * b.rho;
                        if constexpr (!Grad) {
                            const R f = w * (rr - (R)3 * (p1 * p2 * p3) * rr);
                            part[0] += f;
                            row[0] = f;
                        } else {
                            w *= g ? n.w + gk : (R)1;
                            const R qf = (R)5 * (p1 * p2 * p3) - (R)1;
                            const R t3 = (R)3 * rr * w;
                            const R su = t3 * n.e.inv, sa3 = t3 * a.inv, sb3 = t3 * b.inv;
                            const R p23 = p2 * p3, p13 = p1 * p3, p12 = p1 * p2;
                            // grad_a = -c1 u - c2 e_ak + c3 e_bk
                            R c1 = su * qf - sa3 * p23, c2 = sa3 * qf - su * p23,
                              c3 = su * p13 + sa3 * p12;
                            row[0] = c3 * b.x - c1 * ux - c2 * a.x;
                            row[1] = c3 * b.y - c1 * uy - c2 * a.y;
                            row[2] = c3 * b.z - c1 * uz - c2 * a.z;
                            // grad_b = c1' u - c2' e_bk + c3' e_ak
                            c1 = su * qf + sb3 * p13;
                            c2 = sb3 * qf + su * p13;
                            c3 = sb3 * p12 - su * p23;
                            row[kRow - 3] = c1 * ux - c2 * b.x + c3 * a.x;
                            row[kRow - 2] = c1 * uy - c2 * b.y + c3 * a.y;
                            row[kRow - 1] = c1 * uz - c2 * b.z + c3 * a.z;
                            // grad_k by itself: as minus the sum of the other two it
                            // would carry their rounding, which for a pair far
                            // closer than k is 1 / r_ab against grad_k's 1 / r_ak
                            c1 = sa3 * qf - sb3 * p12;
                            c2 = sb3 * qf - sa3 * p12;
                            c3 = sa3 * p23 + sb3 * p13;
                            part[0] += c1 * a.x + c2 * b.x - c3 * ux;
                            part[kCol / 2] += c1 * a.y + c2 * b.y - c3 * uy;
                            part[kCol - 1] += c1 * a.z + c2 * b.z - c3 * uz;
                        }
                    }
                }
            }
            if constexpr (Grad) {
                // six sums over the warp by butterflies, lane p keeps pair p's
#pragma unroll
                for (int d = 0; d < kRow; ++d) {
                    R v = row[d];
                    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                    if (lane == p) rows[d][warp][p] = (double)v;
                }
            } else {
                red[warp][p][lane] = row[0];
            }
        }
        if constexpr (!Grad) {
            __syncwarp();
            if constexpr (sizeof(R) == 4) {
                rows[0][warp][lane] = mbm_tile::row_sum_exact(red[warp], lane);
            } else {
                R t = 0;
#pragma unroll 8
                for (int q = 0; q < 32; ++q) t += red[warp][lane][q];
                rows[0][warp][lane] = (double)t;
            }
            __syncwarp();
        }
#pragma unroll
        for (int d = 0; d < kCol; ++d) col[d] += (double)part[d];
        if constexpr (sizeof(R) == 4 && !Grad) col[0] += (double)low;
        __syncthreads();
        if ((int)threadIdx.x < cnt) {
#pragma unroll
            for (int d = 0; d < kRow; ++d) {
                double t = 0.0;
#pragma unroll
                for (int w = 0; w < kNearWarps; ++w) t += rows[d][w][threadIdx.x];
                if constexpr (Grad) {
                    const int o = d < 3 ? np[threadIdx.x].i : np[threadIdx.x].j;
                    atomicAdd(&out[3 * (size_t)o + d % 3], sign * t);
                } else if constexpr (sizeof(R) == 8) {
                    const int i = np[threadIdx.x].i, j = np[threadIdx.x].j;
                    atomic_add_carried(&out[i], &out_lo[i], t);
                    atomic_add_carried(&out[j], &out_lo[j], t);
                } else {
                    atomicAdd(&out[np[threadIdx.x].i], t);
                    atomicAdd(&out[np[threadIdx.x].j], t);
                }
            }
        }
    }
    if (kv) {
#pragma unroll
        for (int d = 0; d < kCol; ++d)
            if constexpr (Grad) atomicAdd(&out[3 * (size_t)k + d], sign * col[d]);
            else if constexpr (sizeof(R) == 8) atomic_add_carried(&out[k], &out_lo[k], col[d]);
            else atomicAdd(&out[k], col[d]);
    }
}

size_t up256(size_t b) { return mbm_align_up(b, 256); }

}  // namespace

size_t mbm_near_bytes(int64_t N) {
    return up256((size_t)N * 4) + up256((size_t)(N + 1) * 4) * 2 + 256 +
           up256((size_t)N * kNearMax * sizeof(int2)) + up256(mbm_scan_temp_bytes_i32(N + 1));
}

cudaError_t launch_near_list(const float4* xh, const float4* xl, int64_t N, void* mem,
                             int* overflow, int* flags, MbmNear* out, cudaStream_t s) {
    char* q = static_cast<char*>(mem);
    auto take = [&](size_t bytes) {
        char* r = q;
        q += up256(bytes);
        return r;
    };
    out->tau = reinterpret_cast<float*>(take((size_t)N * 4));
    int* cnt = reinterpret_cast<int*>(take((size_t)(N + 1) * 4));
    int* off = reinterpret_cast<int*>(take((size_t)(N + 1) * 4));
    out->count = reinterpret_cast<int*>(take(256));
    auto* excess = out->excess;
    out->pairs = reinterpret_cast<int2*>(take((size_t)N * kNearMax * sizeof(int2)));
    void* tmp = take(mbm_scan_temp_bytes_i32(N + 1));
    const int cap = (int)(N * kNearMax);
    const unsigned rows = (unsigned)((N + kRowWarps) / kRowWarps);
    cudaError_t e;
    if (!excess) {
        excess = reinterpret_cast<unsigned long long*>(out->count + 16);
        e = cudaMemsetAsync(excess, 0, sizeof(*excess), s);
        if (e != cudaSuccess) return e;
    }
    knn_kernel<<<rows, kRowWarps * 32, 0, s>>>(xh, xl, (int)N, out->X, out->min_d2, out->tau,
                                               overflow, flags);
    if (out->groups) {
        auto* cut = reinterpret_cast<float*>(out->count + 32);
        auto* close = reinterpret_cast<unsigned long long*>(out->count + 34);
        group_cut_kernel<<<1, 1024, 0, s>>>(out->tau, (int)N, cut, close);
        group_count_kernel<<<rows, kRowWarps * 32, 0, s>>>(xh, xl, (int)N, cut, close);
        group_raise_kernel<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(out->tau, (int)N, cut,
                                                                       close);
    }
    pairs_kernel<<<rows, kRowWarps * 32, 0, s>>>(xh, xl, (int)N, out->tau, cnt, nullptr, cap,
                                                 excess, nullptr);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = mbm_exclusive_scan_i32(cnt, off, N + 1, tmp, s);
    if (e != cudaSuccess) return e;
    pairs_kernel<<<rows, kRowWarps * 32, 0, s>>>(xh, xl, (int)N, out->tau, cnt, off, cap,
                                                 excess, out->pairs);
    total_kernel<<<1, 1, 0, s>>>(off, (int)N, cap, excess, out->count, overflow);
    return cudaGetLastError();
}

cudaError_t launch_near_triples(const float4* xh, const float4* xl, const double4_32a* X64,
                                int64_t N, const MbmNear& near, const double* g, int what,
                                double sign, double* out, double* out_lo, int num_sms,
                                const int* gate, cudaStream_t s) {
    const unsigned bx = (unsigned)((N + kNearWarps * 32 - 1) / (kNearWarps * 32));
    // about 2 N pairs; enough CTAs for eight per SM, at least one chunk each
    const int64_t chunks = (2 * N + kChunk - 1) / kChunk;
    int64_t by = (8 * (int64_t)(num_sms > 0 ? num_sms : 1) + bx - 1) / bx;
    if (by > chunks) by = chunks;
    const dim3 grid(bx, (unsigned)(by < 1 ? 1 : by));
    const int threads = kNearWarps * 32;
    if (what == MBM_NEAR_PHI) {
        if (X64)
            near_kernel<double, false><<<grid, threads, 0, s>>>(
                xh, xl, X64, (int)N, near.tau, near.pairs, near.count, g, sign, out, out_lo, gate);
        else
            near_kernel<float, false><<<grid, threads, 0, s>>>(
                xh, xl, X64, (int)N, near.tau, near.pairs, near.count, g, sign, out, out_lo, gate);
    } else {
        if (X64)
            near_kernel<double, true><<<grid, threads, 0, s>>>(
                xh, xl, X64, (int)N, near.tau, near.pairs, near.count, g, sign, out, out_lo, gate);
        else
            near_kernel<float, true><<<grid, threads, 0, s>>>(
                xh, xl, X64, (int)N, near.tau, near.pairs, near.count, g, sign, out, out_lo, gate);
    }
    return cudaGetLastError();
}
