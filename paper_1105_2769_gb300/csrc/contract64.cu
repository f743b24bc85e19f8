// FP64 exhaustive potentials and forces as a contraction in exact fp16 products.
//
// The same matrix products as contract.cu (see there for the identity and for the
// near triples that are summed term by term, here in FP64). FP64 runs at 1/64 of
// the FP32 rate, so the products run on the tensor cores: a row of L is cut
// against a power of two a per row and block of 256 or 512 columns, |a L| < 2^7,
// into seven signed base-256 digits (to 2^-48). A product of two digits is below
// 2^14, and the up to seven products of one weight 2^-8g over a stage of 32
// columns sum to less than 2^22: exact in the FP32 accumulator, whatever the
// order. The read-out moves each sum to an integer by one FP32 addition of
// 1.5 2^23 and adds it to a 64-bit fixed-point sum at its weight; products below
// 2^-48 are left out. The 64-bit sums of a block are converted, scaled and added in FP64 by
// the pair pass. Error of the contraction: 4e-17 of a potential (norm, N = 300);
// with the near triples the result is as close to 64 bits as the FP64 sweep's (norm
// and median at or below it for N = 100 to 3 001, unit, uniform and mixture sets). An
// entry far below its row's largest within a block keeps fewer bits than FP64 would,
// so pairs of a tight group are near pairs (near.cu): beside 30 points within 1e-3 of
// the spacing of 8 000 others, potentials were off by 2.1e-12 of sum|phi| and forces by
// 1.2e-12 of sum|grad phi|, and are by 5e-16.
//
// Range. FP32 carries the near test and the exponents, so the points are brought to
// a common unit first (frame.h): |x - x_0| < 2^11. With r >= 2^-19 there, every FP32
// quantity is in range, and r^2 from the two FP32 parts of a point (2^-49 of it) is
// within 2^-17: inside the exponents' margin. A set with a closer pair goes to the
// FP64 sweep, decided on the device (gate); so does one with more than 16 near
// pairs per particle.
//
// Kernels: near pairs; block maxima -> exponents; digit table (operand layout);
// contraction (tcgen05.mma 128 x 128); pair pass in FP64; near triples in FP64.
#include <algorithm>
#include <type_traits>
#include <cuda_fp16.h>

#include "bulk_copy.cuh"
#include "contract.h"
#include "device_math.cuh"
#include "forms.cuh"
#include "frame.h"
#include "near.h"
#include "tcgen05.cuh"

namespace {

constexpr int kDigits = 7;
constexpr int kRows = 128;   // rows and columns of a tile
constexpr int kBK = 32;      // columns k per stage
constexpr int kPiece = kRows * kBK * 2;           // 8 KB: one digit of 128 rows x 32 columns
constexpr int kStageBytes = kDigits * kPiece;     // one operand of a stage
constexpr int kStages = 2;
constexpr int kBufs = 4;     // TMEM accumulators of 128 columns
constexpr int kEpiWarps = 16;
constexpr int kThreads = (kEpiWarps + 2) * 32;
constexpr long long kWaitLimit = 4000000000LL;

// Block of S stages: its 64-bit sums hold the weight-0 products, below 2^19 a
// stage, at 2^base: 2^62 at most.
__host__ __device__ constexpr int base_shift(int S) { return S == 8 ? 40 : 39; }

__device__ __forceinline__ double pow2d(int e) {
    return __longlong_as_double((long long)(e + 1023) << 52);
}

// ---------------------------------------------------------------------------
// Exponents. ea[b][i]: |2^ea l| < 2^7 over the columns k of block b without near
// pairs. A CTA takes 256 rows and one block.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
exponent_kernel(const float4* __restrict__ xh, const float4* __restrict__ xl, int N, int cols,
                const float* __restrict__ tau, int n_pad, int* __restrict__ ea,
                const int* __restrict__ gate) {
    if (*gate) return;
    __shared__ float4 kh[256], kl[256];
    __shared__ float kt[256];
    const int b = blockIdx.y, i = blockIdx.x * 256 + threadIdx.x;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 ih = i < N ? xh[i] : z4, il = i < N ? xl[i] : z4;
    const float ti = i < N ? tau[i] : 0.f;
    float smin = INFINITY;
    for (int k0 = b * cols; k0 < (b + 1) * cols; k0 += 256) {
        const int kk = k0 + threadIdx.x;
        __syncthreads();
        kh[threadIdx.x] = kk < N ? xh[kk] : z4;
        kl[threadIdx.x] = kk < N ? xl[kk] : z4;
        kt[threadIdx.x] = kk < N ? tau[kk] : 0.f;
        __syncthreads();
        const int cnt = min(256, N - k0);
        if (i < N)
            for (int q = 0; q < cnt; ++q) {
                const float s = pair_d2_hilo(ih, il, kh[q], kl[q]);
                if (!mbm_is_near(s, ti, kt[q]) && s < INFINITY) smin = fminf(smin, s);
            }
    }
    int e = 0;
    if (smin < INFINITY) {
        const float y = rsqrtf(smin);
        e = 6 - ilogbf(y * y * y * (kFormMax * 1.0001f));
    }
    if (i < n_pad) ea[(size_t)b * n_pad + i] = e;
}

// ---------------------------------------------------------------------------
// Digit table, in the contraction's operand layout: T[r][row block][kb][digit] is
// 128 rows x 32 columns as core matrices of 8 rows x 8 columns. A thread owns a
// row and 8 columns; a CTA 128 rows x 8 columns x all forms. FP64 carries the
// pair terms and the forms (about 90 operations per pair), integers the digits.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kRows)
digit_kernel(const double4_32a* __restrict__ x4, const float4* __restrict__ xh,
             const float4* __restrict__ xl, int N, const float* __restrict__ tau, int n_pad, int nb,
             int kb0, int nkb, int stages, const int* __restrict__ ea,
             unsigned char* __restrict__ T, const int* __restrict__ gate) {
    if (*gate) return;
    __shared__ double coef[kForms][5];
    const int rb = blockIdx.x, kb = blockIdx.y, k8 = blockIdx.z;
    const int row = threadIdx.x, i = rb * kRows + row;
    if (threadIdx.x < kForms * 5)
        coef[threadIdx.x / 5][threadIdx.x % 5] = form_coef(threadIdx.x / 5, threadIdx.x % 5);
    __syncthreads();
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 ih = i < N ? xh[i] : z4, il = i < N ? xl[i] : z4;
    const float ti = i < N ? tau[i] : 0.f;
    const double4_32a xi = i < N ? x4[i] : make_double4_32a(0, 0, 0, 0);
    // terms in units of 2^-48 of |2^ea l| < 2^7
    const double a = i < N ? pow2d(ea[(size_t)((kb0 + kb) / stages) * n_pad + i] + 48) : 0.0;
    const size_t off = (size_t)(row >> 3) * 512 + k8 * 128 + (row & 7) * 16;
    double v[8][5];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int k = (kb0 + kb) * kBK + k8 * 8 + q;
#pragma unroll
        for (int m = 0; m < 5; ++m) v[q][m] = 0.0;
        if (i < N && k < N && k != i) {
            const float s32 = pair_d2_hilo(ih, il, xh[k], xl[k]);
            if (s32 < INFINITY && !mbm_is_near(s32, ti, tau[k])) {
                const double4_32a xk = x4[k];
                const double dx = xk.x - xi.x, dy = xk.y - xi.y, dz = xk.z - xi.z;
                const double xx = dx * dx, yy = dy * dy, zz = dz * dz;
                const double y = rsqrt(xx + yy + zz), y2 = y * y;
                const double w = a * y * y2 * y2;  // a rho / r^2
                v[q][0] = (xx - zz) * w;
                v[q][1] = (yy - zz) * w;
                v[q][2] = dx * dy * w;
                v[q][3] = dx * dz * w;
                v[q][4] = dy * dz * w;
            }
        }
    }
#pragma unroll 1
    for (int r = 0; r < kForms; ++r) {
        __align__(16) __half d[kDigits][8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            double x = coef[r][0] * v[q][0];
#pragma unroll
            for (int m = 1; m < 5; ++m) x = fma(coef[r][m], v[q][m], x);
            long long X = __double2ll_rn(x);
#pragma unroll
            for (int p = kDigits - 1; p > 0; --p) {
                const int digit = (int)(signed char)(X & 0xff);
                // 1152 + digit is an fp16 with unit spacing
                d[p][q] = __hsub(__ushort_as_half((unsigned short)(0x6400 + 128 + digit)),
                                 __ushort_as_half((unsigned short)(0x6400 + 128)));
                X = (X - digit) >> 8;
            }
            d[0][q] = __hsub(__ushort_as_half((unsigned short)(0x6400 + 256 + (int)X)),
                             __ushort_as_half((unsigned short)(0x6400 + 256)));
        }
        unsigned char* dst = T + (((size_t)r * nb + rb) * nkb + kb) * (size_t)kStageBytes + off;
#pragma unroll
        for (int p = 0; p < kDigits; ++p)
            *reinterpret_cast<uint4*>(dst + p * kPiece) = *reinterpret_cast<const uint4*>(d[p]);
    }
}

// ---------------------------------------------------------------------------
// Contraction.
// ---------------------------------------------------------------------------
// Tile t -> row blocks I <= J.
__device__ __forceinline__ void decode_tile(int t, int& I, int& J) {
    J = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
    while (J * (J + 1) / 2 > t) --J;
    while ((J + 1) * (J + 2) / 2 <= t) ++J;
    I = t - J * (J + 1) / 2;
}

struct ContractSmem {
    unsigned char a[kStages][kStageBytes];
    unsigned char b[kStages][kStageBytes];
    unsigned long long full[kStages], empty[kStages];
    unsigned long long acc_full[kBufs], acc_empty[kBufs];
    unsigned long long done;  // the MMAs have ended
    unsigned tmem;
    volatile int abort;
};

// Bounded wait; the first one to give up tells every role to stop.
__device__ __forceinline__ bool wait_phase(ContractSmem& sm, unsigned long long* bar,
                                           unsigned parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
        if (mbar_try_wait(bar, parity)) return true;
        if (sm.abort) return false;
        if (clock64() - t0 > kWaitLimit) {
            sm.abort = 1;
            return false;
        }
    }
}

// The integer v (|v| < 2^22) at weight 2^shift onto t, with the constant of the
// conversion; a negative shift rounds to nearest.
template <int Shift>
__device__ __forceinline__ void add_shifted(unsigned long long& t, float v) {
    constexpr float kMagic = 12582912.0f + (Shift < 0 ? (float)(1 << (Shift < 0 ? -Shift - 1 : 0)) : 0.f);
    const unsigned raw = __float_as_uint(__fadd_rn(v, kMagic));
    if constexpr (Shift >= 32) t += (unsigned long long)(raw << (Shift - 32)) << 32;
    else if constexpr (Shift >= 0) t += (unsigned long long)raw * (1ull << Shift);
    else t += (unsigned long long)(raw >> -Shift);
}
// What the conversions of one stage add, modulo 2^64.
template <int Base>
__host__ __device__ constexpr unsigned long long stage_bias() {
    unsigned long long s = 0;
    for (int g = 0; g < kDigits; ++g) {
        const int shift = Base - 8 * g;
        const unsigned long long raw = 0x4B400000ull;
        if (shift >= 32) s += (unsigned long long)(unsigned)(raw << (shift - 32)) << 32;
        else if (shift >= 0) s += raw * (1ull << shift);
        else s += raw >> -shift;
    }
    return s;
}

template <int Base, int G>
__device__ __forceinline__ void read_out(unsigned addr, unsigned long long (&t)[32]) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        float v[16];
        tc_ld16(addr + 16 * c, v);
        tc_wait_ld();
#pragma unroll
        for (int q = 0; q < 16; ++q) add_shifted<Base - 8 * G>(t[16 * c + q], v[q]);
    }
}

// C[item][block][column / 2][row][2]: 64-bit sums at 2^Base. One CTA per SM, items
// (form, tile) dealt round robin. Warps 0-15: read-outs, a group of products of
// one weight at a time, onto 32 sums per thread; warp 16: bulk copies (112 KB
// stages); warp 17: MMAs, 28 products a stage. Four accumulators let the MMAs
// run three groups ahead of the read-out, which bounds it: 10.5 ms at N = 3 001,
// three times the products' time. (Two groups as one 32-bit integer per 64-bit
// addition spilled at 96 registers: 11.4.)
template <int Stages>  // stages per block
__global__ void __launch_bounds__(kThreads, 1)
contract64_kernel(const unsigned char* __restrict__ T, int nb, int nkb, int t0, int nt,
                  longlong2* __restrict__ C, int* gate, int expire) {
    // (a CTA of this launch may set it meanwhile: one answer for all threads)
    if (__syncthreads_or(*gate)) return;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    ContractSmem& sm = *reinterpret_cast<ContractSmem*>(smem_raw);
    constexpr int kBase = base_shift(Stages);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&sm.full[s], 1);
            mbar_init(&sm.empty[s], 1);
        }
        for (int a = 0; a < kBufs; ++a) {
            mbar_init(&sm.acc_full[a], 1);
            mbar_init(&sm.acc_empty[a], kEpiWarps);
        }
        mbar_init(&sm.done, 1);
        sm.abort = 0;
        mbar_fence_init();
    }
    if (warp == 0) tc_alloc(smem_u32(&sm.tmem), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = sm.tmem;
    const int n_items = nt * kForms;
    if (warp == kEpiWarps) {
        if (lane == 0) {
            unsigned it = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                const int r = item / nt;
                int I, J;
                decode_tile(t0 + item % nt, I, J);
                const unsigned char* pa = T + ((size_t)r * nb + I) * nkb * kStageBytes;
                const unsigned char* pb = T + ((size_t)r * nb + J) * nkb * kStageBytes;
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % kStages;
                    if (it >= kStages &&
                        !wait_phase(sm, &sm.empty[s], (it / kStages - 1) & 1)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(&sm.full[s], 2 * kStageBytes);
                    bulk_copy_g2s(sm.a[s], pa + (size_t)kb * kStageBytes, kStageBytes, &sm.full[s]);
                    bulk_copy_g2s(sm.b[s], pb + (size_t)kb * kStageBytes, kStageBytes, &sm.full[s]);
                }
            }
            // copies in flight land before shared memory is released
            for (unsigned q = it > kStages ? it - kStages : 0; q < it; ++q)
                mbar_wait_bounded(&sm.full[q % kStages], (q / kStages) & 1, kWaitLimit);
        }
    } else if (warp == kEpiWarps + 1) {
        if (lane == 0) {
            constexpr unsigned idesc = tc_idesc_f16(kRows, kRows);
            unsigned it = 0, grp = 0;  // stages and groups begun
            bool ok = true;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                for (int kb = 0; kb < nkb && ok; ++kb, ++it) {
                    const int s = it % kStages;
                    if (!wait_phase(sm, &sm.full[s], (it / kStages) & 1)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const unsigned ab = smem_u32(sm.a[s]), bb = smem_u32(sm.b[s]);
#pragma unroll 1
                    for (int g = 0; g < kDigits; ++g, ++grp) {
                        const unsigned buf = grp % kBufs;
                        if (grp >= kBufs &&
                            !wait_phase(sm, &sm.acc_empty[buf], (grp / kBufs - 1) & 1)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
#pragma unroll 1
                        for (int p = 0; p <= g; ++p)
#pragma unroll
                            for (int k = 0; k < kBK / 16; ++k)
                                tc_mma_f16(tmem + buf * kRows,
                                           tc_desc(ab + p * kPiece + k * 256, 128, 512),
                                           tc_desc(bb + (g - p) * kPiece + k * 256, 128, 512),
                                           idesc, p + k > 0);
                        tc_commit(smem_u32(&sm.acc_full[buf]));
                    }
                    if (expire) {  // a switch of tests: run out with MMAs under way
                        sm.abort = 1;
                        ok = false;
                    }
                    if (ok) tc_commit(smem_u32(&sm.empty[s]));
                }
            }
            // MMAs in flight end before TMEM and shared memory are released, also those
            // that an expired wait left without a commit
            tc_commit(smem_u32(&sm.done));
            mbar_wait_bounded(&sm.done, 0, kWaitLimit);
        }
    } else {
        // rows 32 (warp % 4) + lane of the tile, columns 32 (warp / 4) + 0..31
        const int row = (warp & 3) * 32 + lane, col = (warp >> 2) * 32;
        const unsigned base = tmem + ((unsigned)(warp & 3) << 21) + col;
        unsigned grp = 0;
        bool ok = true;
        for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
            longlong2* out = C + (size_t)((item % nt) * kForms + item / nt) * (nkb / Stages) *
                                     (kRows * kRows / 2) +
                             (size_t)(col / 2) * kRows + row;
            unsigned long long t[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) t[c] = 0ull;
            for (int kb = 0; kb < nkb && ok; ++kb) {
                auto group = [&](auto G) {
                    if (!ok) return;
                    const unsigned buf = grp % kBufs;
                    ok = __all_sync(0xffffffffu,
                                    wait_phase(sm, &sm.acc_full[buf], (grp / kBufs) & 1));
                    if (!ok) return;
                    tc_fence_after();
                    read_out<kBase, decltype(G)::value>(base + buf * kRows, t);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.acc_empty[buf]);
                    ++grp;
                };
                group(std::integral_constant<int, 0>{});
                group(std::integral_constant<int, 1>{});
                group(std::integral_constant<int, 2>{});
                group(std::integral_constant<int, 3>{});
                group(std::integral_constant<int, 4>{});
                group(std::integral_constant<int, 5>{});
                group(std::integral_constant<int, 6>{});
                if (ok && kb % Stages == Stages - 1) {
                    constexpr unsigned long long bias = stage_bias<kBase>() * Stages;
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        out[(size_t)c * kRows] = make_longlong2((long long)(t[2 * c] - bias),
                                                                (long long)(t[2 * c + 1] - bias));
                        t[2 * c] = t[2 * c + 1] = 0ull;
                    }
                    out += kRows * kRows / 2;
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x == 0 && sm.abort) *gate = 1;  // C is not whole: the sweep solves the set
    if (warp == 0) tc_free(tmem, 512);
}

// ---------------------------------------------------------------------------
// Pair pass in FP64: 16 CTAs per tile, a thread per row and 4 columns, two at a
// time (ten tiles at N = 512 need that many to fill the chip): C^r = sum over the
// slab's blocks of the scaled 64-bit sums, G = sum_r C^r A_r, then rho e.G e or (rho / r)(2 G e - 5 (e.G e) e).
// ---------------------------------------------------------------------------
constexpr int kPairCols = 4;  // columns per thread

template <bool Grad>
__global__ void __launch_bounds__(256)
pair64_kernel(const double4_32a* __restrict__ x4, const float4* __restrict__ xh,
              const float4* __restrict__ xl, int N, int n_pad, int n_blk, int shift, int t0,
              const float* __restrict__ tau, const int* __restrict__ ea,
              const longlong2* __restrict__ C, double sign, double* __restrict__ out,
              double* __restrict__ lo, const int* __restrict__ gate) {
    if (*gate) return;
    constexpr int kVals = Grad ? 3 : 1;
    __shared__ double coef[kForms][5];
    __shared__ double red[8][kPairCols][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int I, J;
    decode_tile(t0 + blockIdx.x, I, J);
    const int row = (warp & 3) * 32 + lane;
    const int c0 = (blockIdx.y * 2 + (warp >> 2)) * kPairCols;
    const int i = I * kRows + row;
    if (threadIdx.x < kForms * 5)
        coef[threadIdx.x / 5][threadIdx.x % 5] = kFormA[threadIdx.x / 5][threadIdx.x % 5];
    __syncthreads();
    if (J * kRows + c0 + kPairCols - 1 <= I * kRows + (warp & 3) * 32) return;  // no j > i (warp-uniform)
    const bool iv = i < N;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 ih = iv ? xh[i] : z4, il = iv ? xl[i] : z4;
    const float ti = iv ? tau[i] : 0.f;
    const double4_32a xi = iv ? x4[i] : make_double4_32a(0, 0, 0, 0);
    double sum[kVals];
#pragma unroll
    for (int d = 0; d < kVals; ++d) sum[d] = 0.0;
    double col[kVals][kPairCols];
#pragma unroll
    for (int cc = 0; cc < kPairCols; cc += 2) {
        const int j0 = J * kRows + c0 + cc;
        double G[2][5];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int m = 0; m < 5; ++m) G[q][m] = 0.0;
        bool on[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int j = j0 + q;
            on[q] = iv && j < N && j > i;
            if (on[q]) {
                const float s = pair_d2_hilo(ih, il, xh[j], xl[j]);
                on[q] = s < INFINITY && !mbm_is_near(s, ti, tau[j]);
            }
        }
        if (on[0] || on[1]) {
            const longlong2* p = C + (size_t)blockIdx.x * kForms * n_blk * (kRows * kRows / 2) +
                                 (size_t)((c0 + cc) / 2) * kRows + row;
            for (int r = 0; r < kForms; ++r) {
                double x0 = 0.0, x1 = 0.0;
                for (int b = 0; b < n_blk; ++b) {
                    const longlong2 v =
                        __ldcs(p + (size_t)(r * n_blk + b) * (kRows * kRows / 2));
                    const int e = -shift - ea[(size_t)b * n_pad + i];
                    x0 = fma((double)v.x, pow2d(e - ea[(size_t)b * n_pad + j0]), x0);
                    x1 = fma((double)v.y, pow2d(e - ea[(size_t)b * n_pad + j0 + 1]), x1);
                }
#pragma unroll
                for (int m = 0; m < 5; ++m) {
                    G[0][m] = fma(coef[r][m], x0, G[0][m]);
                    G[1][m] = fma(coef[r][m], x1, G[1][m]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            double val[kVals];
#pragma unroll
            for (int d = 0; d < kVals; ++d) val[d] = 0.0;
            if (on[q]) {
                const double4_32a xj = x4[j0 + q];
                const double dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
                const double y = rsqrt(dx * dx + dy * dy + dz * dz), rho = y * y * y;
                const double ex = dx * y, ey = dy * y, ez = dz * y;
                const double gx = G[q][0] * ex + G[q][2] * ey + G[q][3] * ez;
                const double gy = G[q][2] * ex + G[q][1] * ey + G[q][4] * ez;
                const double gz = G[q][3] * ex + G[q][4] * ey - (G[q][0] + G[q][1]) * ez;
                const double ege = ex * gx + ey * gy + ez * gz;
                if constexpr (Grad) {
                    const double k = rho * y, u = -5.0 * ege;
                    val[0] = k * (2.0 * gx + u * ex);
                    val[1] = k * (2.0 * gy + u * ey);
                    val[2] = k * (2.0 * gz + u * ez);
                } else {
                    val[0] = 0.5 * rho * ege;
                }
            }
#pragma unroll
            for (int d = 0; d < kVals; ++d) {
                sum[d] += val[d];
                col[d][cc + q] = val[d];
            }
        }
    }
    const int j = J * kRows + c0 + (lane & 3);
#pragma unroll
    for (int d = 0; d < kVals; ++d) {
        __syncwarp();
#pragma unroll
        for (int cc = 0; cc < kPairCols; ++cc) red[warp][cc][lane] = col[d][cc];
        __syncwarp();
        double t = 0.0;  // 4 of the column's 32 rows
#pragma unroll
        for (int q = 0; q < 4; ++q) t += red[warp][lane & 3][(lane >> 2) * 4 + q];
        for (int o = 16; o >= 4; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane < 4 && j < N && t != 0.0) {
            if constexpr (Grad) atomicAdd(&out[3 * (size_t)j + d], sign * t);
            else atomic_add_carried(&out[j], &lo[j], t);
        }
        if (iv && sum[d] != 0.0) {
            if constexpr (Grad) atomicAdd(&out[3 * (size_t)i + d], -sign * sum[d]);
            else atomic_add_carried(&out[i], &lo[i], sum[d]);
        }
    }
}

size_t up256(size_t b) { return mbm_align_up(b, 256); }

}  // namespace

// r^2 of the closest pair that the two FP32 parts of a point resolve, in the frame.
constexpr float kMinDist2 = 3.637979e-12f;  // 2^-38

// Largest N that was measured (7 s a solve).
constexpr int64_t kMaxN64 = 24576;
// Smallest N whose near list looks for tight groups: what a group costs the others grows
// with N (1.3e-13 of sum|grad phi| at N = 3 000, 1.2e-12 at 8 000), the search takes three
// launches.
constexpr int64_t kGroupsMinN = 2048;

// Scratch layout of one solve. The digit table takes 140 bytes per pair of
// particles (58 GB at N = 20 000), so the columns k go in slabs whose table stays
// below kTableMost: C^r is a sum over k and so is all that follows. A slab more is one
// more pair pass (46 ms of FP64 at N = 20 000, against 0.6 s of its contraction).
constexpr size_t kTableMost = (size_t)6 << 30, kSumsMost = (size_t)3 << 30;

struct Plan64 {
    int stages = 8, cols = 0;               // of a block
    int nb = 0, n_blk = 0, n_pad = 0;       // row blocks; column blocks in all
    int slab = 0, tiles = 0, batch = 0;     // column blocks per slab; tiles per pair pass
    size_t table = 0, per_tile = 0, total = 0;
};

static Plan64 plan64(int64_t N, size_t cap) {
    Plan64 p;
    // blocks of 512 columns halve the 64-bit sums to convert; 256 waste less at small N
    p.stages = N > 2048 ? 16 : 8;
    p.cols = p.stages * kBK;
    p.nb = (int)((N + kRows - 1) / kRows);
    p.n_blk = (int)((N + p.cols - 1) / p.cols);
    p.n_pad = (int)mbm_align_up((size_t)p.nb * kRows, 256);
    p.tiles = p.nb * (p.nb + 1) / 2;
    const size_t blk_table = (size_t)kForms * p.nb * p.stages * kStageBytes;
    const size_t blk_sums = (size_t)kForms * kRows * kRows * 8;
    const size_t fixed = 256 + up256((size_t)N * 16) * 2 + up256((size_t)N * 32) +
                         up256((size_t)N * 8) + mbm_near_bytes(N) +
                         up256((size_t)p.n_pad * 4 * p.n_blk) + 4096;
    if (cap < fixed + blk_table + blk_sums) return Plan64{};
    const size_t room = cap - fixed;
    const size_t most = std::min<size_t>(
        p.n_blk, std::min(std::max<size_t>(1, kTableMost / blk_table), room / (blk_table + blk_sums)));
    const int slabs = (int)((p.n_blk + most - 1) / most);
    p.slab = (p.n_blk + slabs - 1) / slabs;  // even slabs
    p.table = blk_table * p.slab;
    p.per_tile = blk_sums * p.slab;
    const size_t sums = std::min(kSumsMost, room - p.table);
    p.batch = (int)std::max<size_t>(1, std::min<size_t>(p.tiles, sums / p.per_tile));
    p.total = fixed + p.table + p.per_tile * p.batch;
    return p;
}

size_t mbm_contract64_bytes(int64_t N, bool forces) {
    if (N < (forces ? kContract64MinForces : kContract64MinPhi) || N > kMaxN64) return 0;
    return plan64(N, (size_t)1 << 60).total;
}

mbm_status mbm_contract64(mbm_ctx* ctx, const double* X, int64_t N, int what, double sign,
                          double* out, cudaStream_t s, bool* done, MbmGate64* gate_out) {
    *done = false;
    if (N > kMaxN64) return MBM_OK;
    size_t cap = (size_t)1 << 60;
    if (ctx->budget) {
        const size_t others = ctx->in_use - ctx->scratch_bytes;
        cap = ctx->budget > others ? ctx->budget - others : 0;
    }
    const Plan64 p = plan64(N, cap);
    if (!p.slab) return MBM_OK;
    const int nb = p.nb, n_pad = p.n_pad;
    const mbm_status rs = mbm_scratch_reserve(ctx, p.total);
    if (rs != MBM_OK) {
        if (rs != MBM_EBUDGET && rs != MBM_ENOMEM) return rs;
        cudaGetLastError();  // no room: the FP64 sweep needs less
        return MBM_OK;
    }
    char* q = static_cast<char*>(ctx->scratch);
    auto take = [&](size_t bytes) {
        char* r = q;
        q += up256(bytes);
        return r;
    };
    int* gate = reinterpret_cast<int*>(take(256));
    auto* counter = reinterpret_cast<unsigned long long*>(gate + 16);
    auto* frame = reinterpret_cast<MbmFrame*>(gate + 32);
    auto* x4 = reinterpret_cast<double4_32a*>(take((size_t)N * 32));
    auto* xh = reinterpret_cast<float4*>(take((size_t)N * 16));
    auto* xl = reinterpret_cast<float4*>(take((size_t)N * 16));
    auto* lo = reinterpret_cast<double*>(take((size_t)N * 8));
    char* near_mem = take(mbm_near_bytes(N));
    int* ea = reinterpret_cast<int*>(take((size_t)n_pad * 4 * p.n_blk));
    auto* T = reinterpret_cast<unsigned char*>(take(p.table));
    auto* C = reinterpret_cast<longlong2*>(take(p.per_tile * p.batch));

    const bool grad = what != MBM_CONTRACT_PHI;
    MBM_CUDA_TRY(cudaMemsetAsync(ctx->d_flags, 0, sizeof(int), s));
    MBM_CUDA_TRY(cudaMemsetAsync(gate, 0, 256, s));
    // potentials, whose terms cancel, carry what their additions round off
    const MbmOut res{out, N * (grad ? 3 : 1), grad ? 10 : 9, grad ? nullptr : lo};
    MBM_CUDA_TRY(launch_frame(X, N, nullptr, frame, xh, xl, x4, nullptr, res, gate, ctx->d_flags,
                              s));
    auto kernel = p.stages == 8 ? contract64_kernel<8> : contract64_kernel<16>;
    MBM_CUDA_TRY(cudaFuncSetAttribute((const void*)kernel,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sizeof(ContractSmem)));
    mbm_time_begin(ctx, s);
    MbmNear near;
    near.X = X;
    near.min_d2 = kMinDist2;
    near.excess = counter + 1;
    near.groups = N > kGroupsMinN;
    MBM_CUDA_TRY(launch_near_list(xh, xl, N, near_mem, gate, ctx->d_flags, &near, s));
    exponent_kernel<<<dim3(n_pad / 256, p.n_blk), 256, 0, s>>>(xh, xl, (int)N, p.cols, near.tau,
                                                              n_pad, ea, gate);
    for (int b0 = 0; b0 < p.n_blk; b0 += p.slab) {
        const int n_blk = std::min(p.slab, p.n_blk - b0), nkb = n_blk * p.stages;
        digit_kernel<<<dim3(nb, nkb, kBK / 8), kRows, 0, s>>>(x4, xh, xl, (int)N, near.tau, n_pad,
                                                              nb, b0 * p.stages, nkb, p.stages, ea,
                                                              T, gate);
        MBM_CUDA_TRY(cudaGetLastError());
        for (int t0 = 0; t0 < p.tiles; t0 += p.batch) {
            const int nt = std::min(p.batch, p.tiles - t0);
            kernel<<<std::min(nt * kForms, std::max(1, ctx->num_sms)), kThreads,
                     sizeof(ContractSmem), s>>>(T, nb, nkb, t0, nt, C, gate, ctx->expire_waits);
            auto pass = grad ? pair64_kernel<true> : pair64_kernel<false>;
            pass<<<dim3(nt, kRows / (2 * kPairCols)), 256, 0, s>>>(
                x4, xh, xl, (int)N, n_pad, n_blk, base_shift(p.stages), t0, near.tau,
                ea + (size_t)b0 * n_pad, C, sign, out, lo, gate);
            MBM_CUDA_TRY(cudaGetLastError());
        }
    }
    MBM_CUDA_TRY(launch_near_triples(xh, xl, x4, N, near, nullptr,
                                     grad ? MBM_NEAR_GRAD : MBM_NEAR_PHI, sign, out, lo,
                                     ctx->num_sms, gate, s));
    MBM_CUDA_TRY(launch_unframe(X, N, frame, xh, xl, x4, res, gate, s));
    gate_out->gate = gate;
    gate_out->counter = counter;
    gate_out->x4 = x4;
    *done = true;
    return MBM_OK;
}
