// Exhaustive potentials, forces and VJPs as a contraction on the tensor cores.
//
// Identity. For three points the direction-cosine form is
//   phi = rho_ij rho_ik rho_jk (1 - 3 Tr(E_ij E_jk E_ki)),  E = e e^T, rho = r^-3,
// and because the three edges of a triangle are coplanar (1 + 2 Tr(EEE) = the
// sum of the squared cosines), phi = -9 Tr(B_ij B_jk B_ki) with B = rho (E - I/3).
// Tr(B^3) is a cubic form in the five components of a symmetric traceless
// matrix; it is a sum of ten cubes of linear forms, -9 Tr(B^3) = sum_r l_r(B)^3,
// so with L^r_ij = l_r(B_ij) (symmetric, zero diagonal: the triples with equal
// members drop out by themselves) and C^r = L^r L^r:
//   Phi_i       = (1/2) sum_j sum_r L^r_ij C^r_ij,
//   dE / dx_j   = sum_{i} sum_r C^r_ij grad_j L^r_ij      (E = (1/3) sum Phi),
//   VJP of Phi  : C^r_ij replaced by (g_i + g_j) C^r_ij + sum_k g_k L^r_ik L^r_jk.
// The ten matrix products are the only cubic work: 30 multiply-adds per
// unordered triple (each of its three pairs), for a potential or for forces.
// The forms' coefficients were found by least squares over ten real cubes
// (nine do not suffice numerically) and polished to 40 digits; among the
// solutions the one of least sum_r |l_r|^6 is taken, which keeps the cancellation
// between the ten terms small.
//
// Precision. Each particle's three nearest neighbours are left out of the matrices
// and the triples that hold such a pair are summed term by term (near.cu): they
// carry 86-96 % of a potential and all of its large terms. The rest is smooth. A
// row of L is cut against a power of two a per row and 256 columns, |a L| <= 2^15,
// into h = fp16(a L) and l = fp16(2^11 (a L - h)): 22 bits. The tensor cores
// multiply fp16 exactly and add in FP32 with truncation (8e-8 of a sum per 16
// terms, measured), so h h is read out every 64 columns, h l + l h (2^-11 smaller)
// every 256, and both are added in FP32, round to nearest. l l is left out. Median
// error against 64 bits at N = 2 600 (in brackets the FP32 triple sweep):
// potentials 1.7e-8 (5.6e-8) on uniform sets, 2.5e-8 (1.0e-7) in the unit cube,
// 2.8e-8 (9.7e-8) on mixtures; forces 1.6e-7 (3.4e-7), 1.9e-7 (3.3e-7), 2.1e-7
// (3.8e-7). Without the split, three pieces and eight products were needed for the
// sweep's accuracy: forces of 8 192 particles took 29 ms against 16.
// Range. FP32 carries everything but the sums, down to products of three edges
// (r^6) and of r^-10, so the points are brought to a common unit first (frame.h):
// |x - x_0| < 2^11, and r >= 2^-11.5 there keeps a triple's r^-10 within 2^-128 and
// 2^115. The two FP32 parts of a point resolve such distances to 2^-25.
//
// A set with a closer pair, a set with more than 16 near pairs per particle (many
// equal distances), and one where a bounded wait ran out, are left to the FP32 sweep
// behind, decided on the device (gate); that sweep returns at once otherwise.
//
// Kernels: near pairs (near.cu); block maxima -> scales; piece table (stored in
// the operand layout, so a stage is two kinds of bulk copies and no tensor map);
// contraction (tcgen05.mma 128 x 256, warp-specialised, persistent); pair pass
// over the tiles' C; near triples. Large N runs in slabs of columns k and batches
// of tiles; all sums are linear in both.
#include <algorithm>
#include <cuda_fp16.h>

#include "bulk_copy.cuh"
#include "contract.h"
#include "device_math.cuh"
#include "forms.cuh"
#include "frame.h"
#include "near.h"
#include "tcgen05.cuh"

namespace {

constexpr int kPieces = 2;
constexpr int kBlk = 256;      // rows per table block, and columns that share a scale
constexpr int kBM = 128;       // tile rows
constexpr int kBN = 256;       // tile columns
constexpr int kBK = 32;        // columns k per pipeline stage
constexpr int kKbPerBlk = kBlk / kBK;
constexpr int kWin = 64;       // columns k per read-out of h h
constexpr int kKbPerWin = kWin / kBK;
constexpr int kWinPerBlk = kBlk / kWin;
constexpr int kPieceB = kBN * kBK * 2;  // 16 KB: one piece of 256 rows x 32 columns
constexpr int kPieceA = kBM * kBK * 2;
constexpr int kStages = 4;
// Factor slots: a block's factors are copied when at most half a block of MMAs is
// in flight, which waited for the accumulators of the block before.
constexpr int kFactorSlots = 4;
constexpr float kLowScale = 1.0f / 2048.0f;
constexpr int kEpiWarps = 16;
constexpr int kThreads = (kEpiWarps + 2) * 32;
constexpr int kGroup = 8;  // J tiles walked together: their rows and 19 I tiles stay in L2
constexpr long long kWaitLimit = 4000000000LL;

__device__ __forceinline__ float pow2f(int e) {  // 2^e, 0 below the normal range
    return e < -126 ? 0.f : __int_as_float((min(e, 127) + 127) << 23);
}

// ---------------------------------------------------------------------------
// Scales. ea[b][i]: exponent of a(i, b), the power of two with |a l| <= 2^15 over
// the 256 columns k of block b without near pairs (times |g_k| for the weighted
// table). A CTA takes 256 rows and one block, its columns in shared memory.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlk)
scale_kernel(const float4* __restrict__ xh, const float4* __restrict__ xl, int N, int b0,
             const float* __restrict__ tau, const double* __restrict__ g, int n_pad,
             int* __restrict__ ea, int* __restrict__ row_ea, const int* __restrict__ gate) {
    if (*gate) return;
    __shared__ float4 kh[kBlk], kl[kBlk];
    __shared__ float kg[kBlk], kt[kBlk];
    const int b = blockIdx.y, k0 = (b0 + b) * kBlk;
    const int i = blockIdx.x * kBlk + threadIdx.x;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const int kk = k0 + threadIdx.x;
    kh[threadIdx.x] = kk < N ? xh[kk] : z4;
    kl[threadIdx.x] = kk < N ? xl[kk] : z4;
    kt[threadIdx.x] = kk < N ? tau[kk] : 0.f;
    kg[threadIdx.x] = g && kk < N ? fabsf((float)g[kk]) : 1.f;
    __syncthreads();
    const float4 ih = i < N ? xh[i] : z4, il = i < N ? xl[i] : z4;
    const float ti = i < N ? tau[i] : 0.f;
    const int cnt = min(kBlk, N - k0);
    float best = 0.f;  // largest rho (or |g| rho) of the block
    if (i < N) {
        float smin = INFINITY;
        for (int q = 0; q < cnt; ++q) {
            const float s = pair_d2_hilo(ih, il, kh[q], kl[q]);
            // (the particle itself has s = 0 <= tau)
            if (mbm_is_near(s, ti, kt[q]) || !(s < INFINITY)) continue;
            if (g) {
                const float y = rsqrtf(s);
                best = fmaxf(best, kg[q] * (y * y * y));
            } else {
                smin = fminf(smin, s);
            }
        }
        if (!g && smin < INFINITY) {
            const float y = rsqrtf(smin);
            best = y * y * y;
        }
    }
    int e = 127;  // nothing in this block
    if (best > 0.f && best < INFINITY) e = 14 - ilogbf(best * (kFormMax * 1.0001f));
    if (best > 0.f) e = max(-120, min(126, e));
    ea[(size_t)b * n_pad + i] = e;
    if (i < N) atomicMin(&row_ea[i], e);
}

// Smallest row exponent (the reference of the relative scales).
__global__ void ref_kernel(const int* __restrict__ row_ea, int N, int* __restrict__ ref) {
    int m = 126;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x)
        m = min(m, row_ea[i]);
    m = __reduce_min_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMin(ref, m);
}

// f[b][i] = 2^(row exponent - block exponent) <= 1.
__global__ void __launch_bounds__(kBlk)
factor_kernel(const int* __restrict__ ea, const int* __restrict__ row_ea, int n_pad, int N,
              float* __restrict__ f) {
    const int i = blockIdx.x * kBlk + threadIdx.x;
    const size_t o = (size_t)blockIdx.y * n_pad + i;
    const int e = ea[o];
    f[o] = i < N && e < 127 ? pow2f(row_ea[i] - e) : 0.f;
}

// ---------------------------------------------------------------------------
// Piece table, in the contraction's operand layout: T[r][row block][kb][piece]
// is 256 rows x 32 columns as core matrices of 8 rows x 8 columns (128 bytes),
// [row group][column group][row][column]. A CTA writes all forms and pieces of
// 256 rows x 8 columns; a thread owns a row (16-byte stores, 128 contiguous bytes
// per 8 rows). FP32 pair terms: what they lose (2^-23) is weighed by the
// contraction's small share of a result; two-term numbers took 2.4 times as long.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlk)
table_kernel(const float4* __restrict__ xh, const float4* __restrict__ xl, int N, int b0,
             const float* __restrict__ tau, const double* __restrict__ g, int n_pad, int nb,
             int nkb, const int* __restrict__ ea, unsigned char* __restrict__ T,
             const int* __restrict__ gate) {
    if (*gate) return;
    __shared__ float coef[kForms][5];
    __shared__ float4 kh[8], kl[8];
    __shared__ float kg[8], kt[8];
    const int rb = blockIdx.x, kb = blockIdx.y, k8 = blockIdx.z;
    const int k0 = b0 * kBlk + kb * kBK + k8 * 8;
    const int row = threadIdx.x, i = rb * kBlk + row;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (threadIdx.x < kForms * 5)
        coef[threadIdx.x / 5][threadIdx.x % 5] = (float)form_coef(threadIdx.x / 5, threadIdx.x % 5);
    if (threadIdx.x < 8) {
        const int k = k0 + threadIdx.x;
        kh[threadIdx.x] = k < N ? xh[k] : z4;
        kl[threadIdx.x] = k < N ? xl[k] : z4;
        kt[threadIdx.x] = k < N ? tau[k] : 0.f;
        kg[threadIdx.x] = g && k < N ? (float)g[k] : 1.f;
    }
    __syncthreads();
    const float4 ih = i < N ? xh[i] : z4, il = i < N ? xl[i] : z4;
    // two exact factors: one alone may pass the FP32 range
    const float ti = i < N ? tau[i] : 0.f;
    const int e = ea[(size_t)(kb / kKbPerBlk) * n_pad + i];
    const int e1 = e / 2;
    const float a1 = pow2f(e1), a2 = pow2f(e - e1);
    float v[8][5];  // (Exx - Ezz, Eyy - Ezz, Exy, Exz, Eyz) a rho
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const float dx = (kh[q].x - ih.x) + (kl[q].x - il.x);
        const float dy = (kh[q].y - ih.y) + (kl[q].y - il.y);
        const float dz = (kh[q].z - ih.z) + (kl[q].z - il.z);
        const float s = pair_d2_hilo(ih, il, kh[q], kl[q]);
        const bool ok = i < N && k0 + q < N && k0 + q != i && s < INFINITY &&
                        !mbm_is_near(s, ti, kt[q]);
        float y = rsqrtf(s);
        y = fmaf(0.5f * y, fmaf(-s * y, y, 1.0f), y);
        const float ex = dx * y, ey = dy * y, ez = dz * y;
        const float rho = (y * y * y) * kg[q] * a1 * a2;
        const float tx = ex * rho, ty = ey * rho, tz = ez * rho, zz = ez * tz;
        v[q][0] = ok ? fmaf(ex, tx, -zz) : 0.f;
        v[q][1] = ok ? fmaf(ey, ty, -zz) : 0.f;
        v[q][2] = ok ? ex * ty : 0.f;
        v[q][3] = ok ? ex * tz : 0.f;
        v[q][4] = ok ? ey * tz : 0.f;
    }
    const size_t off = (size_t)(row >> 3) * 512 + k8 * 128 + (row & 7) * 16;
#pragma unroll 1
    for (int r = 0; r < kForms; ++r) {
        __align__(16) __half h8[8], l8[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            float x = coef[r][0] * v[q][0];
#pragma unroll
            for (int m = 1; m < 5; ++m) x = fmaf(coef[r][m], v[q][m], x);
            h8[q] = __float2half_rn(x);
            l8[q] = __float2half_rn((x - __half2float(h8[q])) * 2048.0f);
        }
        unsigned char* dst =
            T + (((size_t)r * nb + rb) * nkb + kb) * (size_t)(kPieces * kPieceB) + off;
        *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(h8);
        *reinterpret_cast<uint4*>(dst + kPieceB) = *reinterpret_cast<const uint4*>(l8);
    }
}

// ---------------------------------------------------------------------------
// Contraction.
// ---------------------------------------------------------------------------
// Tile t -> (I in 128-row blocks, J in 256-row blocks) over the tiles that
// hold a pair i < j, J in groups of kGroup and I outermost inside a group, so
// that tiles running together share rows in L2. nb (nb + 1) tiles in all.
__device__ __forceinline__ void decode_tile(int t, int nb, int& I, int& J) {
    for (int g = 0;; ++g) {
        const int w = min(kGroup, nb - g * kGroup);
        const int rect = 2 * g * kGroup * w, cnt = rect + w * (w + 1);
        if (t >= cnt) {
            t -= cnt;
            continue;
        }
        if (t < rect) {
            I = t / w;
            J = g * kGroup + t % w;
            return;
        }
        t -= rect;
        for (int row = 0;; ++row) {  // row 2 g kGroup + row has w - row / 2 tiles
            const int c = w - row / 2;
            if (t < c) {
                I = 2 * g * kGroup + row;
                J = g * kGroup + row / 2 + t;
                return;
            }
            t -= c;
        }
    }
}

struct ContractSmem {
    unsigned char a[kStages][kPieces * kPieceA];
    unsigned char b[kStages][kPieces * kPieceB];
    float fj[kFactorSlots][kBN], fi[kFactorSlots][kBM];  // scale factors of a window
    unsigned long long factors[kFactorSlots];
    unsigned long long full[kStages], empty[kStages];
    unsigned long long acc_full[2], acc_empty[2];
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

// Adds one accumulator window (64 columns of the warp's 32 rows), scaled.
__device__ __forceinline__ void drain(unsigned addr, const float* fj, float2 fi,
                                      float2 (&acc)[32]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float v[16];
        tc_ld16(addr + 16 * c, v);
        tc_wait_ld();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 w = reinterpret_cast<const float4*>(fj + 16 * c)[q];
            float2& a0 = acc[8 * c + 2 * q];
            float2& a1 = acc[8 * c + 2 * q + 1];
            a0 = f2_fma(f2_mul(make_float2(v[4 * q], v[4 * q + 1]), fi), make_float2(w.x, w.y), a0);
            a1 = f2_fma(f2_mul(make_float2(v[4 * q + 2], v[4 * q + 3]), fi),
                        make_float2(w.z, w.w), a1);
        }
    }
}

// C[tile][r][column / 4][row][4] = sum over the slab's k of A_ik B_jk, in units
// of the row scales. One CTA per SM, items (form, tile) dealt round robin,
// forms outermost. Warps 0-15: read-outs to registers, C at the end; warp 16: bulk
// copies (48 KB stages of 32 columns); warp 17: MMAs. The accumulators fill
// TMEM: 256 columns for h h and 256 for h l + l h; each is drained while the
// other is computed.
__global__ void __launch_bounds__(kThreads, 1)
contract_kernel(const unsigned char* __restrict__ TA, const unsigned char* __restrict__ TB,
                const float* __restrict__ fA, const float* __restrict__ fB, int n_pad, int nb,
                int nkb, int t0, int nt, float* __restrict__ C, int* gate, int expire) {
    // (a CTA of this launch may set it meanwhile: one answer for all threads)
    if (__syncthreads_or(*gate)) return;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    ContractSmem& sm = *reinterpret_cast<ContractSmem*>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&sm.full[s], 1);
            mbar_init(&sm.empty[s], 1);
        }
        for (int q = 0; q < kFactorSlots; ++q) mbar_init(&sm.factors[q], 1);
        for (int a = 0; a < 2; ++a) {
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
    const size_t stage_src = (size_t)kPieces * kPieceB;
    if (warp == kEpiWarps) {
        if (lane == 0) {
            unsigned it = 0, win = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                const int r = item / nt;
                int I, J;
                decode_tile(t0 + item % nt, nb, I, J);
                const unsigned char* pa =
                    TA + ((size_t)r * nb + (I >> 1)) * nkb * stage_src + (I & 1) * kPieceA;
                const unsigned char* pb = TB + ((size_t)r * nb + J) * nkb * stage_src;
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % kStages;
                    if (it >= kStages &&
                        !wait_phase(sm, &sm.empty[s], (it / kStages - 1) & 1)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(&sm.full[s], kPieces * (kPieceA + kPieceB));
                    for (int p = 0; p < kPieces; ++p)
                        bulk_copy_g2s(sm.a[s] + p * kPieceA, pa + kb * stage_src + p * kPieceB,
                                      kPieceA, &sm.full[s]);
                    bulk_copy_g2s(sm.b[s], pb + kb * stage_src, kPieces * kPieceB, &sm.full[s]);
                    if (kb % kKbPerBlk == 0) {
                        const int q = win++ % kFactorSlots;
                        const size_t w = (size_t)(kb / kKbPerBlk) * n_pad;
                        mbar_arrive_expect_tx(&sm.factors[q], (kBM + kBN) * sizeof(float));
                        bulk_copy_g2s(sm.fj[q], fB + w + J * kBN, kBN * sizeof(float),
                                      &sm.factors[q]);
                        bulk_copy_g2s(sm.fi[q], fA + w + I * kBM, kBM * sizeof(float),
                                      &sm.factors[q]);
                    }
                }
            }
            // copies in flight land before shared memory is released
            for (unsigned q = it > kStages ? it - kStages : 0; q < it; ++q)
                mbar_wait_bounded(&sm.full[q % kStages], (q / kStages) & 1, kWaitLimit);
            for (unsigned q = win > kFactorSlots ? win - kFactorSlots : 0; q < win; ++q)
                mbar_wait_bounded(&sm.factors[q % kFactorSlots], (q / kFactorSlots) & 1, kWaitLimit);
        }
    } else if (warp == kEpiWarps + 1) {
        if (lane == 0) {
            constexpr unsigned idesc = tc_idesc_f16(kBM, kBN);
            unsigned it = 0, win = 0, blk = 0;  // stages, windows and blocks handed over
            bool ok = true;
            // (expire, a switch of tests: this role gives up after its first window)
            const int items = expire ? 0 : n_items, kbs = expire ? kKbPerWin : nkb;
            int item = blockIdx.x;
            do {
                for (int kb = 0; kb < kbs; kb += kKbPerWin, ++win) {
                    const bool first = kb % kKbPerBlk == 0;
                    const bool last = kb % kKbPerBlk == kKbPerBlk - kKbPerWin;
                    if (win && !wait_phase(sm, &sm.acc_empty[0], (win - 1) & 1)) {
                        ok = false;
                        break;
                    }
#pragma unroll 1
                    for (int u = 0; u < kKbPerWin && ok; ++u) {
                        const unsigned q = it + u;
                        if (!wait_phase(sm, &sm.full[q % kStages], (q / kStages) & 1)) ok = false;
                        if (!ok) break;
                        tc_fence_after();
                        const unsigned ab = smem_u32(sm.a[q % kStages]);
                        const unsigned bb = smem_u32(sm.b[q % kStages]);
#pragma unroll
                        for (int k = 0; k < kBK / 16; ++k)
                            tc_mma_f16(tmem, tc_desc(ab + k * 256, 128, 512),
                                       tc_desc(bb + k * 256, 128, 512), idesc, u + k > 0);
                    }
                    if (!ok) break;
                    tc_commit(smem_u32(&sm.acc_full[0]));
                    if (first && blk && !wait_phase(sm, &sm.acc_empty[1], (blk - 1) & 1)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
#pragma unroll 1
                    for (int u = 0; u < kKbPerWin; ++u, ++it) {
                        const unsigned ab = smem_u32(sm.a[it % kStages]);
                        const unsigned bb = smem_u32(sm.b[it % kStages]);
#pragma unroll
                        for (int k = 0; k < kBK / 16; ++k) {
                            tc_mma_f16(tmem + kBN, tc_desc(ab + k * 256, 128, 512),
                                       tc_desc(bb + kPieceB + k * 256, 128, 512), idesc,
                                       !(first && u + k == 0));
                            tc_mma_f16(tmem + kBN, tc_desc(ab + kPieceA + k * 256, 128, 512),
                                       tc_desc(bb + k * 256, 128, 512), idesc, true);
                        }
                        if (last && u == kKbPerWin - 1) {
                            tc_commit(smem_u32(&sm.acc_full[1]));
                            ++blk;
                        }
                        tc_commit(smem_u32(&sm.empty[it % kStages]));
                    }
                }
                item += gridDim.x;
            } while (item < items && ok);
            if (expire) sm.abort = 1;
            // MMAs in flight end before TMEM and shared memory are released, also those
            // that an expired wait left without a commit
            tc_commit(smem_u32(&sm.done));
            mbar_wait_bounded(&sm.done, 0, kWaitLimit);
        }
    } else {
        // rows 32 (warp % 4) + lane of the tile, columns 64 (warp / 4) + 0..63
        const int row = (warp & 3) * 32 + lane, col = (warp >> 2) * 64;
        const unsigned base = tmem + ((unsigned)(warp & 3) << 21) + col;
        unsigned win = 0, blk = 0;
        bool ok = true;
        // waits for accumulator `a`, adds it and hands it back
        auto take = [&](int a, unsigned phase, const float* fj, float fi, float2(&acc)[32]) {
            if (!__all_sync(0xffffffffu, wait_phase(sm, &sm.acc_full[a], phase & 1))) return false;
            tc_fence_after();
            drain(base + a * kBN, fj, f2_splat(fi), acc);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.acc_empty[a]);
            return true;
        };
        for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
            float2 acc[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) acc[c] = make_float2(0.f, 0.f);
            for (int b = 0; b < nkb / kKbPerBlk && ok; ++b, ++blk) {
                const unsigned slot = blk % kFactorSlots;
                ok = __all_sync(0xffffffffu,
                                wait_phase(sm, &sm.factors[slot], (blk / kFactorSlots) & 1));
                const float fi = sm.fi[slot][row];
                const float* fj = &sm.fj[slot][col];
                for (int w = 0; w < kWinPerBlk && ok; ++w, ++win) ok = take(0, win, fj, fi, acc);
                if (ok) ok = take(1, blk, fj, fi * kLowScale, acc);
            }
            if (ok) {
                float4* out = reinterpret_cast<float4*>(C) +
                              (size_t)((item % nt) * kForms + item / nt) * (kBM * kBN / 4) +
                              (size_t)(col / 4) * kBM + row;
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    out[c * kBM] = make_float4(acc[2 * c].x, acc[2 * c].y, acc[2 * c + 1].x,
                                               acc[2 * c + 1].y);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x == 0 && sm.abort) *gate = 1;  // C is not whole
    if (warp == 0) tc_free(tmem, 512);
}

// ---------------------------------------------------------------------------
// Pair pass: four CTAs per tile, a thread per row and 32 columns, four columns
// at a time: G = sum_r C^r A_r (five components), then the pair's potential
// rho e.G e or its gradient (rho / r)(2 G e - 5 (e.G e) e). Column sums go
// through a transposed shared buffer. Near pairs have no entry in L.
// ---------------------------------------------------------------------------
enum : int { kPhi = 0, kForce = 1, kVjp = 2 };

constexpr int kStep = 16;      // columns between two column sums
constexpr int kPairCols = 64;  // columns of a tile per CTA: 20 tiles alone left SMs idle

template <int Mode>
__global__ void __launch_bounds__(256)
pair_kernel(const float4* __restrict__ xh, const float4* __restrict__ xl, int N, int nb, int t0,
            const float* __restrict__ tau, const float* __restrict__ C,
            const float* __restrict__ Cg, const double* __restrict__ g,
            const int* __restrict__ row_ea, const int* __restrict__ row_eag,
            const int* __restrict__ ref, double sign, double* __restrict__ out,
            const int* __restrict__ gate) {
    if (*gate) return;
    constexpr int kVals = Mode == kPhi ? 1 : 3;
    __shared__ float4 jh[kBN], jl[kBN];
    __shared__ float wj[kBN], gj[kBN], tj[kBN];
    __shared__ float coef[kForms][5];  // A_r
    __shared__ float red[8][kStep][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int I, J;
    decode_tile(t0 + blockIdx.x, nb, I, J);
    const int row = (warp & 3) * 32 + lane, half = warp >> 2;
    const int i = I * kBM + row;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const int eref = *ref;
    {
        const int j = J * kBN + threadIdx.x;
        jh[threadIdx.x] = j < N ? xh[j] : z4;
        jl[threadIdx.x] = j < N ? xl[j] : z4;
        wj[threadIdx.x] = j < N ? pow2f(eref - row_ea[j]) : 0.f;
        tj[threadIdx.x] = j < N ? tau[j] : 0.f;
        gj[threadIdx.x] = Mode == kVjp && j < N ? (float)g[j] : 0.f;
        if (threadIdx.x < kForms * 5)
            coef[threadIdx.x / 5][threadIdx.x % 5] = (float)kFormA[threadIdx.x / 5][threadIdx.x % 5];
    }
    __syncthreads();
    const bool iv = i < N;
    const float4 ih = iv ? xh[i] : z4, il = iv ? xl[i] : z4;
    const float ti = iv ? tau[i] : 0.f;
    const int ei = iv ? row_ea[i] : 0;
    const float wi = iv ? pow2f(eref - ei) : 0.f;
    const float gi = Mode == kVjp && iv ? (float)g[i] : 0.f;
    // C is in units of A_i A_j; the weighted one in units of Ag_i A_j
    const float cg_scale = Mode == kVjp && iv ? pow2f(ei - row_eag[i]) : 0.f;
    const float rho_scale1 = iv ? pow2f(ei / 2) : 0.f, rho_scale2 = iv ? pow2f(ei - ei / 2) : 0.f;
    const float4* Cp = reinterpret_cast<const float4*>(C) +
                       (size_t)blockIdx.x * kForms * (kBM * kBN / 4) + row;
    const float4* Cq = Mode == kVjp ? reinterpret_cast<const float4*>(Cg) +
                                          (size_t)blockIdx.x * kForms * (kBM * kBN / 4) + row
                                    : nullptr;
    double sum[kVals];
#pragma unroll
    for (int d = 0; d < kVals; ++d) sum[d] = 0.0;
    const int cbeg = blockIdx.y * kPairCols + half * (kPairCols / 2);
    for (int c0 = cbeg; c0 < cbeg + kPairCols / 2; c0 += kStep) {
        // no pair j > i in these columns (warp-uniform)
        if (J * kBN + c0 + kStep - 1 <= I * kBM + (warp & 3) * 32) continue;
        float part[kVals], col[kVals][kStep];
#pragma unroll
        for (int d = 0; d < kVals; ++d) part[d] = 0.f;
#pragma unroll
        for (int cc = 0; cc < kStep; cc += 4) {
            const int c4 = (c0 + cc) >> 2;
            float G[4][5];  // sum_r C^r A_r
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int m = 0; m < 5; ++m) G[q][m] = 0.f;
#pragma unroll
            for (int r = 0; r < kForms; ++r) {
                float4 v = __ldcs(Cp + (size_t)(r * (kBN / 4) + c4) * kBM);
                if (Mode == kVjp) {
                    const float4 u = __ldcs(Cq + (size_t)(r * (kBN / 4) + c4) * kBM);
                    const int c = c0 + cc;
                    v.x = fmaf(v.x, gi + gj[c], u.x * cg_scale);
                    v.y = fmaf(v.y, gi + gj[c + 1], u.y * cg_scale);
                    v.z = fmaf(v.z, gi + gj[c + 2], u.z * cg_scale);
                    v.w = fmaf(v.w, gi + gj[c + 3], u.w * cg_scale);
                }
                const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int m = 0; m < 5; ++m) {
                    const float a = coef[r][m];
#pragma unroll
                    for (int q = 0; q < 4; ++q) G[q][m] = fmaf(a, x[q], G[q][m]);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int c = c0 + cc + q, j = J * kBN + c;
                const bool on = iv && j < N && j > i;
                float val[kVals];
                const float dx = (jh[c].x - ih.x) + (jl[c].x - il.x);
                const float dy = (jh[c].y - ih.y) + (jl[c].y - il.y);
                const float dz = (jh[c].z - ih.z) + (jl[c].z - il.z);
                const float s = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
                float y = rsqrtf(s);
                y = fmaf(0.5f * y, fmaf(-s * y, y, 1.0f), y);
                const bool ok = on && s < INFINITY &&
                                !mbm_is_near(pair_d2_hilo(ih, il, jh[c], jl[c]), ti, tj[c]);
                const float ex = ok ? dx * y : 0.f, ey = ok ? dy * y : 0.f, ez = ok ? dz * y : 0.f;
                const float rho = ok ? (y * y * y) * rho_scale1 * rho_scale2 : 0.f;
                // G is symmetric and traceless: (xx, yy, xy, xz, yz)
                const float gx = fmaf(G[q][3], ez, fmaf(G[q][2], ey, G[q][0] * ex));
                const float gy = fmaf(G[q][4], ez, fmaf(G[q][1], ey, G[q][2] * ex));
                const float gz = fmaf(-(G[q][0] + G[q][1]), ez, fmaf(G[q][4], ey, G[q][3] * ex));
                const float ege = fmaf(ez, gz, fmaf(ey, gy, ex * gx));
                if (Mode == kPhi) {
                    val[0] = rho * ege;
                } else {
                    const float k = ok ? rho * y : 0.f, u = -5.0f * ege;
                    val[0] = k * fmaf(u, ex, 2.0f * gx);
                    val[kVals / 2] = k * fmaf(u, ey, 2.0f * gy);
                    val[kVals - 1] = k * fmaf(u, ez, 2.0f * gz);
                }
#pragma unroll
                for (int d = 0; d < kVals; ++d) {
                    part[d] = fmaf(val[d], wj[c], part[d]);
                    col[d][cc + q] = val[d] * wi * wi;
                }
            }
        }
        // row sums are in units of A_i^2 A_ref, column sums of A_j A_ref^2
#pragma unroll
        for (int d = 0; d < kVals; ++d) sum[d] += (double)part[d];
        const int j = J * kBN + c0 + (lane & 15);
        const double unit = j < N ? ldexp(1.0, -row_ea[j] - 2 * eref) : 0.0;
#pragma unroll
        for (int d = 0; d < kVals; ++d) {
            __syncwarp();
#pragma unroll
            for (int cc = 0; cc < kStep; ++cc) red[warp][cc][lane] = col[d][cc];
            __syncwarp();
            float t = 0.f;  // 16 of the column's 32 rows
#pragma unroll
            for (int q = 0; q < 16; ++q) t += red[warp][lane & 15][(lane >> 4) * 16 + q];
            t += __shfl_xor_sync(0xffffffffu, t, 16);
            if (lane < kStep && j < N && t != 0.f) {
                const double v = unit * (double)t;
                if (Mode == kPhi) atomicAdd(&out[j], 0.5 * v);
                else atomicAdd(&out[3 * (size_t)j + d], sign * v);
            }
        }
    }
    if (iv) {
        const double unit = ldexp(1.0, -2 * ei - eref);
#pragma unroll
        for (int d = 0; d < kVals; ++d) {
            if (sum[d] == 0.0) continue;
            const double v = unit * sum[d];
            if (Mode == kPhi) atomicAdd(&out[i], 0.5 * v);
            else atomicAdd(&out[3 * (size_t)i + d], -sign * v);
        }
    }
}

size_t up256(size_t b) { return mbm_align_up(b, 256); }

// Scratch layout and slab / batch sizes for one solve.
struct Plan {
    int nb = 0, n_pad = 0, n_blk = 0;  // row blocks; scale blocks of k per slab
    int tiles = 0, batch = 0;          // tiles in all, tiles per pair pass
    size_t table = 0, cbuf = 0, total = 0;
};

// Slabs have 4 096 columns (fewer where their table would pass 16 GB), whatever
// the room: sums over a slab are FP32 and results should not depend on what else
// the device holds. Only a context budget that is too small for that shortens them.
// A potential's scratch has room for the pair table of the sweep behind, which solves
// a set that the contraction gives back (the contraction's own buffers are free by
// then), up to kTableRoom (N = 33 000). Beyond, that sweep forms its pair terms itself.
constexpr size_t kTableRoom = (size_t)9 << 30;

Plan make_plan(int64_t N, int what, size_t cap) {
    const bool weighted = what == MBM_CONTRACT_VJP;
    Plan p;
    p.nb = (int)((N + kBlk - 1) / kBlk);
    p.n_pad = p.nb * kBlk;
    p.tiles = p.nb * (p.nb + 1);
    const int copies = weighted ? 2 : 1;
    const size_t per_blk = (size_t)kForms * p.nb * kKbPerBlk * kPieces * kPieceB * copies;
    const size_t per_tile = (size_t)kForms * kBM * kBN * sizeof(float) * copies;
    const size_t fixed =
        up256((size_t)p.n_pad * (weighted ? 40 : 32)) + 8 * (size_t)p.n_pad + mbm_near_bytes(N) +
        131072;
    // per 256 columns of a slab: ea and f (and the weighted ones)
    const size_t per_blk_f = (size_t)p.n_pad * 8 * copies;
    if (cap < fixed) return Plan{};
    const size_t room = cap - fixed;
    int n_blk = (int)std::min<size_t>(std::min(p.nb, 16),
                                      std::max<size_t>(1, ((size_t)16 << 30) / per_blk));
    const size_t c_most = std::min<size_t>((size_t)2 << 30, per_tile * p.tiles);
    const size_t c_least = std::min(c_most, 152 * per_tile);
    while (n_blk > 1 && (per_blk + per_blk_f) * n_blk + c_least > room) --n_blk;
    const size_t table = (per_blk + per_blk_f) * n_blk;
    if (table + per_tile > room) return Plan{};
    const int slabs = (p.nb + n_blk - 1) / n_blk;
    p.n_blk = (p.nb + slabs - 1) / slabs;  // even slabs
    p.batch = (int)(std::min(c_most, room - table) / per_tile);
    p.table = per_blk / copies * p.n_blk;
    p.cbuf = per_tile / copies * p.batch;
    p.total = fixed + (per_blk + per_blk_f) * p.n_blk + per_tile * p.batch;
    if (what == MBM_CONTRACT_PHI) {
        const size_t sweep = fixed + per_blk_f * p.n_blk + pair_table_bytes(N);
        if (pair_table_bytes(N) <= kTableRoom && sweep <= cap) p.total = std::max(p.total, sweep);
    }
    return p;
}

}  // namespace

// r^2 of the closest pair that the contraction takes, in the frame (see Range above).
constexpr float kMinDist2 = 1.1920929e-7f;  // 2^-23

constexpr int64_t kContractMaxN = (int64_t)1 << 20;  // tile numbers fit an int

static Plan plan_for(int64_t N, int what, size_t cap) {
    return N <= kContractMaxN ? make_plan(N, what, cap) : Plan{};
}

size_t mbm_contract_bytes(int64_t N, bool forces) {
    if (N < (forces ? kContractMinForces : kContractMinPhi)) return 0;
    return plan_for(N, forces ? MBM_CONTRACT_FORCES : MBM_CONTRACT_PHI, (size_t)1 << 60).total;
}

mbm_status mbm_contract(mbm_ctx* ctx, const double* X, int64_t N, const double* g, int what,
                        double sign, double* out, cudaStream_t s, bool* done, MbmGate* gate_out) {
    *done = false;
    size_t cap = (size_t)1 << 60;
    if (ctx->budget) {
        const size_t others = ctx->in_use - ctx->scratch_bytes;
        cap = ctx->budget > others ? ctx->budget - others : 0;
    }
    const bool weighted = what == MBM_CONTRACT_VJP;
    const Plan p = plan_for(N, what, cap);
    if (!p.n_blk) return MBM_OK;
    const mbm_status rs = mbm_scratch_reserve(ctx, p.total);
    if (rs != MBM_OK) {
        if (rs != MBM_EBUDGET && rs != MBM_ENOMEM) return rs;
        cudaGetLastError();  // no room: the triple sweep needs less
        return MBM_OK;
    }
    char* q = static_cast<char*>(ctx->scratch);
    auto take = [&](size_t bytes) {
        char* r = q;
        q += up256(bytes);
        return r;
    };
    const int n_pad = p.n_pad;
    auto* head = reinterpret_cast<int*>(take(256));  // 0 gate, 1 reference exponent
    int* gate = head;
    int* ref = head + 1;
    auto* counter = reinterpret_cast<unsigned long long*>(head + 16);
    auto* frame = reinterpret_cast<MbmFrame*>(head + 32);
    auto* xh = reinterpret_cast<float4*>(take((size_t)N * 16));
    auto* xl = reinterpret_cast<float4*>(take((size_t)N * 16));
    auto* gs = weighted ? reinterpret_cast<double*>(take((size_t)N * 8)) : nullptr;
    char* near_mem = take(mbm_near_bytes(N));
    auto* row_ea = reinterpret_cast<int*>(take((size_t)n_pad * 4));
    auto* row_eag = reinterpret_cast<int*>(take((size_t)n_pad * 4));
    const size_t per_b = (size_t)n_pad * 4 * p.n_blk;
    auto* ea = reinterpret_cast<int*>(take(per_b));
    auto* f = reinterpret_cast<float*>(take(per_b));
    int* eag = weighted ? reinterpret_cast<int*>(take(per_b)) : nullptr;
    float* fg = weighted ? reinterpret_cast<float*>(take(per_b)) : nullptr;
    auto* T = reinterpret_cast<unsigned char*>(take(p.table));
    auto* Tg = weighted ? reinterpret_cast<unsigned char*>(take(p.table)) : nullptr;
    auto* C = reinterpret_cast<float*>(take(p.cbuf));
    auto* Cg = weighted ? reinterpret_cast<float*>(take(p.cbuf)) : nullptr;

    const int n_out = what == MBM_CONTRACT_PHI ? 1 : 3;
    MBM_CUDA_TRY(cudaMemsetAsync(ctx->d_flags, 0, sizeof(int), s));
    MBM_CUDA_TRY(cudaMemsetAsync(head, 0, 256, s));
    MBM_CUDA_TRY(cudaMemsetAsync(ref, 0x7f, 4, s));
    MBM_CUDA_TRY(cudaMemsetAsync(row_ea, 0x7f, up256((size_t)n_pad * 4) * 2, s));
    const MbmOut res{out, N * n_out, n_out == 1 ? 9 : 10};
    MBM_CUDA_TRY(launch_frame(X, N, g, frame, xh, xl, nullptr, gs, res, gate, ctx->d_flags, s));

    MBM_CUDA_TRY(cudaFuncSetAttribute((const void*)contract_kernel,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sizeof(ContractSmem)));
    mbm_time_begin(ctx, s);
    MbmNear near;
    near.X = X;
    near.min_d2 = kMinDist2;
    near.excess = counter + 1;
    MBM_CUDA_TRY(launch_near_list(xh, xl, N, near_mem, gate, ctx->d_flags, &near, s));
    // Row exponents come from all columns: with several slabs a first pass over
    // them finds the row exponents before any table is built.
    const int slabs = (p.nb + p.n_blk - 1) / p.n_blk;
    auto scales = [&](int b0, int nblk) {
        const dim3 grid(p.nb, nblk);
        scale_kernel<<<grid, kBlk, 0, s>>>(xh, xl, (int)N, b0, near.tau, nullptr, n_pad, ea,
                                           row_ea, gate);
        if (weighted)
            scale_kernel<<<grid, kBlk, 0, s>>>(xh, xl, (int)N, b0, near.tau, gs, n_pad, eag,
                                               row_eag, gate);
    };
    if (slabs > 1)
        for (int b0 = 0; b0 < p.nb; b0 += p.n_blk) scales(b0, std::min(p.n_blk, p.nb - b0));
    for (int b0 = 0; b0 < p.nb; b0 += p.n_blk) {
        const int nblk = std::min(p.n_blk, p.nb - b0), nkb = nblk * kKbPerBlk;
        scales(b0, nblk);
        if (b0 == 0)
            ref_kernel<<<std::min(p.nb, 64), kBlk, 0, s>>>(row_ea, (int)N, ref);
        factor_kernel<<<dim3(p.nb, nblk), kBlk, 0, s>>>(ea, row_ea, n_pad, (int)N, f);
        const dim3 tgrid(p.nb, nkb, kBK / 8);
        table_kernel<<<tgrid, kBlk, 0, s>>>(xh, xl, (int)N, b0, near.tau, nullptr, n_pad, p.nb,
                                            nkb, ea, T, gate);
        if (weighted) {
            factor_kernel<<<dim3(p.nb, nblk), kBlk, 0, s>>>(eag, row_eag, n_pad, (int)N, fg);
            table_kernel<<<tgrid, kBlk, 0, s>>>(xh, xl, (int)N, b0, near.tau, gs, n_pad, p.nb, nkb,
                                                eag, Tg, gate);
        }
        MBM_CUDA_TRY(cudaGetLastError());
        for (int t0 = 0; t0 < p.tiles; t0 += p.batch) {
            const int nt = std::min(p.batch, p.tiles - t0);
            const int grid = std::min(nt * kForms, std::max(1, ctx->num_sms));
            contract_kernel<<<grid, kThreads, sizeof(ContractSmem), s>>>(
                T, T, f, f, n_pad, p.nb, nkb, t0, nt, C, gate, ctx->expire_waits);
            if (weighted)
                contract_kernel<<<grid, kThreads, sizeof(ContractSmem), s>>>(
                    Tg, T, fg, f, n_pad, p.nb, nkb, t0, nt, Cg, gate, ctx->expire_waits);
            auto pass = [&](auto kernel) {
                kernel<<<dim3(nt, kBN / kPairCols), 256, 0, s>>>(xh, xl, (int)N, p.nb, t0, near.tau,
                                                                 C, Cg, gs, row_ea, row_eag, ref,
                                                                 sign, out, gate);
            };
            if (what == MBM_CONTRACT_PHI) pass(pair_kernel<kPhi>);
            else if (what == MBM_CONTRACT_FORCES) pass(pair_kernel<kForce>);
            else pass(pair_kernel<kVjp>);
            MBM_CUDA_TRY(cudaGetLastError());
        }
    }
    MBM_CUDA_TRY(launch_near_triples(xh, xl, nullptr, N, near, gs,
                                     what == MBM_CONTRACT_PHI ? MBM_NEAR_PHI : MBM_NEAR_GRAD, sign,
                                     out, nullptr, ctx->num_sms, gate, s));
    MBM_CUDA_TRY(launch_unframe(X, N, frame, xh, xl, nullptr, res, gate, s));
    gate_out->gate = gate;
    gate_out->counter = counter;
    gate_out->xh = xh;
    gate_out->xl = xl;
    gate_out->room = T;
    gate_out->room_bytes =
        p.total - (size_t)(reinterpret_cast<char*>(T) - static_cast<char*>(ctx->scratch));
    *done = true;
    return MBM_OK;
}
