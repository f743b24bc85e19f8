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
// Precision. The tensor cores multiply fp16 exactly and add in FP32 with
// truncation, which would lose 1e-7 of a sum per 16 terms. Each row of L is
// therefore cut into three pieces against a power of two a per row and window
// of 64 columns, |a L| <= 2^15: h, a multiple of 2^7 (8 bits), the rounding m of
// the rest to fp16 and the rounding l of what is left. Products h h are integers
// in units of 2^14, so their sums over a window are exact (measured: bit-exact
// up to 256 columns); the other products but l l go to a second accumulator,
// whose truncation is 2^-8 smaller where h carries the value. Both are added to
// FP32 sums (round to nearest) window by window. Median error against 64 bits at
// N = 2 600 (in brackets the FP32 triple sweep): potentials 4.1e-8 (5.6e-8) on
// uniform sets, 8.1e-8 (1.0e-7) in the unit cube, 7.9e-8 (9.7e-8) on mixtures;
// forces 2.7e-7 (3.4e-7), 2.6e-7 (3.3e-7), 2.6e-7 (3.8e-7). Windows of 256 columns
// were 10 % faster but off by 1.7e-6 on a mixture.
// Pieces have a floor relative to the largest entry of their window, so a set
// whose tightest pairs are 50 times closer than everything around them loses
// digits (isolated dimers at 1/100: 7e-6). The pair pass sums a bound of that
// error next to the terms' magnitudes; a set over the bound is solved again by
// the FP32 sweep behind it, decided on the device (gate), and that sweep returns
// at once otherwise.
//
// Kernels: window maxima -> scales; piece table (stored in the operand layout,
// so a stage is two kinds of bulk copies and no tensor map); contraction
// (tcgen05.mma 128 x 256, warp-specialised, persistent); pair pass over the
// tiles' C. Large N runs in slabs of columns k and batches of tiles; all sums
// are linear in both.
#include <algorithm>
#include <cuda_fp16.h>

#include "bulk_copy.cuh"
#include "contract.h"
#include "device_math.cuh"
#include "tcgen05.cuh"
#include "tile_fp32.cuh"

namespace {

constexpr int kForms = 10;
constexpr int kPieces = 3;
constexpr int kBlk = 256;      // rows per table block, and columns per scale block
constexpr int kBM = 128;       // tile rows
constexpr int kBN = 256;       // tile columns
constexpr int kBK = 32;        // columns k per pipeline stage
constexpr int kKbPerBlk = kBlk / kBK;
constexpr int kWin = 64;       // columns k that share a scale and an accumulator window
constexpr int kKbPerWin = kWin / kBK;
constexpr int kWinPerBlk = kBlk / kWin;
// Factor slots: a window's factors are copied when the MMAs of the window two
// before it are done, which waited for the accumulators of the one three before.
constexpr int kFactorSlots = 4;
constexpr int kFlush = 8;      // windows summed in registers before C takes them
constexpr int kPieceB = kBN * kBK * 2;  // 16 KB: one piece of 256 rows x 32 columns
constexpr int kPieceA = kBM * kBK * 2;
constexpr int kStages = 3;
constexpr int kEpiWarps = 16;
constexpr int kThreads = (kEpiWarps + 2) * 32;
constexpr int kGroup = 8;  // J tiles walked together: their rows and 19 I tiles stay in L2
constexpr long long kWaitLimit = 4000000000LL;

// A_r of l_r(B) = A_r : B, symmetric traceless: xx, yy, xy, xz, yz.
__constant__ double kFormA[kForms][5] = {
    {0.81051314900914676226, -1.0137444298135470439, 0.69187178704706466114, 0.10879332789123717943,
     -0.60113244553623436798},
    {0.29033471318095339961, -0.0037013574801380397359, -0.72945247235092144289,
     -0.48361735206812446962, -1.2002939641387707073},
    {0.56687761555815049061, -0.73198503004752586383, 0.77502100982572152509,
     -0.52554704820191995188, 1.1260055012436281024},
    {0.32794829997931705277, -1.1326061797678746186, -0.75463606268664968689,
     -0.21929916513785778691, 0.2800933877523261306},
    {-0.97297445172993803997, 0.29341922256285760709, 0.90751192347309499305,
     0.32759516889683504779, 0.19146086840943790974},
    {-0.67316138985808209333, 0.46260916239411561729, -0.054408203924041754195, -1.1509903099773033,
     0.17733809272697340492},
    {-0.017877295745476926793, 0.72594943548244305062, 0.18789931162397575175,
     1.0813915903289111131, -0.75562451530097259604},
    {0.13857796836323824696, 0.19482576157814381221, -0.26028666636158319084,
     0.78643885767995610097, 0.97182503734766801594},
    {-1.3260688300585429969, 0.63825499910587256587, -0.89891222534809540828,
     0.37904860109016530897, -0.13692011279071057931},
    {0.9208917500732497988, 0.48297899581067608991, 0.22434594372376326752,
     -0.36411353209625681955, 0.076469687931274560653}};
// largest |l_r(E)| over unit vectors and forms (the largest |eigenvalue| of an A_r)
constexpr float kFormMax = 1.8573f;

// Coefficients of l_r on (Exx - Ezz, Eyy - Ezz, Exy, Exz, Eyz).
struct FormCoef {
    float ch[kForms][5], cl[kForms][5];
};
__device__ __forceinline__ double form_coef(int r, int m) {
    return m < 2 ? kFormA[r][m] : 2.0 * kFormA[r][m];
}

// Split of the coefficients for exact chains: ch a multiple of 2^-10, cl the rest.
__device__ __forceinline__ void form_split(int r, int m, float& ch, float& cl) {
    const double c = form_coef(r, m);
    ch = rintf((float)(c * 1024.0)) / 1024.0f;
    cl = (float)(c - (double)ch);
}
// The same for a component |v| <= 1: vh a multiple of 2^-11, so that the five
// products ch vh are multiples of 2^-21 whose sum stays below 8: exact in FP32.
__device__ __forceinline__ void comp_split(float h, float l, float& vh, float& vl) {
    constexpr float kGrid = 1.5f * 4096.0f;
    vh = __fsub_rn(__fadd_rn(h, kGrid), kGrid);
    vl = __fadd_rn(__fsub_rn(h, vh), l);
}
__device__ __forceinline__ void form_value(const float (&ch)[5], const float (&cl)[5],
                                           const float (&vh)[5], const float (&vl)[5], float& H,
                                           float& Lw) {
    H = 0.f;
    Lw = 0.f;
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        H = __fmaf_rn(ch[m], vh[m], H);
        Lw = __fmaf_rn(ch[m], vl[m], Lw);
        Lw = __fmaf_rn(cl[m], __fadd_rn(vh[m], vl[m]), Lw);
    }
}

// ----- double-float helpers -----
struct df {
    float h, l;
};
__device__ __forceinline__ df df_fast(float a, float b) {  // |a| >= |b|
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ df df_mul(df a, df b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    return df_fast(p, e);
}
__device__ __forceinline__ df df_add(df a, df b) {
    const float s = __fadd_rn(a.h, b.h);
    const float t = __fsub_rn(s, a.h);
    float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
    e = __fadd_rn(e, __fadd_rn(a.l, b.l));
    return df_fast(s, e);
}
__device__ __forceinline__ df df_diff(float qh, float ql, float ph, float pl) {
    const float s = __fsub_rn(qh, ph);
    const float t = __fsub_rn(s, qh);
    const float e = __fsub_rn(__fsub_rn(qh, __fsub_rn(s, t)), __fadd_rn(ph, t));
    return df_fast(s, __fadd_rn(e, __fsub_rn(ql, pl)));
}

// Pair terms to about 2^-40: v = (Exx - Ezz, Eyy - Ezz, Exy, Exz, Eyz) and
// rho = r^-3. False if the pair is coincident or not finite (terms then zero).
struct PairDf {
    df v[5], rho;
    float s, y;  // r^2 and 1/r to FP32
};
__device__ __forceinline__ bool pair_df(float4 ph, float4 pl, float4 qh, float4 ql, PairDf& o) {
    const df dx = df_diff(qh.x, ql.x, ph.x, pl.x);
    const df dy = df_diff(qh.y, ql.y, ph.y, pl.y);
    const df dz = df_diff(qh.z, ql.z, ph.z, pl.z);
    const df xx = df_mul(dx, dx), yy = df_mul(dy, dy), zz = df_mul(dz, dz);
    const df s = df_add(df_add(xx, yy), zz);
    o.s = s.h;
    if (!(s.h > 0.f) || !(s.h < INFINITY)) return false;
    // 1/r: hardware estimate and one Newton step, kept as a two-term number
    const float y0 = rsqrtf(s.h);
    const float p = __fmul_rn(y0, y0), pe = __fmaf_rn(y0, y0, -p);
    const float q = __fmul_rn(s.h, p), qe = __fmaf_rn(s.h, p, -q);
    const float res = __fsub_rn(__fsub_rn(1.0f, q), __fmaf_rn(s.l, p, __fmaf_rn(s.h, pe, qe)));
    const df y = df_fast(y0, __fmul_rn(__fmul_rn(0.5f, y0), res));
    const df y2 = df_mul(y, y);
    o.y = y.h;
    o.rho = df_mul(y2, y);
    const df ez = df_mul(zz, y2);
    const df nez = {-ez.h, -ez.l};
    o.v[0] = df_add(df_mul(xx, y2), nez);
    o.v[1] = df_add(df_mul(yy, y2), nez);
    o.v[2] = df_mul(df_mul(dx, dy), y2);
    o.v[3] = df_mul(df_mul(dx, dz), y2);
    o.v[4] = df_mul(df_mul(dy, dz), y2);
    return true;
}

__device__ __forceinline__ float pow2f(int e) {  // 2^e, 0 below the normal range
    return e < -126 ? 0.f : __int_as_float((min(e, 127) + 127) << 23);
}

// ---------------------------------------------------------------------------
// Scales. ea[w][i]: exponent of a(i, w), the power of two with |a l| <= 2^15
// over the 64 columns k of window w (times |g_k| for the weighted table). A
// CTA takes 256 rows and one window; its columns are staged in shared memory.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlk)
scale_kernel(const float4* __restrict__ xh, const float4* __restrict__ xl, int N, int w0,
             const double* __restrict__ g, int n_pad, int* __restrict__ ea,
             int* __restrict__ row_ea, int* __restrict__ flags) {
    __shared__ float4 kh[kWin], kl[kWin];
    __shared__ float kg[kWin];
    const int w = blockIdx.y, k0 = (w0 + w) * kWin;
    const int i = blockIdx.x * kBlk + threadIdx.x;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (threadIdx.x < kWin) {
        const int kk = k0 + threadIdx.x;
        kh[threadIdx.x] = kk < N ? xh[kk] : z4;
        kl[threadIdx.x] = kk < N ? xl[kk] : z4;
        kg[threadIdx.x] = g && kk < N ? fabsf((float)g[kk]) : 1.f;
    }
    __syncthreads();
    const float4 ih = i < N ? xh[i] : z4, il = i < N ? xl[i] : z4;
    const int cnt = min(kWin, N - k0);
    float best = 0.f;  // largest rho (or |g| rho) of the window
    bool bad = false;
    if (i < N) {
        float smin = INFINITY;
        for (int q = 0; q < cnt; ++q) {
            const float s = pair_d2_hilo(ih, il, kh[q], kl[q]);
            const bool self = k0 + q == i;
            bad |= !self && !(s > 0.f);
            if (!self && s > 0.f && s < INFINITY) {
                if (g) {
                    const float y = rsqrtf(s);
                    best = fmaxf(best, kg[q] * (y * y * y));
                } else {
                    smin = fminf(smin, s);
                }
            }
        }
        if (!g && smin < INFINITY) {
            const float y = rsqrtf(smin);
            best = y * y * y;
        }
    }
    if (bad && !g) atomicOr(flags, MBM_FLAG_COINCIDENT);
    int e = 127;  // nothing in this window
    if (best > 0.f && best < INFINITY) e = 14 - ilogbf(best * (kFormMax * 1.0001f));
    if (best > 0.f) e = max(-120, min(126, e));
    ea[(size_t)w * n_pad + i] = e;
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

// f[w][i] = 2^(row exponent - window exponent) <= 1; for the error bound its
// maximum over the four windows of a 256-column block, fb[b][i], and that
// maximum over 16 rows, fb16[b][i / 16].
__global__ void __launch_bounds__(kBlk)
factor_kernel(const int* __restrict__ ea, const int* __restrict__ row_ea, int n_pad, int N,
              float* __restrict__ f, float* __restrict__ fb, float* __restrict__ fb16) {
    const int b = blockIdx.y, i = blockIdx.x * kBlk + threadIdx.x;
    const int er = i < N ? row_ea[i] : 0;
    float m = 0.f;
    for (int q = 0; q < kWinPerBlk; ++q) {
        const size_t o = (size_t)(b * kWinPerBlk + q) * n_pad + i;
        const int e = ea[o];
        const float v = i < N && e < 127 ? pow2f(er - e) : 0.f;
        f[o] = v;
        m = fmaxf(m, v);
    }
    fb[(size_t)b * n_pad + i] = m;
    if (!fb16) return;
    for (int o = 8; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 15) == 0) fb16[(size_t)b * (n_pad / 16) + i / 16] = m;
}

// ---------------------------------------------------------------------------
// Piece table, in the contraction's operand layout: T[r][row block][kb][piece]
// is 256 rows x 32 columns as core matrices of 8 rows x 8 columns (128 bytes),
// [row group][column group][row][column]. A CTA writes all forms and pieces of
// 256 rows x 8 columns; a thread owns a row (16-byte stores, 128 contiguous bytes per 8 rows). FP32-pipe bound: ~140 operations
// per pair and ~30 per form; the form is an exact FMA chain on the leading
// bits plus a small one on the rest.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlk)
table_kernel(const float4* __restrict__ xh, const float4* __restrict__ xl, int N, int b0,
             const double* __restrict__ g, int n_pad, int nb, int nkb, const int* __restrict__ ea,
             unsigned char* __restrict__ T) {
    __shared__ FormCoef fc;
    __shared__ float4 kh[kBK], kl[kBK];
    __shared__ float kg[kBK], kgl[kBK];
    const int rb = blockIdx.x, kb = blockIdx.y;
    const int k0 = b0 * kBlk + kb * kBK;
    const int row = threadIdx.x, i = rb * kBlk + row;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (threadIdx.x < kForms * 5) {
        const int r = threadIdx.x / 5, m = threadIdx.x % 5;
        form_split(r, m, fc.ch[r][m], fc.cl[r][m]);
    }
    if (threadIdx.x < kBK) {
        const int k = k0 + threadIdx.x;
        kh[threadIdx.x] = k < N ? xh[k] : z4;
        kl[threadIdx.x] = k < N ? xl[k] : z4;
        const double gk = g && k < N ? g[k] : 1.0;
        kg[threadIdx.x] = (float)gk;
        kgl[threadIdx.x] = (float)(gk - (double)(float)gk);
    }
    __syncthreads();
    const float4 ih = i < N ? xh[i] : z4, il = i < N ? xl[i] : z4;
    // two exact factors: one alone may pass the FP32 range
    const int e = ea[(size_t)(kb / kKbPerWin) * n_pad + i];
    const int e1 = e / 2;
    const float a1 = pow2f(e1), a2 = pow2f(e - e1);
    constexpr float kMagic = 1.5f * 1073741824.0f;  // rounds to multiples of 2^7
    {
        const int k8 = blockIdx.z;
        float vh[8][5], vl[8][5], rh[8], rl[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int kk = k8 * 8 + q, k = k0 + kk;
            PairDf p;
            const bool ok = i < N && k < N && k != i && pair_df(ih, il, kh[kk], kl[kk], p);
            df rho = {0.f, 0.f};
            if (ok) {
                rho = p.rho;
                if (g) rho = df_mul(rho, df{kg[kk], kgl[kk]});
                rho = {rho.h * a1 * a2, rho.l * a1 * a2};
            }
            rh[q] = rho.h;
            rl[q] = rho.l;
#pragma unroll
            for (int m = 0; m < 5; ++m)
                comp_split(ok ? p.v[m].h : 0.f, ok ? p.v[m].l : 0.f, vh[q][m], vl[q][m]);
        }
        const size_t off = (size_t)(row >> 3) * 512 + k8 * 128 + (row & 7) * 16;
#pragma unroll 1
        for (int r = 0; r < kForms; ++r) {
            float ch[5], cl[5];
#pragma unroll
            for (int m = 0; m < 5; ++m) {
                ch[m] = fc.ch[r][m];
                cl[m] = fc.cl[r][m];
            }
            __align__(16) __half h8[8], m8[8], l8[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                float H, Lw;
                form_value(ch, cl, vh[q], vl[q], H, Lw);
                const float p = __fmul_rn(H, rh[q]);
                float x = __fmaf_rn(H, rh[q], -p);
                x = __fmaf_rn(H, rl[q], x);
                x = __fmaf_rn(Lw, rh[q], x);
                const float hi = __fsub_rn(__fadd_rn(p, kMagic), kMagic);
                const float rem = __fadd_rn(__fsub_rn(p, hi), x);
                const __half mh = __float2half_rn(rem);
                h8[q] = __float2half_rn(hi);
                m8[q] = mh;
                l8[q] = __float2half_rn(__fsub_rn(rem, __half2float(mh)));
            }
            unsigned char* dst =
                T + (((size_t)r * nb + rb) * nkb + kb) * (size_t)(kPieces * kPieceB) + off;
            *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(h8);
            *reinterpret_cast<uint4*>(dst + kPieceB) = *reinterpret_cast<const uint4*>(m8);
            *reinterpret_cast<uint4*>(dst + 2 * kPieceB) = *reinterpret_cast<const uint4*>(l8);
        }
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
// forms outermost. Warps 0-15: accumulator windows to registers every 64
// columns and to C every 512 (shorter FP32 chains); warp 16: bulk copies
// (72 KB stages of 32 columns); warp 17: MMAs (8 products of pieces). The
// accumulators fill TMEM: 256 columns for h h and 256 for the rest; each is
// drained while the other is computed. (The rest in two halves of 128 columns
// reads A twice and is bound by shared memory: forces of 8 192 particles took
// 40.6 ms against 27.1; scale factors read from global memory in the drain: 37.1.)
__global__ void __launch_bounds__(kThreads, 1)
contract_kernel(const unsigned char* __restrict__ TA, const unsigned char* __restrict__ TB,
                const float* __restrict__ fA, const float* __restrict__ fB, int n_pad, int nb,
                int nkb, int t0, int nt, float* __restrict__ C, int* __restrict__ flags) {
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
                    if (kb % kKbPerWin == 0) {
                        const int q = win++ % kFactorSlots;
                        const size_t w = (size_t)(kb / kKbPerWin) * n_pad;
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
            // products but h h, as (piece of A, piece of B), the largest last:
            // what follows an addition truncates it
            constexpr int kOther = 7;
            constexpr int pa[kOther] = {2, 1, 0, 2, 0, 1, 1}, pb[kOther] = {1, 2, 2, 0, 1, 0, 1};
            unsigned it = 0, win = 0;  // stages used, windows handed over
            bool ok = true;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                for (int kb = 0; kb < nkb; kb += kKbPerWin, ++win) {
                    // h h of the whole window, then the rest: the previous window's
                    // second accumulator is drained under the former, the first
                    // one under the latter
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
                    if (win && !wait_phase(sm, &sm.acc_empty[1], (win - 1) & 1)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
#pragma unroll 1
                    for (int u = 0; u < kKbPerWin; ++u, ++it) {
                        const unsigned ab = smem_u32(sm.a[it % kStages]);
                        const unsigned bb = smem_u32(sm.b[it % kStages]);
#pragma unroll
                        for (int q = 0; q < kOther; ++q)
#pragma unroll
                            for (int k = 0; k < kBK / 16; ++k)
                                tc_mma_f16(tmem + kBN,
                                           tc_desc(ab + pa[q] * kPieceA + k * 256, 128, 512),
                                           tc_desc(bb + pb[q] * kPieceB + k * 256, 128, 512), idesc,
                                           u + q + k > 0);
                        if (u == kKbPerWin - 1) tc_commit(smem_u32(&sm.acc_full[1]));
                        tc_commit(smem_u32(&sm.empty[it % kStages]));
                    }
                }
            }
            // MMAs in flight end before TMEM and shared memory are released
            if (it > 0)
                mbar_wait_bounded(&sm.empty[(it - 1) % kStages], ((it - 1) / kStages) & 1,
                                  kWaitLimit);
        }
    } else {
        // rows 32 (warp % 4) + lane of the tile, columns 64 (warp / 4) + 0..63
        const int row = (warp & 3) * 32 + lane, col = (warp >> 2) * 64;
        const unsigned base = tmem + ((unsigned)(warp & 3) << 21) + col;
        const int n_win = nkb / kKbPerWin;
        unsigned win = 0;
        bool ok = true;
        for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
            int I, J;
            decode_tile(t0 + item % nt, nb, I, J);
            float4* out = reinterpret_cast<float4*>(C) +
                          (size_t)((item % nt) * kForms + item / nt) * (kBM * kBN / 4) +
                          (size_t)(col / 4) * kBM + row;
            float2 acc[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) acc[c] = make_float2(0.f, 0.f);
            for (int w = 0; w < n_win; ++w, ++win) {
                const unsigned slot = win % kFactorSlots;
                if (!__all_sync(0xffffffffu,
                                wait_phase(sm, &sm.factors[slot], (win / kFactorSlots) & 1))) {
                    ok = false;
                    break;
                }
                const float2 fi = f2_splat(sm.fi[slot][row]);
                const float* fj = &sm.fj[slot][col];
#pragma unroll 1
                for (int a = 0; a < 2; ++a) {
                    if (!__all_sync(0xffffffffu, wait_phase(sm, &sm.acc_full[a], win & 1))) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    drain(base + a * kBN, fj, fi, acc);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.acc_empty[a]);
                }
                if (!ok) break;
                if (w % kFlush == kFlush - 1 || w == n_win - 1) {
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        float4 v = make_float4(acc[2 * c].x, acc[2 * c].y, acc[2 * c + 1].x,
                                               acc[2 * c + 1].y);
                        if (w >= kFlush) {
                            const float4 u = out[c * kBM];
                            v = make_float4(v.x + u.x, v.y + u.y, v.z + u.z, v.w + u.w);
                        }
                        out[c * kBM] = v;
                        acc[2 * c] = acc[2 * c + 1] = make_float2(0.f, 0.f);
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x == 0 && sm.abort) atomicOr(flags, MBM_FLAG_TIMEOUT);
    if (warp == 0) tc_free(tmem, 512);
}

// ---------------------------------------------------------------------------
// Pair pass: four CTAs per tile, a thread per row and 32 columns, four columns
// at a time. Potentials: rho sum_r l_r(E) C^r, the forms as exact as in the table
// (summing C^r A_r first costs two more roundings where the terms cancel).
// Gradients: G = sum_r C^r A_r and (rho / r)(2 G e - 5 (e.G e) e). Column sums go
// through a transposed shared buffer. Next to the result it sums, per particle,
// the magnitudes of the pair terms and the bound of the slices' error.
// ---------------------------------------------------------------------------
enum : int { kPhi = 0, kForce = 1, kVjp = 2 };

// Pieces are floating-point down to a floor of 2^-25 in units of |a L| <= 2^15;
// a block's C is off by at most that times the other factor (2^15), twice, in
// units of a_i a_j, and ten forms of |l| <= 1.86 rho add up to about four times one.
constexpr float kSliceErr = 1.0f / 128.0f;
// Of the summed magnitudes. The bound takes every entry of a window at the floor
// against the largest of 16 columns, so it is far above the error: mixtures and
// unit cubes reach 3e-5 with no loss, dimers 20 times closer than their
// spacing 0.1 with none, 50 times 20 with the first loss (1e-6).
constexpr double kGateTol = 1.0 / 64.0;

constexpr int kStep = 16;      // columns between two column sums
constexpr int kPairCols = 64;  // columns of a tile per CTA: 20 tiles alone left SMs idle

template <int Mode>
__global__ void __launch_bounds__(256)
pair_kernel(const float4* __restrict__ xh, const float4* __restrict__ xl, int N, int n_pad, int nb,
            int n_blk, int t0, const float* __restrict__ C, const float* __restrict__ Cg,
            const double* __restrict__ g, const int* __restrict__ row_ea,
            const int* __restrict__ row_eag, const int* __restrict__ ref,
            const float* __restrict__ fb, const float* __restrict__ fb16,
            const float* __restrict__ fbg, double sign, double* __restrict__ out,
            double* __restrict__ mag, double* __restrict__ err) {
    constexpr int kVals = Mode == kPhi ? 3 : 5;  // components, magnitude, error bound
    __shared__ float4 jh[kBN], jl[kBN];
    __shared__ float wj[kBN], gj[kBN];
    __shared__ float coef[kForms][5];  // gradients: A_r
    __shared__ FormCoef fc;            // potentials
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
        gj[threadIdx.x] = Mode == kVjp && j < N ? (float)g[j] : 0.f;
        if (threadIdx.x < kForms * 5) {
            const int r = threadIdx.x / 5, m = threadIdx.x % 5;
            coef[r][m] = (float)kFormA[r][m];
            form_split(r, m, fc.ch[r][m], fc.cl[r][m]);
        }
    }
    __syncthreads();
    const bool iv = i < N;
    const float4 ih = iv ? xh[i] : z4, il = iv ? xl[i] : z4;
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
        float slice = 0.f, slice_g = 0.f;  // bound of |delta C| in units of A_i A_j
        if (iv) {
            const float* mj = fb16 + (J * kBN + c0) / kStep;
            for (int b = 0; b < n_blk; ++b) {
                const float m = mj[(size_t)b * (n_pad / kStep)];
                slice = fmaf(fb[(size_t)b * n_pad + i], m, slice);
                if (Mode == kVjp) slice_g = fmaf(fbg[(size_t)b * n_pad + i], m, slice_g);
            }
            slice *= kSliceErr;
            slice_g *= kSliceErr * cg_scale;
        }
#pragma unroll
        for (int cc = 0; cc < kStep; cc += 4) {
            const int c4 = (c0 + cc) >> 2;
            float G[4][5];             // gradients: sum_r C^r A_r
            float T[4];                // potentials: sum_r l_r C^r
            float vh[4][5], vl[4][5], rho[4];
            if (Mode == kPhi) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int c = c0 + cc + q, j = J * kBN + c;
                    PairDf p;
                    const bool ok = pair_df(ih, il, jh[c], jl[c], p) && iv && j < N && j > i;
                    T[q] = 0.f;
                    rho[q] = ok ? p.rho.h * rho_scale1 * rho_scale2 : 0.f;
#pragma unroll
                    for (int m = 0; m < 5; ++m)
                        comp_split(ok ? p.v[m].h : 0.f, ok ? p.v[m].l : 0.f, vh[q][m], vl[q][m]);
                }
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int m = 0; m < 5; ++m) G[q][m] = 0.f;
            }
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
                if (Mode == kPhi) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float H, Lw;
                        form_value(fc.ch[r], fc.cl[r], vh[q], vl[q], H, Lw);
                        T[q] = fmaf(__fadd_rn(H, Lw), x[q], T[q]);
                    }
                } else {
#pragma unroll
                    for (int m = 0; m < 5; ++m) {
                        const float a = coef[r][m];
#pragma unroll
                        for (int q = 0; q < 4; ++q) G[q][m] = fmaf(a, x[q], G[q][m]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int c = c0 + cc + q, j = J * kBN + c;
                const bool on = iv && j < N && j > i;
                float val[kVals];  // components, their magnitude, the error bound
                float bound = slice;
                if (Mode == kVjp) bound = fmaf(slice, fabsf(gi + gj[c]), slice_g);
                if (Mode == kPhi) {
                    val[0] = T[q] * rho[q];
                    val[1] = fabsf(val[0]);
                    val[2] = bound * rho[q];
                } else {
                    const float dx = (jh[c].x - ih.x) + (jl[c].x - il.x);
                    const float dy = (jh[c].y - ih.y) + (jl[c].y - il.y);
                    const float dz = (jh[c].z - ih.z) + (jl[c].z - il.z);
                    const float s = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
                    float y = rsqrtf(s);
                    y = fmaf(0.5f * y, fmaf(-s * y, y, 1.0f), y);
                    const bool ok = on && s > 0.f && s < INFINITY;
                    const float ex = ok ? dx * y : 0.f, ey = ok ? dy * y : 0.f,
                                ez = ok ? dz * y : 0.f;
                    const float k = ok ? (y * y * y) * rho_scale1 * rho_scale2 * y : 0.f;
                    // G is symmetric and traceless: (xx, yy, xy, xz, yz)
                    const float gx = fmaf(G[q][3], ez, fmaf(G[q][2], ey, G[q][0] * ex));
                    const float gy = fmaf(G[q][4], ez, fmaf(G[q][1], ey, G[q][2] * ex));
                    const float gz =
                        fmaf(-(G[q][0] + G[q][1]), ez, fmaf(G[q][4], ey, G[q][3] * ex));
                    const float u = -5.0f * fmaf(ez, gz, fmaf(ey, gy, ex * gx));
                    val[0] = k * fmaf(u, ex, 2.0f * gx);
                    val[1] = k * fmaf(u, ey, 2.0f * gy);
                    val[2] = k * fmaf(u, ez, 2.0f * gz);
                    val[kVals - 2] = fmaxf(fabsf(val[0]), fmaxf(fabsf(val[1]), fabsf(val[2])));
                    val[kVals - 1] = bound * k;
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
                if (d == kVals - 2) atomicAdd(&mag[j], v);
                else if (d == kVals - 1) atomicAdd(&err[j], v);
                else if (Mode == kPhi) atomicAdd(&out[j], 0.5 * v);
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
            if (d == kVals - 2) atomicAdd(&mag[i], v);
            else if (d == kVals - 1) atomicAdd(&err[i], v);
            else if (Mode == kPhi) atomicAdd(&out[i], 0.5 * v);
            else atomicAdd(&out[3 * (size_t)i + d], -sign * v);
        }
    }
}

// Gate: some particle's summed error bound passes the tolerance.
__global__ void __launch_bounds__(kBlk)
gate_kernel(const double* __restrict__ mag, const double* __restrict__ err, int N,
            int* __restrict__ gate) {
    const int i = blockIdx.x * kBlk + threadIdx.x;
    if (i < N && err[i] > kGateTol * mag[i]) *gate = 1;
}

__global__ void zero_if_kernel(const int* __restrict__ gate, double* __restrict__ out, int64_t n) {
    if (!*gate) return;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = 0.0;
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
Plan make_plan(int64_t N, bool weighted, size_t cap) {
    Plan p;
    p.nb = (int)((N + kBlk - 1) / kBlk);
    p.n_pad = p.nb * kBlk;
    p.tiles = p.nb * (p.nb + 1);
    const int copies = weighted ? 2 : 1;
    const size_t per_blk = (size_t)kForms * p.nb * kKbPerBlk * kPieces * kPieceB * copies;
    const size_t per_tile = (size_t)kForms * kBM * kBN * sizeof(float) * copies;
    const size_t fixed = up256((size_t)p.n_pad * 32) + 16 * (size_t)p.n_pad +
                         2 * 4 * (size_t)p.n_pad + 131072;
    // per 256 columns of a slab: ea and f per window, fb (and the weighted ones), fb16
    const size_t per_blk_f = (size_t)p.n_pad * (8 * kWinPerBlk + 4) * copies + (size_t)p.n_pad / 4;
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
    return p;
}

}  // namespace

constexpr int64_t kContractMaxN = (int64_t)1 << 20;  // tile numbers fit an int

static Plan plan_for(int64_t N, bool weighted, size_t cap) {
    return N <= kContractMaxN ? make_plan(N, weighted, cap) : Plan{};
}

size_t mbm_contract_bytes(int64_t N, bool forces) {
    if (N < (forces ? kContractMinForces : kContractMinPhi)) return 0;
    return plan_for(N, false, (size_t)1 << 60).total;
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
    const Plan p = plan_for(N, weighted, cap);
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
    auto* xh = reinterpret_cast<float4*>(take((size_t)N * 16));
    auto* xl = reinterpret_cast<float4*>(take((size_t)N * 16));
    auto* mag = reinterpret_cast<double*>(take((size_t)n_pad * 8));
    auto* err = reinterpret_cast<double*>(take((size_t)n_pad * 8));
    auto* row_ea = reinterpret_cast<int*>(take((size_t)n_pad * 4));
    auto* row_eag = reinterpret_cast<int*>(take((size_t)n_pad * 4));
    const size_t per_w = (size_t)n_pad * 4 * kWinPerBlk * p.n_blk, per_b = (size_t)n_pad * 4 * p.n_blk;
    auto* ea = reinterpret_cast<int*>(take(per_w));
    auto* f = reinterpret_cast<float*>(take(per_w));
    auto* fb = reinterpret_cast<float*>(take(per_b));
    auto* fb16 = reinterpret_cast<float*>(take(per_b / 16));
    int* eag = weighted ? reinterpret_cast<int*>(take(per_w)) : nullptr;
    float* fg = weighted ? reinterpret_cast<float*>(take(per_w)) : nullptr;
    float* fbg = weighted ? reinterpret_cast<float*>(take(per_b)) : nullptr;
    auto* T = reinterpret_cast<unsigned char*>(take(p.table));
    auto* Tg = weighted ? reinterpret_cast<unsigned char*>(take(p.table)) : nullptr;
    auto* C = reinterpret_cast<float*>(take(p.cbuf));
    auto* Cg = weighted ? reinterpret_cast<float*>(take(p.cbuf)) : nullptr;

    const int n_out = what == MBM_CONTRACT_PHI ? 1 : 3;
    MBM_CUDA_TRY(cudaMemsetAsync(ctx->d_flags, 0, sizeof(int), s));
    MBM_CUDA_TRY(cudaMemsetAsync(head, 0, 256, s));
    MBM_CUDA_TRY(cudaMemsetAsync(ref, 0x7f, 4, s));
    MBM_CUDA_TRY(cudaMemsetAsync(mag, 0, up256((size_t)n_pad * 8) * 2, s));
    MBM_CUDA_TRY(cudaMemsetAsync(row_ea, 0x7f, up256((size_t)n_pad * 4) * 2, s));
    MBM_CUDA_TRY(cudaMemsetAsync(out, 0, (size_t)N * n_out * sizeof(double), s));
    MBM_CUDA_TRY(launch_pack_hilo(X, N, xh, xl, ctx->d_flags, s));

    MBM_CUDA_TRY(cudaFuncSetAttribute((const void*)contract_kernel,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sizeof(ContractSmem)));
    mbm_time_begin(ctx, s);
    // Row exponents come from all columns: with several slabs a first pass over
    // them finds the row exponents before any table is built.
    const int slabs = (p.nb + p.n_blk - 1) / p.n_blk;
    auto scales = [&](int b0, int nblk) {
        const dim3 grid(p.nb, nblk * kWinPerBlk);
        scale_kernel<<<grid, kBlk, 0, s>>>(xh, xl, (int)N, b0 * kWinPerBlk, nullptr, n_pad, ea,
                                           row_ea, ctx->d_flags);
        if (weighted)
            scale_kernel<<<grid, kBlk, 0, s>>>(xh, xl, (int)N, b0 * kWinPerBlk, g, n_pad, eag,
                                               row_eag, ctx->d_flags);
    };
    if (slabs > 1)
        for (int b0 = 0; b0 < p.nb; b0 += p.n_blk) scales(b0, std::min(p.n_blk, p.nb - b0));
    for (int b0 = 0; b0 < p.nb; b0 += p.n_blk) {
        const int nblk = std::min(p.n_blk, p.nb - b0), nkb = nblk * kKbPerBlk;
        scales(b0, nblk);
        if (b0 == 0)
            ref_kernel<<<std::min(p.nb, 64), kBlk, 0, s>>>(row_ea, (int)N, ref);
        factor_kernel<<<dim3(p.nb, nblk), kBlk, 0, s>>>(ea, row_ea, n_pad, (int)N, f, fb, fb16);
        table_kernel<<<dim3(p.nb, nkb, kBK / 8), kBlk, 0, s>>>(xh, xl, (int)N, b0, nullptr, n_pad, p.nb, nkb,
                                                      ea, T);
        if (weighted) {
            // fb16 keeps the unweighted maxima: the weighted rows meet unweighted columns
            factor_kernel<<<dim3(p.nb, nblk), kBlk, 0, s>>>(eag, row_eag, n_pad, (int)N, fg, fbg,
                                                            nullptr);
            table_kernel<<<dim3(p.nb, nkb, kBK / 8), kBlk, 0, s>>>(xh, xl, (int)N, b0, g, n_pad, p.nb, nkb,
                                                          eag, Tg);
        }
        MBM_CUDA_TRY(cudaGetLastError());
        for (int t0 = 0; t0 < p.tiles; t0 += p.batch) {
            const int nt = std::min(p.batch, p.tiles - t0);
            const int grid = std::min(nt * kForms, std::max(1, ctx->num_sms));
            contract_kernel<<<grid, kThreads, sizeof(ContractSmem), s>>>(
                T, T, f, f, n_pad, p.nb, nkb, t0, nt, C, ctx->d_flags);
            if (weighted)
                contract_kernel<<<grid, kThreads, sizeof(ContractSmem), s>>>(
                    Tg, T, fg, f, n_pad, p.nb, nkb, t0, nt, Cg, ctx->d_flags);
            if (what == MBM_CONTRACT_PHI)
                pair_kernel<kPhi><<<dim3(nt, kBN / kPairCols), 256, 0, s>>>(xh, xl, (int)N, n_pad, p.nb, nblk, t0, C, Cg,
                                                     g, row_ea, row_eag, ref, fb, fb16, fbg, sign, out,
                                                     mag, err);
            else if (what == MBM_CONTRACT_FORCES)
                pair_kernel<kForce><<<dim3(nt, kBN / kPairCols), 256, 0, s>>>(xh, xl, (int)N, n_pad, p.nb, nblk, t0, C,
                                                       Cg, g, row_ea, row_eag, ref, fb, fb16, fbg,
                                                       sign, out, mag, err);
            else
                pair_kernel<kVjp><<<dim3(nt, kBN / kPairCols), 256, 0, s>>>(xh, xl, (int)N, n_pad, p.nb, nblk, t0, C, Cg,
                                                     g, row_ea, row_eag, ref, fb, fb16, fbg, sign, out,
                                                     mag, err);
            MBM_CUDA_TRY(cudaGetLastError());
        }
    }
    gate_kernel<<<p.nb, kBlk, 0, s>>>(mag, err, (int)N, gate);
    const int64_t n_val = N * n_out;
    zero_if_kernel<<<(unsigned)((n_val + 255) / 256), 256, 0, s>>>(gate, out, n_val);
    MBM_CUDA_TRY(cudaGetLastError());
    gate_out->gate = gate;
    gate_out->counter = counter;
    gate_out->xh = xh;
    gate_out->xl = xl;
    *done = true;
    return MBM_OK;
}
