// Step a4 of the mixed path with the panel updates on the tcgen05 tensor
// cores (a4 arithmetic QMC_A4_TENSOR).
//
// The Gauss-Jordan elimination with partial pivoting of k_gj / k_gj_ff
// (implicit pivoting: rows never move, a row map records the pivots; after
// the last panel the array holds Res with X^-1[a][b] = Res[pp[a]][ipp[b]]),
// on a float-pair work matrix (~48-bit significand), in panels of kGtB = 32
// columns, as launches over all matrices of a walker chunk:
//
//   k_gt_init    float-pair copy of X (rows padded to an even length) and ||X||_inf
//   per panel jb:
//   k_gt_panel   one CTA per matrix eliminates the n x 32 panel, one thread per
//                row (pivot = the first row with the largest |entry| among
//                the rows not used yet: the pivots of LU with partial
//                pivoting), in sub-panels of 8 held in registers, and writes
//                the operands of the panel's update in exact BF16 slices: the
//                panel P [n][32] (row i scaled by 2^-E_i) and the pivot rows
//                U [32][n] as they were before the update (column j scaled
//                by 2^-F_j), seven slices of 7 bits
//                each (the scheme of the C1/C5 products, one slice more)
//   k_gt_update  X[i][j] <- [i is not a pivot row of the panel] X[i][j]
//                           + sum_c P[i][c] U[c][j]
//                for every column j outside the panel; a CTA per one or several tiles of 128 rows,
//                warp-specialised (warps moving the old values by tensor TMA
//                and the operands by bulk copies, an MMA warp, 16 epilogue
//                warps), loops over
//                the 32-column tiles and issues, per tile, 2 K16
//                steps x 28 slice-pair MMAs into seven TMEM
//                accumulators, one per order d = i + j <= 6 of the pair: each
//                sums at most 7 x 32 products of at most 128 x 128 units of
//                2^-7(d+2), below 2^24 units, so every kept product is added
//                exactly; the dropped orders d >= 7 are below ~2^-47 of the
//                update (float pairs: 2^-48).  The epilogue adds orders 0..3
//                as float pairs and 4..6 (below 2^-21 of the update) first in
//                FP32 (rounding ~2^-46), scales by 2^(E_i + F_j) as two exact
//                FP32 multiplications and adds the result to the float-pair X
//   k_gt_final   ||X^-1||_inf, kappa_inf, log|det| and its sign, D^-1 = X^-T
//
// Matrices with kappa_inf above the threshold, a zero pivot, a non-finite
// result or an expired bounded wait are flagged, and the FP64 recomputation
// (C1 from the positions and the FP64 elimination) replaces them, exactly as
// for k_gj_ff.
#include <cooperative_groups.h>
#include <math.h>
#include <string.h>

#include <algorithm>

#include "f64_bits.cuh"
#include "ff_math.cuh"
#include "qmc_internal.cuh"
#include "slices.cuh"
#include "umma.cuh"

namespace qmc {

namespace cg = cooperative_groups;

constexpr int kGtB = 32;                             // panel width = K of the update
constexpr int kGtThreads = 256;                      // init and final kernels
constexpr int kGtWarps = kGtThreads / 32;
constexpr int kGtEpWarps = 16;                       // update kernel: 4 lane quadrants x 4 groups of 8 columns,
constexpr int kGtUpThreads = 32 * (kGtEpWarps + 3);  // plus the X, B and MMA warps
constexpr int kGtN = 32;                             // columns per update tile (= the panel width)
constexpr int kGtSl = 7;                             // slices per operand
constexpr uint32_t kGtAPlane = 128 * kGtB * 2;       // [128 rows][32 K] BF16, K-major, 64-byte swizzle: 8 KB
constexpr uint32_t kGtBPlane = kGtB * kGtN * 2;      // [32 K][32 columns] BF16, MN-major, 64-byte swizzle: 2 KB
constexpr uint32_t kGtBSbo = 512;                    // next group of 8 K rows (one 32-column atom each)
constexpr int kGtBs = 3;                             // stages of pivot-row slices
constexpr int kGtXs = 3;                             // stages of old values
constexpr uint32_t kGtXStage = 128 * kGtN * 8;       // [2 halves][128 rows][16 float pairs], 128-byte swizzle
constexpr uint32_t kGtATmem = 256;                   // TMEM: 7 accumulators of 32 columns at 0, the panel
constexpr uint32_t kGtAtCols = kGtSl * 16;           // slices (7 x 16 columns) of two row tiles from 256

// MN-major, 64-byte swizzle, one 32-column atom per group of 8 K rows: byte
// offset of the 16-byte chunk holding columns n0..n0+7 of K row r
__device__ __forceinline__ uint32_t b_off32c(int r, int n0)
{
    return (uint32_t)((r >> 3) * kGtBSbo + (r & 7) * 64 + ((((n0 & 31) >> 3) ^ ((r & 7) >> 1)) << 4));
}

struct GtState {                                     // per matrix, kept across the panel launches
    float mag_h, mag_l;                              // |det| = (mag_h + mag_l) 2^mag_e
    int mag_e, neg, sing;
    float xnorm;                                     // ||X||_inf
    int pad[2];
};

struct GtLayout {                                    // scratch of one matrix
    size_t w, a, b, e, f, pp, used, piv, state, per;
};

__host__ __device__ inline size_t gt_al(size_t x) { return (x + 255) & ~(size_t)255; }

// row stride of the float-pair work matrix: n rounded up to even, so that every row and
// every 32-column segment of it starts on a 16-byte boundary (the bulk copies' rule)
__host__ __device__ inline int gt_ld(int n) { return (n + 1) & ~1; }

__host__ __device__ inline GtLayout gt_layout(int n)
{
    const size_t nt = (size_t)(n + 127) / 128, nc = (size_t)(n + kGtN - 1) / kGtN;
    GtLayout L;
    size_t o = 0;
    L.w = o; o += gt_al(8 * (size_t)n * gt_ld(n));     // the float-pair work matrix [n][gt_ld(n)]
    L.a = o; o += nt * kGtSl * kGtAPlane;             // [row tile][slice] planes of P
    L.b = o; o += nc * kGtSl * kGtBPlane;             // [column tile][slice] planes of U
    L.e = o; o += gt_al(4 * nt * 128);                // E_i
    L.f = o; o += gt_al(4 * nt * 128);                // F_j
    L.pp = o; o += gt_al(2 * (size_t)n);              // pivot row of each column
    L.used = o; o += gt_al(2 * (size_t)n);            // row already a pivot
    L.piv = o; o += gt_al((size_t)n);                 // row is a pivot of the current panel
    L.state = o; o += 256;
    L.per = gt_al(o);
    return L;
}

struct GtJobs {
    GjJob j[2];
    unsigned char *scr[2];                           // scratch of matrix m: scr + m * per
    int nj;
    int jb;                                          // current panel
    unsigned long long wait_ns;                      // limit of each wait (WaitCfg)
    int expire_m;                                    // test hook: matrix whose first update wait runs out
    CUtensorMap tmw[2];                              // the work matrices of job q as [matrix][row][column]
};

// Float-pair copy of X and ||X||_inf; a cluster of CTAs shares a matrix's rows where the matrices
// are few.  Both this kernel and k_gt_final only move data, but were bound by the FP64 pipe's
// conversions; on the integer pipes (f64_bits.cuh), 4096 matrices of 528 rows: 8.5 -> 3.8 ms
// (18.3 GB, 4.9 TB/s); 74 matrices, spread: 0.69 -> 0.11 ms.
__global__ void __launch_bounds__(kGtThreads) k_gt_init(GtJobs js)
{
    cg::cluster_group cluster = cg::this_cluster();
    const int nrank = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const GjJob &J = js.j[blockIdx.y];
    const int m = blockIdx.x / nrank;
    if (m >= J.count) return;                            // (the same for a whole cluster)
    const int n = J.n;
    const GtLayout L = gt_layout(n);
    unsigned char *sc = js.scr[blockIdx.y] + (size_t)m * L.per;
    const double *__restrict__ X = J.X + (size_t)m * J.x_stride;
    float2 *__restrict__ Wk = reinterpret_cast<float2 *>(sc + L.w);
    const int ld = gt_ld(n);
    short *used = reinterpret_cast<short *>(sc + L.used);
    unsigned char *piv = sc + L.piv;
    __shared__ float red_f[kGtWarps];
    __shared__ float s_max;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    float rmax = 0.f;
    for (int i = rank * kGtWarps + wid; i < n; i += nrank * kGtWarps) {
        float rs = 0.f;
#pragma unroll 4
        for (int c = lane; c < n; c += 32) {
            const float2 v = split_f64(X[(size_t)i * n + c]);
            Wk[(size_t)i * ld + c] = v;
            rs += fabsf(v.x);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) rs += __shfl_xor_sync(0xffffffffu, rs, o);
        rmax = fmaxf(rmax, rs);
    }
    if (lane == 0) red_f[wid] = rmax;
    if (rank == 0)
        for (int i = t; i < n; i += kGtThreads) {
            used[i] = 0;
            piv[i] = 0;
        }
    __syncthreads();
    if (t == 0) {
        float xm = 0.f;
        for (int q = 0; q < kGtWarps; ++q) xm = fmaxf(xm, red_f[q]);
        s_max = xm;
    }
    if (nrank > 1) cluster.sync();
    if (t == 0 && rank == 0) {
        float xm = s_max;
        for (int r = 1; r < nrank; ++r) xm = fmaxf(xm, *cluster.map_shared_rank(&s_max, r));
        GtState s0;
        s0.mag_h = 1.f; s0.mag_l = 0.f; s0.mag_e = 0; s0.neg = 0; s0.sing = 0; s0.xnorm = xm;
        s0.pad[0] = s0.pad[1] = 0;
        *reinterpret_cast<GtState *>(sc + L.state) = s0;
    }
    if (nrank > 1) cluster.sync();                       // no CTA leaves before its maximum is read
}

// Operand B of the update: the pivot rows before the update (zero in the panel's columns and for
// c >= w), scaled per column: first the column exponents (one thread per column, its 32 values
// loaded at once), then the slices (8 columns of one pivot row per thread, 16-byte stores).
__device__ __forceinline__ void gt_operand_b(unsigned char *sc, const GtLayout &L, int n, int jb, int w,
                                             const short *ppS)
{
    const float2 *__restrict__ Wk = reinterpret_cast<const float2 *>(sc + L.w);
    const int ld = gt_ld(n);
    int *Fcol = reinterpret_cast<int *>(sc + L.f);
    unsigned char *Bpl = sc + L.b;
    for (int col = threadIdx.x; col < n; col += blockDim.x) {
        const bool vcol = !(col >= jb && col < jb + w);
        float mx = 0.f;
#pragma unroll
        for (int c = 0; c < kGtB; ++c) mx = fmaxf(mx, (vcol && c < w) ? fabsf(Wk[(size_t)ppS[c] * ld + col].x) : 0.f);
        Fcol[col] = exp_bound(mx);
    }
    __syncthreads();
    const int nch = (n + 7) / 8;
    for (int it = threadIdx.x; it < kGtB * nch; it += blockDim.x) {
        const int c = it / nch, col0 = (it - c * nch) * 8;
        uint32_t o[kGtSl][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float s7[2][kGtSl];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int col = col0 + 2 * q + h;
                const bool v = c < w && col < n && !(col >= jb && col < jb + w);
                slice_n<kGtSl>(v ? Wk[(size_t)ppS[c] * ld + col] : make_float2(0.f, 0.f), col < n ? Fcol[col] : 0, s7[h]);
            }
#pragma unroll
            for (int j = 0; j < kGtSl; ++j) o[j][q] = bf16_pair(s7[0][j], s7[1][j]);
        }
        unsigned char *b = Bpl + (size_t)(col0 / kGtN) * kGtSl * kGtBPlane + b_off32c(c, col0 % kGtN);
#pragma unroll
        for (int j = 0; j < kGtSl; ++j)
            *reinterpret_cast<uint4 *>(b + (size_t)j * kGtBPlane) = make_uint4(o[j][0], o[j][1], o[j][2], o[j][3]);
    }
}

// |x| as an integer that orders like it; 0 for NaN (never a pivot) and 0
__device__ __forceinline__ unsigned gt_key(float x)
{
    const unsigned b = __float_as_uint(x) & 0x7fffffffu;
    return b > 0x7f800000u ? 0u : b;
}

// The largest key of a warp and the smallest index that has it, in every lane.
__device__ __forceinline__ void gt_warp_max(unsigned &k, int &i)
{
    const unsigned m = __reduce_max_sync(0xffffffffu, k);
    i = (int)__reduce_min_sync(0xffffffffu, k == m ? (unsigned)i : 0x7fffffffu);
    k = m;
}

__device__ __forceinline__ float2 gt_neg2(float2 a) { return make_float2(-a.x, -a.y); }

// ff::fma2 for two values at once (packed FP32, the same roundings): (ah, al) + (xh, xl) (yh, yl)
__device__ __forceinline__ void gt_fma2x2(float2 &ah, float2 &al, float2 xh, float2 xl, float2 yh, float2 yl)
{
    const float2 p = __fmul2_rn(xh, yh);
    float2 pe = __ffma2_rn(xh, yh, gt_neg2(p));
    pe = __ffma2_rn(xh, yl, pe);
    pe = __ffma2_rn(xl, yh, pe);
    const float2 s = __fadd2_rn(ah, p), bb = __fadd2_rn(s, gt_neg2(ah));
    float2 se = __fadd2_rn(__fadd2_rn(ah, gt_neg2(__fadd2_rn(s, gt_neg2(bb)))), __fadd2_rn(p, gt_neg2(bb)));
    se = __fadd2_rn(se, __fadd2_rn(al, pe));
    ah = __fadd2_rn(s, se);
    al = __fadd2_rn(se, gt_neg2(__fadd2_rn(ah, gt_neg2(s))));
}

// ff::two_sum for two values at once
__device__ __forceinline__ void gt_two_sum2(float2 a, float2 b, float2 &s, float2 &e)
{
    s = __fadd2_rn(a, b);
    const float2 bb = __fadd2_rn(s, gt_neg2(a));
    e = __fadd2_rn(__fadd2_rn(a, gt_neg2(__fadd2_rn(s, gt_neg2(bb)))), __fadd2_rn(b, gt_neg2(bb)));
}

__device__ __forceinline__ float2 gt_dup(float x) { return make_float2(x, x); }

// The panel kernel: one thread per row.  The 32 columns are eliminated in four sub-panels of 8,
// whose columns sit in the thread's registers: each pivot step updates only those 8 columns (the
// pivot column becomes the column of the step's Gauss-Jordan transformation); the other 24 lie
// in shared memory (pairs of columns {h, h', l, l'}, rows of 12 x 16 bytes, swizzled) and take
// the sub-panel's 8 pivots afterwards, two column pairs at a time in packed FP32; then the
// registers change places with the next sub-panel's columns.
//
// kSeq = false (up to kGtSeqMin - 1 rows): the sub-panel's composed transformation T = I + W S (W:
// the 8 transformation columns, S: the 8 pivot rows from before the sub-panel) as one rank-8 update,
//   X[i][j] <- [i not a pivot of the sub-panel] X[i][j] + sum_k W[i][k] X[p_k][j].
// kSeq = true: the 8 steps one after the other, X[i][j] <- X[i][j] - X[i][p_k's column] prow_k[j] with
// the multipliers of each step kept in registers and the scaled pivot rows prow_k formed by 24
// threads in step order: the roundings of a column-by-column elimination.  (The two differ in their
// last bits, which an ill-conditioned matrix amplifies; each size keeps the one that it has had.)
//
// What bounds it is the FP32 pipe (15 operations per float-float multiply-add) and the chain of a
// step: a REDUX search for the pivot (first of the rows not used yet with the largest |entry|), two
// barriers, the pivot row scaled by its owner's warp.  Up to 544 rows, two CTAs fit on an SM (2 x
// 107 KB, 56 registers a thread): one runs in the other's waits; for no more matrices than SMs, one
// with 92 registers.  Measured: 4096 matrices of 528 rows, 17 panels, 54.0 (a warp per row) -> 47.6
// (one CTA per SM) -> 42.0 ms (two); 74 of 528 rows 1.77 ms with one, 2.05 with two; 1024 of 866 rows,
// 28 panels, 55.5 -> 35.2 ms.
constexpr int kGtSeqMin = 545;
constexpr int kGpSub = 8;
constexpr int kGpLd = 12;                                // float4 per shared-memory row
// float4 j of row r lies at j ^ gp_sw(r): conflict-free without padding
__device__ __forceinline__ int gp_sw(int r) { return (r >> 1) & 3; }

template <int kMaxT, bool kSeq, int kCtas>
__global__ void __launch_bounds__(kMaxT, kCtas) k_gt_panel(GtJobs js)
{
    const GjJob &J = js.j[blockIdx.y];
    const int m = blockIdx.x;
    const int n = J.n, jb = js.jb;
    if (m >= J.count || jb >= n) return;
    const GtLayout L = gt_layout(n);
    unsigned char *sc = js.scr[blockIdx.y] + (size_t)m * L.per;
    GtState *st = reinterpret_cast<GtState *>(sc + L.state);
    if (st->sing) return;
    float2 *__restrict__ Wk = reinterpret_cast<float2 *>(sc + L.w);
    const int ld = gt_ld(n);
    short *pp_g = reinterpret_cast<short *>(sc + L.pp);
    short *used_g = reinterpret_cast<short *>(sc + L.used);
    unsigned char *piv_g = sc + L.piv;

    extern __shared__ __align__(16) unsigned char gp_smem[];
    __shared__ float4 U_s[kGpSub][12];                    // pivot rows of the sub-panel, other columns
    __shared__ float2 raw_s[kGpSub], prow_s[kGpSub];      // the step's pivot row on the sub-panel: raw, scaled
    __shared__ float2 pinv_s[kGpSub], mul_s[kGpSub][kGpSub];   // kSeq: 1 / pivot, multipliers of the pivot rows
    __shared__ short ppS[kGtB];
    __shared__ unsigned red_k[kMaxT / 32];
    __shared__ int red_i[kMaxT / 32];
    __shared__ GtState S_s;

    const int t = threadIdx.x, lane = t & 31, wid = t >> 5, nwarps = blockDim.x >> 5;
    const int w = min(kGtB, n - jb);
    const int i = t;                                      // this thread's row
    const bool row_ok = i < n;
    float4 *P = reinterpret_cast<float4 *>(gp_smem), *row = P + (size_t)t * kGpLd;
    const int sw = gp_sw(t);
    // the previous panel's pivots stop being pivots of the current panel
    if (jb > 0 && t < kGtB) piv_g[pp_g[jb - kGtB + t]] = 0;
    float2 xh[4], xl[4];                                  // the sub-panel's columns 2 q, 2 q + 1 of this row
    {
        const float2 *src = Wk + (size_t)(row_ok ? i : 0) * ld + jb;
#pragma unroll
        for (int q = 0; q < kGtB / 2; ++q) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row_ok && w == kGtB) v = *reinterpret_cast<const float4 *>(src + 2 * q);
            else if (row_ok) {
                if (2 * q < w) { v.x = src[2 * q].x; v.y = src[2 * q].y; }
                if (2 * q + 1 < w) { v.z = src[2 * q + 1].x; v.w = src[2 * q + 1].y; }
            }
            if (q < 4) {
                xh[q] = make_float2(v.x, v.z);
                xl[q] = make_float2(v.y, v.w);
            } else {
                row[(q - 4) ^ sw] = make_float4(v.x, v.z, v.y, v.w);
            }
        }
    }
    bool used = !row_ok || used_g[i] != 0;
    if (t == (int)blockDim.x - 32) S_s = *st;             // (read and written by this thread only)
    bool sing = false;
    auto elem = [&](int c) { return (c & 1) ? make_float2(xh[c >> 1].y, xl[c >> 1].y) : make_float2(xh[c >> 1].x, xl[c >> 1].x); };

#pragma unroll 1
    for (int sb = 0; sb < kGtB / kGpSub && sb * kGpSub < w; ++sb) {
        const int c0 = sb * kGpSub;
        const int nk = min(kGpSub, w - c0);               // pivots of this sub-panel
        int my_k = -1;                                    // this row's step, if it is one of them
        float2 mf[kSeq ? kGpSub : 1];                     // kSeq: the row's multiplier of each step
#pragma unroll
        for (int cc = 0; cc < kGpSub; ++cc) {
            if (cc >= nk) break;
            // block-wide argmax of |x[c]| over the rows not used yet
            const float2 xc = elem(cc);
            unsigned k = used ? 0u : gt_key(xc.x);
            int p = used ? n : i;
            gt_warp_max(k, p);
            if (lane == 0) { red_k[wid] = k; red_i[wid] = p; }
            __syncthreads();
            k = lane < nwarps ? red_k[lane] : 0u;
            p = lane < nwarps ? red_i[lane] : n;
            gt_warp_max(k, p);
            if (k == 0u) {                                // every warp sees the same candidates
                sing = true;
                break;
            }
            if (wid == p >> 5) {                          // the pivot row, scaled a column per lane
                if (i == p) {
#pragma unroll
                    for (int q = 0; q < kGpSub; ++q) raw_s[q] = elem(q);
                    used = true;
                    my_k = cc;
                }
                __syncwarp();
                const float2 pinv = ff::inv(raw_s[cc]);
                if (lane < kGpSub) prow_s[lane] = lane == cc ? pinv : ff::mul(raw_s[lane], pinv);
                if (lane == 0) {
                    ppS[c0 + cc] = (short)p;
                    if (kSeq) pinv_s[cc] = pinv;
                }
            }
            __syncthreads();
            if (t == (int)blockDim.x - 32) {              // (the last warp has the fewest rows)
                const float2 pv = raw_s[cc];
                const float2 a = pv.x < 0.f ? ff::neg(pv) : pv;
                const float2 mg = ff::mul(make_float2(S_s.mag_h, S_s.mag_l), a);
                int ex;
                frexpf(mg.x, &ex);
                S_s.mag_h = ldexpf(mg.x, -ex);
                S_s.mag_l = ldexpf(mg.y, -ex);
                S_s.mag_e += ex;
                S_s.neg ^= pv.x < 0.f;
            }
            // the step on the sub-panel's 8 columns: the pivot column starts from zero
            const float2 f = ff::neg(xc);
            if constexpr (kSeq) mf[cc] = f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 y0 = prow_s[2 * q], y1 = prow_s[2 * q + 1];
                const float2 yh = make_float2(y0.x, y1.x), yl = make_float2(y0.y, y1.y);
                if (i == p) {
                    xh[q] = yh;
                    xl[q] = yl;
                } else {
                    if (2 * q == cc) xh[q].x = xl[q].x = 0.f;
                    if (2 * q + 1 == cc) xh[q].y = xl[q].y = 0.f;
                    gt_fma2x2(xh[q], xl[q], gt_dup(f.x), gt_dup(f.y), yh, yl);
                }
            }
        }
        if (sing) break;
        // the pivot rows' other columns, from before the sub-panel
        for (int q = t; q < nk * 12; q += blockDim.x) {
            const int p = ppS[c0 + q / 12];
            U_s[q / 12][q % 12] = P[p * kGpLd + ((q % 12) ^ gp_sw(p))];
        }
        if constexpr (kSeq)
            if (my_k >= 0)
#pragma unroll
                for (int c = 0; c < kGpSub; ++c) mul_s[my_k][c] = mf[c];
        __syncthreads();
        if constexpr (kSeq) {
            // prow_k of the other columns, in step order: one thread per column
            if (t < 24) {
                float *u = reinterpret_cast<float *>(&U_s[0][t >> 1]) + (t & 1);
                float2 pr[kGpSub];
#pragma unroll
                for (int k = 0; k < kGpSub; ++k) {
                    if (k >= nk) break;
                    float2 v = make_float2(u[k * 48], u[k * 48 + 2]);
#pragma unroll
                    for (int c = 0; c < k; ++c) v = ff::fma2(v, mul_s[k][c], pr[c]);
                    pr[k] = ff::mul(v, pinv_s[k]);
                    u[k * 48] = pr[k].x;
                    u[k * 48 + 2] = pr[k].y;
                }
            }
            __syncthreads();
        }
        // the sub-panel's pivots on the other 24 columns of this row
        const bool any_piv = __any_sync(0xffffffffu, my_k >= 0);
#pragma unroll 1
        for (int j = 0; j < 12; j += 2) {
            float4 a0 = row[j ^ sw], a1 = row[(j + 1) ^ sw];
            if (!kSeq && my_k >= 0) a0 = a1 = make_float4(0.f, 0.f, 0.f, 0.f);
            float2 h0 = make_float2(a0.x, a0.y), l0 = make_float2(a0.z, a0.w);
            float2 h1 = make_float2(a1.x, a1.y), l1 = make_float2(a1.z, a1.w);
#pragma unroll
            for (int k = 0; k < kGpSub; ++k) {
                if (k >= nk) break;
                const float4 u0 = U_s[k][j], u1 = U_s[k][j + 1];
                const float2 f = kSeq ? mf[kSeq ? k : 0] : elem(k);
                gt_fma2x2(h0, l0, gt_dup(f.x), gt_dup(f.y), make_float2(u0.x, u0.y), make_float2(u0.z, u0.w));
                gt_fma2x2(h1, l1, gt_dup(f.x), gt_dup(f.y), make_float2(u1.x, u1.y), make_float2(u1.z, u1.w));
                if (kSeq && any_piv && my_k == k) {       // the pivot row of step k becomes prow_k
                    h0 = make_float2(u0.x, u0.y); l0 = make_float2(u0.z, u0.w);
                    h1 = make_float2(u1.x, u1.y); l1 = make_float2(u1.z, u1.w);
                }
            }
            row[j ^ sw] = make_float4(h0.x, h0.y, l0.x, l0.y);
            row[(j + 1) ^ sw] = make_float4(h1.x, h1.y, l1.x, l1.y);
        }
        // the registers change places with the next sub-panel's columns: area sb of the row (4 column
        // pairs) then holds this one's
        if (sb < kGtB / kGpSub - 1) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 v = row[(4 * sb + q) ^ sw];
                row[(4 * sb + q) ^ sw] = make_float4(xh[q].x, xh[q].y, xl[q].x, xl[q].y);
                xh[q] = make_float2(v.x, v.y);
                xl[q] = make_float2(v.z, v.w);
            }
        }
    }
    if (sing) {
        if (t == 0) st->sing = 1;
        return;
    }
    // a short last panel leaves the loop early: the areas from its last sub-panel on still hold
    // the columns after it, in order; those columns are all zero and not stored
    const int last = min((w + kGpSub - 1) / kGpSub, kGtB / kGpSub) - 1;      // last sub-panel eliminated
    const int swaps = min(last + 1, kGtB / kGpSub - 1);
    // column pair q of the panel: area q / 4 before the swaps' end, the registers after
    auto pair_at = [&](int q) {
        const int g = q >> 2;
        if (g < swaps) return row[q ^ sw];
        if (g == swaps) return make_float4(xh[q & 3].x, xh[q & 3].y, xl[q & 3].x, xl[q & 3].y);
        return row[(q - 4) ^ sw];
    };
    // the eliminated panel is part of the result; operand A: the row scaled by its exponent, seven
    // slices, [row tile][slice] planes, 16-byte chunks of 8 columns
    if (row_ok) {
        float mx = 0.f;
        float2 *dst = Wk + (size_t)i * ld + jb;
#pragma unroll
        for (int q = 0; q < kGtB / 2; ++q) {
            const float4 v = pair_at(q);
            mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
            if (w == kGtB) *reinterpret_cast<float4 *>(dst + 2 * q) = make_float4(v.x, v.z, v.y, v.w);
            else {
                if (2 * q < w) dst[2 * q] = make_float2(v.x, v.z);
                if (2 * q + 1 < w) dst[2 * q + 1] = make_float2(v.y, v.w);
            }
        }
        const int E = exp_bound(mx);
        reinterpret_cast<int *>(sc + L.e)[i] = E;
        unsigned char *base = sc + L.a + (size_t)(i >> 7) * kGtSl * kGtAPlane;
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
            uint32_t o[kGtSl][4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 v = pair_at(4 * ch + q);
                float s0[kGtSl], s1[kGtSl];
                slice_n<kGtSl>(make_float2(v.x, v.z), E, s0);
                slice_n<kGtSl>(make_float2(v.y, v.w), E, s1);
#pragma unroll
                for (int j = 0; j < kGtSl; ++j) o[j][q] = bf16_pair(s0[j], s1[j]);
            }
#pragma unroll
            for (int j = 0; j < kGtSl; ++j)
                *reinterpret_cast<uint4 *>(base + (size_t)j * kGtAPlane + a_off64(i & 127, ch)) =
                    make_uint4(o[j][0], o[j][1], o[j][2], o[j][3]);
        }
    }
    // bookkeeping of the pivots
    if (t < w) {
        const int p = ppS[t];
        pp_g[jb + t] = (short)p;
        used_g[p] = 1;
        piv_g[p] = 1;
    }
    if (t == (int)blockDim.x - 32) *st = S_s;
    gt_operand_b(sc, L, n, jb, w, ppS);
}

static_assert(kGtN == kGtB, "a column tile of the update is exactly one panel");

// Bounded wait of one thread with the CTA's abort flag: false on timeout (which sets the
// flag) or as soon as another role has set it.
__device__ __forceinline__ bool gt_wait1(uint32_t mbar, uint32_t parity, uint64_t limit_ns, volatile int *abort)
{
    const uint64_t t0 = globaltimer();
    while (true) {
        if (mbar_try_wait(mbar, parity)) return true;
        if (*abort) return false;
        if (globaltimer() - t0 > limit_ns) {
            *abort = 1;
            return false;
        }
    }
}

// The same for a whole warp, which stays converged: every lane polls (the phase, once
// complete, stays complete until this warp has arrived for it), the decisions are taken
// together.  A warp left diverged here (one lane polling, the others parked) made each
// following elect.sync -- the MMA warp issues every MMA through one -- cost ~300 cycles.
__device__ __forceinline__ bool gt_wait_warp(uint32_t mbar, uint32_t parity, uint64_t limit_ns, volatile int *abort,
                                             int lane)
{
    const uint64_t t0 = globaltimer();
    while (true) {
        const bool done = mbar_try_wait(mbar, parity);
        if (__all_sync(0xffffffffu, done)) return true;
        if (__any_sync(0xffffffffu, *abort != 0)) return false;
        int late = lane == 0 && globaltimer() - t0 > limit_ns;
        late = __shfl_sync(0xffffffffu, late, 0);
        if (late) {
            if (lane == 0) *abort = 1;
            return false;
        }
    }
}

// A few CTAs per matrix (launch_gj_tc says how many), one CTA per SM, each over every gridDim.x-th
// tile of 128 rows, four roles:
//   X warp          the tile's old float pairs in and the updated ones out by tensor TMA
//                   (two 16-column boxes of 128 rows each way, 128-byte swizzle; rows and
//                   columns outside the matrix are zero-filled on load, clipped on store),
//                   three stages
//   B warp          bulk copies of each column tile's 7 pivot-row slice planes, three stages
//   MMA warp        the row tile's 7 panel planes (one bulk copy), then per column tile the
//                   2 K16 x 28 slice-pair MMAs into the seven accumulators (7 x 32 TMEM
//                   columns) once the epilogue has read the previous tile's
//   16 epilogue     TMEM lane quadrant x 8 columns: the seven order sums, the old values
//   warps           read from and the results written back to the stage in shared memory;
//                   warps 0..3 move the panel planes, half a row tile ahead, into one of two
//                   places in TMEM, where the MMAs read them (A from TMEM: per MMA only the 1 KB B slice is read from shared
//                   memory, instead of 4 KB of A + 1 KB of B, which bounded the MMAs)
// The panel's own column tile is final and skipped.  Every wait is bounded; one that runs
// out sets the CTA's abort flag and every role leaves at its next wait; the matrix goes to
// the FP64 recomputation, and the copies and MMAs in flight drain before TMEM is freed.
__global__ void __launch_bounds__(kGtUpThreads, 1) k_gt_update(const __grid_constant__ GtJobs js, int z0)
{
    extern __shared__ __align__(1024) unsigned char gt_smem[];
    unsigned char *base = gt_smem + ((1024 - (smem_u32(gt_smem) & 1023)) & 1023);
    constexpr int kBars = 2 + 2 * kGtBs + 2 * kGtXs + 2;
    __shared__ __align__(8) uint64_t bar[kBars];
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort, s_never;

    const int z = z0 + blockIdx.z;
    const int q = z % js.nj, m = z / js.nj;
    const GjJob &J = js.j[q];
    const int n = J.n, jb = js.jb;
    // this CTA's row tiles: blockIdx.x, + gridDim.x, ...
    const int rt0 = blockIdx.x, drt = gridDim.x;
    if (m >= J.count || jb >= n || rt0 * 128 >= n) return;
    const int nrt = ((n + 127) / 128 - rt0 + drt - 1) / drt;
    const int nc = (n + kGtN - 1) / kGtN;
    const int jp = jb / kGtN;                                    // the panel's own column tile
    const int ntl = nc - 1;                                      // column tiles updated
    if (ntl == 0) return;
    const GtLayout L = gt_layout(n);
    unsigned char *sc = js.scr[q] + (size_t)m * L.per;
    const GtState *st = reinterpret_cast<const GtState *>(sc + L.state);
    if (st->sing) return;
    const int nseq = nrt * ntl;                                  // tiles of this CTA, row tile by row tile
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const uint64_t tmap = reinterpret_cast<uint64_t>(&js.tmw[q]);

    unsigned char *As = base;                                    // 7 x 8 KB
    unsigned char *Bs = As + kGtSl * kGtAPlane;                  // 3 x 7 x 2 KB
    unsigned char *Xs = Bs + kGtBs * kGtSl * kGtBPlane;          // 3 x 2 x 16 KB
    int *Fs = reinterpret_cast<int *>(Xs + kGtXs * kGtXStage);   // [nc * 32] column exponents F_j
    float *Fsc = reinterpret_cast<float *>(Fs + nc * kGtN);      // [nc * 32] 2^F_j where |F_j| <= 60, else 0
    const uint32_t b0 = smem_u32(&bar[0]);
    const uint32_t bA = b0;
    auto BF = [&](int sb) { return b0 + 8u * (uint32_t)(1 + sb); };
    auto BE = [&](int sb) { return b0 + 8u * (uint32_t)(1 + kGtBs + sb); };
    auto XF = [&](int sx) { return b0 + 8u * (uint32_t)(1 + 2 * kGtBs + sx); };
    auto XW = [&](int sx) { return b0 + 8u * (uint32_t)(1 + 2 * kGtBs + kGtXs + sx); };
    const uint32_t bTF = b0 + 8u * (uint32_t)(1 + 2 * kGtBs + 2 * kGtXs);   // accumulators complete
    const uint32_t bTE = bTF + 8u;                                         // ... and read
    const uint32_t bAT = bTF + 16u;                                        // panel slices in TMEM
    auto col_tile = [&](int i) { return i < jp ? i : i + 1; };

    const int *Fcol = reinterpret_cast<const int *>(sc + L.f);
    // a tile whose column exponents all lie in [-60, 60] takes the fast scaling in the epilogue
    __shared__ int tile_ok[1024 / kGtN];
    if (t < 1024 / kGtN) tile_ok[t] = 1;
    __syncthreads();
    for (int c = t; c < nc * kGtN; c += kGtUpThreads) {
        const int F = c < n ? Fcol[c] : 0;
        const bool in = F >= -60 && F <= 60;
        Fs[c] = F;
        Fsc[c] = in ? __int_as_float((127 + F) << 23) : 0.f;
        if (!in) tile_ok[c / kGtN] = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;"
                     :: "r"(smem_u32(&tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (t == 32) {
        mbar_init(bA, 1);
        for (int sb = 0; sb < kGtBs; ++sb) { mbar_init(BF(sb), 1); mbar_init(BE(sb), 1); }
        for (int sx = 0; sx < kGtXs; ++sx) { mbar_init(XF(sx), 1); mbar_init(XW(sx), kGtEpWarps); }
        mbar_init(bTF, 1);
        mbar_init(bTE, kGtEpWarps);
        mbar_init(bAT, 4);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
        s_never = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    int nld = 0, nb = 0, nmma = 0, na = 0;                       // tiles loaded / copied / multiplied, row tiles of A loaded

    if (warp == kGtEpWarps) {
        // ---- X warp: stage sx holds tile i; before tile i + 3 is loaded into it, tile i is
        // stored and the store has finished reading the stage
        if (lane == 0) {
            struct Tile { int i, r0; };                          // column tile number, first row
            auto next = [&](Tile &c) { if (++c.i == ntl) { c.i = 0; c.r0 += drt * 128; } };
            auto store = [&](int sx, const Tile &c) {
                const uint32_t xs = smem_u32(Xs + sx * kGtXStage);
                const int c0 = col_tile(c.i) * kGtN;
                tma_store_3d(tmap, xs, c0, c.r0, m);
                tma_store_3d(tmap, xs + kGtXStage / 2, c0 + 16, c.r0, m);
                bulk_commit();
            };
            Tile ld = {0, rt0 * 128}, sd = ld;                   // the next tile to load, to store
            for (int q = 0; q < nseq; ++q) {
                const int sx = q % kGtXs;
                if (q >= kGtXs) {
                    if (!gt_wait1(XW(sx), ((q / kGtXs) - 1) & 1, js.wait_ns, &s_abort)) break;
                    store(sx, sd);
                    next(sd);
                    bulk_wait_read0();
                }
                const uint32_t xs = smem_u32(Xs + sx * kGtXStage);
                const int c0 = col_tile(ld.i) * kGtN;
                mbar_expect_tx(XF(sx), kGtXStage);
                tma_load_3d(tmap, xs, c0, ld.r0, m, XF(sx));
                tma_load_3d(tmap, xs + kGtXStage / 2, c0 + 16, ld.r0, m, XF(sx));
                next(ld);
                nld = q + 1;
            }
            if (nld == nseq)
                for (int q = max(0, nseq - kGtXs); q < nseq; ++q) {
                    if (!gt_wait1(XW(q % kGtXs), (q / kGtXs) & 1, js.wait_ns, &s_abort)) break;
                    store(q % kGtXs, sd);
                    next(sd);
                }
            bulk_wait_all0();                                    // every store complete
        }
    } else if (warp == kGtEpWarps + 1) {
        // ---- B warp
        if (lane == 0)
            for (int q = 0, i = 0; q < nseq; ++q, i = i + 1 == ntl ? 0 : i + 1) {
                const int sb = q % kGtBs;
                if (q >= kGtBs && !gt_wait1(BE(sb), ((q / kGtBs) - 1) & 1, js.wait_ns, &s_abort)) break;
                mbar_expect_tx(BF(sb), kGtSl * kGtBPlane);
                bulk_g2s(smem_u32(Bs + sb * kGtSl * kGtBPlane), sc + L.b + (size_t)col_tile(i) * kGtSl * kGtBPlane,
                         kGtSl * kGtBPlane, BF(sb));
                nb = q + 1;
            }
    } else if (warp == kGtEpWarps + 2) {
        // ---- MMA warp: warp-uniform control flow, one elected lane issues each MMA and commit
        auto load_a = [&](int it) {                              // the row tile's panel planes
            if (lane == 0) {
                mbar_expect_tx(bA, kGtSl * kGtAPlane);
                bulk_g2s(smem_u32(As), sc + L.a + (size_t)(rt0 + it * drt) * kGtSl * kGtAPlane, kGtSl * kGtAPlane, bA);
            }
            na = it + 1;
            __syncwarp();
        };
        load_a(0);
        const uint32_t idesc = umma_idesc_f16(128, kGtN, 1);
        bool ok = true;
        for (int it = 0; it < nrt && ok; ++it) {
            if (!gt_wait_warp(bAT, it & 1, js.wait_ns, &s_abort, lane)) break;
            if (it + 1 < nrt) load_a(it + 1);                    // the planes are in TMEM: their stage is free
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t atm = tmem + kGtATmem + (uint32_t)((it & 1) * kGtAtCols);
            for (int i = 0; i < ntl; ++i) {
                const int q = it * ntl + i, sb = q % kGtBs;
                if (!gt_wait_warp(BF(sb), (q / kGtBs) & 1, js.wait_ns, &s_abort, lane)) { ok = false; break; }
                if (q >= 1 && !gt_wait_warp(bTE, (q - 1) & 1, js.wait_ns, &s_abort, lane)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t dB = umma_desc_sw64_mn(smem_u32(Bs + sb * kGtSl * kGtBPlane), kGtBSbo, kGtBSbo);
#pragma unroll
                for (int kk = 0; kk < kGtB / 16; ++kk)
#pragma unroll
                    for (int d = 0; d < kGtSl; ++d)
#pragma unroll
                        for (int ii = 0; ii <= d; ++ii) {
                            const int j = d - ii;
                            const uint32_t at = atm + (uint32_t)((ii * 2 + kk) * 8);
                            const uint64_t bd = dB + ((j * kGtBPlane + 2 * kk * kGtBSbo) >> 4);
                            if (kk == 0 && ii == 0) umma_bf16_ts_warp<0>(tmem + d * kGtN, at, bd, idesc);
                            else umma_bf16_ts_warp<1>(tmem + d * kGtN, at, bd, idesc);
                        }
                umma_commit_warp(BE(sb));                        // the B stage may be refilled
                umma_commit_warp(bTF);                           // the accumulators may be read
                nmma = q + 1;
            }
        }
    } else {
        // ---- epilogue warps: row r of the tile (TMEM lane), columns cg * 8 .. + 7 of each column tile
        const int quad = warp & 3, cg = warp >> 2;
        const int r = quad * 32 + lane;
        const uint32_t tlane = (uint32_t)(quad * 32) << 16;
        const uint32_t tl = tmem + tlane + (uint32_t)(cg * 8);
        // the panel planes of the CTA's row tile `it` into TMEM (two places in turn): this thread's
        // row, its 32 K values packed in pairs (the 64-byte swizzle of the shared-memory planes undone)
        auto move_a = [&](int it) {
            if (!gt_wait_warp(bA, it & 1, js.wait_ns, &s_abort, lane)) return;
#pragma unroll 1
            for (int ii = 0; ii < kGtSl; ++ii) {
                uint32_t w[16];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const uint4 u = *reinterpret_cast<const uint4 *>(As + ii * kGtAPlane + a_off64(r, c));
                    w[4 * c] = u.x; w[4 * c + 1] = u.y; w[4 * c + 2] = u.z; w[4 * c + 3] = u.w;
                }
                tmem_st16(tmem + tlane + kGtATmem + (uint32_t)((it & 1) * kGtAtCols + 16 * ii), w);
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(bAT);
        };
        // this thread's row of the row tile `it`: exponent E_i and whether it is one of the panel's
        // pivot rows; loaded a row tile ahead
        int E_nx = 0, piv_nx = 0;
        auto row_info = [&](int it) {
            const int i_row = (rt0 + it * drt) * 128 + r;
            const bool ok = i_row < n;
            E_nx = ok ? reinterpret_cast<const int *>(sc + L.e)[i_row] : 0;
            piv_nx = ok ? (sc + L.piv)[i_row] : 0;
        };
        row_info(0);
        if (warp < 4) move_a(0);
        // this thread's four 16-byte chunks of a stage (128-byte swizzle: chunk ^ (row & 7))
        const uint32_t xoff = (uint32_t)((cg >> 1) * (kGtXStage / 2) + r * 128);
        const int ck0 = (cg & 1) * 4;
        // test hook: the first panel's first wait of the chosen matrix runs out
        const bool expire = m == js.expire_m && jb == 0 && rt0 == 0;
        bool live = true;
        for (int it = 0, q = 0; it < nrt && live; ++it) {
            const int nr = min(128, n - (rt0 + it * drt) * 128);
            const int E = E_nx;
            const bool is_piv = piv_nx != 0;
            // 2^(E + F) as two exact multiplications by 2^E and 2^F when both lie in [-60, 60]: the
            // order sums are 0 or at least 2^-56 in magnitude (multiples of the smallest unit), so the
            // product with 2^E is a normal float, and the final rounding equals scale_pow2's
            const bool E_ok = E >= -60 && E <= 60;
            const float sE = __int_as_float((127 + (E_ok ? E : 0)) << 23);
            // the next row tile's planes move well before its first MMA (their place was read by the
            // MMAs of the row tile before this one, all complete)
            const int i_move = it + 1 < nrt ? ntl / 2 : -1;
            for (int i = 0; i < ntl; ++i, ++q) {
                if (i == i_move) {
                    row_info(it + 1);
                    if (warp < 4) move_a(it + 1);
                }
                const int sx = q % kGtXs;
                bool ok;
                if (expire && q == 0) {
                    int f = 0;
                    if (lane == 0) {
                        f = flag_wait(&s_never, js.wait_ns);
                        if (!f) s_abort = 1;
                    }
                    ok = __shfl_sync(0xffffffffu, f, 0) != 0;
                } else {
                    ok = gt_wait_warp(bTF, q & 1, js.wait_ns, &s_abort, lane);
                }
                if (!ok) { live = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (quad * 32 >= nr) {                               // a ragged tile's warp without rows
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bTE);
                    if (!gt_wait_warp(XF(sx), (q / kGtXs) & 1, js.wait_ns, &s_abort, lane)) { live = false; break; }
                    if (lane == 0) mbar_arrive(XW(sx));
                    continue;
                }
                uint32_t v[kGtSl][8];
#pragma unroll
                for (int d = 0; d < kGtSl; ++d) tmem_ld8_async(tl + (uint32_t)(d * kGtN), v[d]);
                tmem_wait_ld(v);
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(bTE);
                // the seven order sums, exact integers in their units: orders 0..3 added as float
                // pairs, orders 4..6 (below 2^-21 of the update) first in FP32 (rounding ~2^-46);
                // two columns at a time (packed FP32)
                float2 hs[4], ls[4];
                auto ord = [&](int d, int k) {
                    return make_float2(__uint_as_float(v[d][2 * k]), __uint_as_float(v[d][2 * k + 1]));
                };
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float2 sh, se;
                    gt_two_sum2(ord(0, k), ord(1, k), hs[k], ls[k]);
                    gt_two_sum2(hs[k], ord(2, k), sh, se);
                    ls[k] = __fadd2_rn(ls[k], se);
                    gt_two_sum2(sh, ord(3, k), hs[k], se);
                    ls[k] = __fadd2_rn(ls[k], se);
                    ls[k] = __fadd2_rn(ls[k], __fadd2_rn(ord(4, k), __fadd2_rn(ord(5, k), ord(6, k))));
                }
                if (!gt_wait_warp(XF(sx), (q / kGtXs) & 1, js.wait_ns, &s_abort, lane)) { live = false; break; }
                unsigned char *xs = Xs + sx * kGtXStage + xoff;
                const int ct = col_tile(i);
                const int c0 = ct * kGtN + cg * 8;
                const bool fast = E_ok && tile_ok[ct];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float4 *p4 = reinterpret_cast<float4 *>(xs + (((ck0 + k) ^ (r & 7)) << 4));
                    float4 o = *p4;
                    if (is_piv) o = make_float4(0.f, 0.f, 0.f, 0.f);
                    float2 uh, ul;
                    if (fast) {
                        const float2 f = *reinterpret_cast<const float2 *>(Fsc + c0 + 2 * k), e2 = gt_dup(sE);
                        uh = __fmul2_rn(__fmul2_rn(hs[k], e2), f);
                        ul = __fmul2_rn(__fmul2_rn(ls[k], e2), f);
                    } else {
                        const int ex0 = E + Fs[c0 + 2 * k], ex1 = E + Fs[c0 + 2 * k + 1];
                        uh = make_float2(scale_pow2(hs[k].x, ex0), scale_pow2(hs[k].y, ex1));
                        ul = make_float2(scale_pow2(ls[k].x, ex0), scale_pow2(ls[k].y, ex1));
                    }
                    // ff::add of the old values and the update
                    const float2 xh = make_float2(o.x, o.z), xl = make_float2(o.y, o.w);
                    float2 sm, e;
                    gt_two_sum2(xh, uh, sm, e);
                    e = __fadd2_rn(e, __fadd2_rn(xl, ul));
                    const float2 h = __fadd2_rn(sm, e);
                    const float2 l = __fadd2_rn(e, gt_neg2(__fadd2_rn(h, gt_neg2(sm))));
                    *p4 = make_float4(h.x, l.x, h.y, l.y);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // for the TMA store
                __syncwarp();
                if (lane == 0) mbar_arrive(XW(sx));
            }
        }
    }
    __syncthreads();
    if (s_abort && t == 0 && J.redo) J.redo[m * J.redo_stride] = 1;   // recomputed in FP64
    // nothing may land in this CTA's shared memory or TMEM after it exits: the copying
    // threads wait for their last copies, the MMA thread for its last commits (in a normal
    // run all of these have completed or complete at once)
    if (s_abort && warp == kGtEpWarps && lane == 0)
        for (int i = max(0, nld - kGtXs); i < nld; ++i) mbar_wait(XF(i % kGtXs), (i / kGtXs) & 1, kDrainNs);
    if (s_abort && warp == kGtEpWarps + 1 && lane == 0)
        for (int i = max(0, nb - kGtBs); i < nb; ++i) mbar_wait(BF(i % kGtBs), (i / kGtBs) & 1, kDrainNs);
    if (warp == kGtEpWarps + 2 && lane == 0) {
        if (s_abort && na > 0) mbar_wait(bA, (na - 1) & 1, kDrainNs);
        for (int i = max(0, nmma - kGtBs); i < nmma; ++i) mbar_wait(BE(i % kGtBs), (i / kGtBs) & 1, kDrainNs);
        if (nmma > 0) mbar_wait(bTF, (nmma - 1) & 1, kDrainNs);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" :: "r"(tmem) : "memory");
}

// ||X^-1||_inf (the rows of X^-1 are the rows of the result, columns permuted) and
// D^-1 = X^-T in one pass over the result, 32 x 32 tiles; a cluster shares a matrix's row blocks
// where the matrices are few.  4096 matrices of 528 rows: 7.3 -> 3.7 ms;
// 74, spread: 1.12 -> 0.13 ms.
__global__ void __launch_bounds__(kGtThreads) k_gt_final(GtJobs js, double kappa_max)
{
    cg::cluster_group cluster = cg::this_cluster();
    const int nrank = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const GjJob &J = js.j[blockIdx.y];
    const int m = blockIdx.x / nrank;
    if (m >= J.count) return;                            // (the same for a whole cluster)
    const int n = J.n;
    const GtLayout L = gt_layout(n);
    unsigned char *sc = js.scr[blockIdx.y] + (size_t)m * L.per;
    const GtState S = *reinterpret_cast<const GtState *>(sc + L.state);
    if (S.sing) {                                        // a zero pivot in the float pairs: FP64 decides
        if (threadIdx.x == 0 && rank == 0 && J.redo) J.redo[m * J.redo_stride] = 1;
        return;
    }
    const float2 *__restrict__ Wk = reinterpret_cast<const float2 *>(sc + L.w);
    const int ld = gt_ld(n);
    double *__restrict__ Dout = J.Dinv + (size_t)m * J.d_stride;
    const short *pp_g = reinterpret_cast<const short *>(sc + L.pp);
    __shared__ float2 tile[2][32 * 33];
    __shared__ short pp[1024];
    __shared__ float red_f[kGtWarps];
    __shared__ float s_max;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    constexpr int RW = 32 / kGtWarps;                    // rows of a tile per warp
    for (int i = t; i < n; i += kGtThreads) pp[i] = pp_g[i];
    __syncthreads();
    float imax = 0.f;
    int buf = 0;
    for (int kb = 32 * rank; kb < n; kb += 32 * nrank) {
        float rs[RW];
        const float2 *row[RW];
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            const int k = kb + wid + r * kGtWarps;
            rs[r] = 0.f;
            row[r] = k < n ? Wk + (size_t)pp[k] * ld : nullptr;
        }
        // the tiles alternate between two buffers: one barrier each
        for (int cb = 0; cb < n; cb += 32, buf ^= 1) {
            const int c = cb + lane;
            float2 v[RW];
#pragma unroll
            for (int r = 0; r < RW; ++r) v[r] = (row[r] && c < n) ? row[r][c] : make_float2(0.f, 0.f);
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                tile[buf][(wid + r * kGtWarps) * 33 + lane] = v[r];
                if (c < n) rs[r] += fabsf(v[r].x);
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                const int cr = cb + wid + r * kGtWarps, k = kb + lane;
                if (cr < n && k < n)
                    Dout[(size_t)pp[cr] * n + k] = join_f64(tile[buf][lane * 33 + wid + r * kGtWarps]);
            }
        }
#pragma unroll
        for (int r = 0; r < RW; ++r) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) rs[r] += __shfl_xor_sync(0xffffffffu, rs[r], o);
            imax = fmaxf(imax, rs[r]);
        }
    }
    if (lane == 0) red_f[wid] = imax;
    __syncthreads();
    if (t == 0) {
        float im = 0.f;
        for (int q = 0; q < kGtWarps; ++q) im = fmaxf(im, red_f[q]);
        s_max = im;
    }
    if (nrank > 1) cluster.sync();
    if (rank == 0) {
        // parity of the row permutation k -> pp[k]: its inversions
        int inv = 0;
        for (int i = t; i < n; i += kGtThreads)
            for (int j = i + 1; j < n; ++j) inv ^= pp[j] < pp[i];
        const int par = __syncthreads_count(inv) & 1;
        if (t == 0) {
            float im = s_max;
            for (int r = 1; r < nrank; ++r) im = fmaxf(im, *cluster.map_shared_rank(&s_max, r));
            const double kappa = (double)S.xnorm * (double)im;
            const double logabs = log((double)S.mag_h + (double)S.mag_l) + S.mag_e * 0.69314718055994530942;
            if (J.logabs) J.logabs[(size_t)m * J.la_stride] = logabs;
            if (J.sign) J.sign[(size_t)m * J.la_stride] = (par ^ S.neg) ? -1.0 : 1.0;
            if (J.redo && !(kappa <= kappa_max && isfinite(logabs))) J.redo[m * J.redo_stride] = 1;
        }
    }
    if (nrank > 1) cluster.sync();                       // no CTA leaves before its maximum is read
}

// init and final: CTAs per matrix, up to 8 (the portable cluster size) while the matrices give
// fewer than eight CTAs (what an SM holds) to each of 152 SMs
template <typename... Args>
static cudaError_t gt_clusters(void (*kern)(Args...), dim3 g1, int n_jobs, cudaStream_t st, Args... args)
{
    unsigned c = 1;
    while (c < 8 && (size_t)g1.x * n_jobs * c < 152 * 8) c *= 2;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = c;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(g1.x * c, g1.y);
    cfg.blockDim = dim3(kGtThreads);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// The largest block of the panel kernel: one thread per row.
constexpr int kGtMaxRows = 896;

bool gjtc_fits(int nmax) { return nmax <= kGtMaxRows; }

size_t gjtc_bytes(int n_up, int n_dn, int nw)
{
    size_t b = 0;
    if (n_up > 0) b += gt_layout(n_up).per * (size_t)nw;
    if (n_dn > 0) b += gt_layout(n_dn).per * (size_t)nw;
    return b + 256;
}

// The update kernel's tensor maps: job q's work matrices as a 3-D tensor of 8-byte float
// pairs [count][n][n] (row stride gt_ld(n), matrix stride the scratch per matrix), boxes of
// 16 columns x 128 rows with 128-byte swizzle.
static cudaError_t gt_tensor_maps(GtJobs &js)
{
    for (int q = 0; q < 2; ++q) {
        memset(&js.tmw[q], 0, sizeof(CUtensorMap));
        if (q >= js.nj || js.j[q].count == 0) continue;
        const int n = js.j[q].n;
        const GtLayout L = gt_layout(n);
        const uint64_t dim[3] = {(uint64_t)n, (uint64_t)n, (uint64_t)js.j[q].count};
        const uint64_t stride[2] = {(uint64_t)gt_ld(n) * 8, (uint64_t)L.per};
        const uint32_t box[3] = {16, 128, 1};
        const cudaError_t e = tmap_encode(&js.tmw[q], CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 3, js.scr[q] + L.w, dim,
                                          stride, box, CU_TENSOR_MAP_SWIZZLE_128B);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_gj_tc(const GjJob *jobs, int n_jobs, void *scratch, cudaStream_t st, double kappa_max,
                         const WaitCfg &wc)
{
    GtJobs js;
    int nmax = 0, cmax = 0;
    unsigned char *p = static_cast<unsigned char *>(scratch);
    for (int q = 0; q < 2; ++q) {
        js.j[q] = jobs[q < n_jobs ? q : 0];
        if (q >= n_jobs) js.j[q].count = 0;
        js.scr[q] = p;
        if (q < n_jobs) p += gt_layout(js.j[q].n).per * (size_t)js.j[q].count;
        nmax = max(nmax, js.j[q].n);
        cmax = max(cmax, js.j[q].count);
    }
    js.nj = n_jobs;
    js.jb = 0;
    js.wait_ns = wc.limit_ns;
    js.expire_m = (wc.expire_kernels & QMC_EXPIRE_A4) ? wc.expire_w : -1;
    if (cmax == 0 || n_jobs == 0) return cudaSuccess;
    if (!gjtc_fits(nmax)) return cudaErrorInvalidConfiguration;
    // 56 KB of panel slices, 3 x 14 KB of pivot-row slices, 3 x 32 KB of old values, the
    // column exponents: one CTA per SM
    const size_t sm_up = 1024 + kGtSl * (size_t)(kGtAPlane + kGtBs * kGtBPlane) + kGtXs * (size_t)kGtXStage +
                         8 * (size_t)((nmax + kGtN - 1) / kGtN * kGtN);
    cudaError_t e;
    if ((e = gt_tensor_maps(js)) != cudaSuccess) return e;
    const int nthr = (nmax + 31) / 32 * 32;
    const size_t sm_panel = sizeof(float4) * (size_t)nthr * kGpLd;
    // one thread per row; the register budget follows the block
    // two CTAs per SM where there is more than one per SM to run (figures at the kernel)
    constexpr auto two = k_gt_panel<544, false, 2>, one = k_gt_panel<544, false, 1>, seq = k_gt_panel<kGtMaxRows, true, 1>;
    const bool share = cmax * n_jobs > 152;
    const auto panel = nmax >= kGtSeqMin ? seq : (share ? two : one);
    e = nmax >= kGtSeqMin ? allow_smem<seq>(sm_panel) : (share ? allow_smem<two>(sm_panel) : allow_smem<one>(sm_panel));
    if (e != cudaSuccess) return e;
    if ((e = allow_smem<k_gt_update>(sm_up)) != cudaSuccess) return e;
    const dim3 g1(cmax, n_jobs);
    if ((e = gt_clusters(k_gt_init, g1, n_jobs, st, js)) != cudaSuccess) return e;
    const int nt = (nmax + 127) / 128;
    const int nz = cmax * n_jobs;
    // CTAs per matrix of the update, each walking over its row tiles.  Many tiles: three row tiles
    // each; the CTAs of a matrix share its B planes in L2, which one CTA finds evicted on its
    // return (4096 matrices of 528 rows, 1 / 2 / 3 / 5 CTAs each: 59.5 / 57.3 / 59.5 / 63.9 ms, one
    // tile per CTA without the loop 62.2; 1024 of 866 rows, 1 / 2 / 3 / 7: 66.1 / 63.1 / 61.5 / 63.1,
    // 62.2).  Few tiles: one each, unless a schedule on 152 SMs is shorter by 15% with a CTA's
    // prologue counted as 0.35 of a row tile (74 of 528 rows, 1 / 2 / 3 / 5: 2.00 / 1.34 / 1.70 /
    // 1.46 ms; 128 of 528 rows, 1 / 5: 2.16 / 2.27; a gain of 9% by this count is none: 128 of 866
    // rows, 1 / 7: 8.64 / 8.06).
    int nt_up = (nt + 2) / 3;
    if ((long long)nz * nt < 16 * 152) {
        auto cost = [&](int d) { return ((nz * d + 151) / 152) * (20 * ((nt + d - 1) / d) + 7); };
        int best = cost(nt) * 85 / 100;
        nt_up = nt;
        for (int d = 1; d < nt; ++d)
            if (cost(d) < best) {
                best = cost(d);
                nt_up = d;
            }
    }
    for (int jb = 0; jb < nmax; jb += kGtB) {
        js.jb = jb;
        panel<<<g1, nthr, sm_panel, st>>>(js);
        for (int z0 = 0; z0 < nz; z0 += 65535) {
            const int zn = nz - z0 < 65535 ? nz - z0 : 65535;
            k_gt_update<<<dim3(nt_up, 1, zn), kGtUpThreads, sm_up, st>>>(js, z0);
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((e = gt_clusters(k_gt_final, g1, n_jobs, st, js, kappa_max)) != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace qmc
