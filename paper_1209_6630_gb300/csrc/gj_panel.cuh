// Panel elimination of the FP64 Gauss-Jordan kernels (k_gj, k_redo_panel),
// one CTA, the panel [n][NB] in shared memory.
//
// What bounds it is the FP64 pipe, which takes a warp instruction every 16
// cycles whatever lanes are active, and the latency of a column step: so the
// pivot search compares the magnitudes' bits as integers (REDUX instead of FP64
// compares and shuffles), one warp alone divides and scales the pivot row, the
// logarithms of the pivots are left to the end of the panel (one per lane),
// and a step has two barriers.  Pairs of columns are swizzled by row, so that
// the threads' accesses (one row each) meet two-way bank conflicts at most (the
// unswizzled layout had 16-way ones).
#pragma once

#include <cuda_runtime.h>

namespace qmc {

// element (row i, column c) of the swizzled panel
template <int NB>
__device__ __forceinline__ int gj_at(int i, int c)
{
    const int s = (NB < 16 ? i / (16 / NB) : i) & (NB / 2 - 1);
    return i * NB + ((((c >> 1) ^ s) << 1) | (c & 1));
}

// |x| as an integer that orders like it; 0 for NaN (never a pivot) and 0
__device__ __forceinline__ unsigned long long gj_key(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
    return b > 0x7ff0000000000000ull ? 0ull : b;
}

// The largest key of a warp and the smallest index that has it, in every lane.
__device__ __forceinline__ void gj_warp_max(unsigned long long &k, int &i)
{
    const unsigned hi = (unsigned)(k >> 32), lo = (unsigned)k;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    i = (int)__reduce_min_sync(0xffffffffu, (hi == mh && lo == ml) ? (unsigned)i : 0x7fffffffu);
    k = (unsigned long long)mh << 32 | ml;
}

template <int NB>
struct GjPanelShared {
    double prow[NB];                 // the step's pivot row, scaled; 1 / pivot in its own column
    double piv[NB];                  // pivots of the panel
    unsigned long long key[32];      // per warp: pivot candidate
    int idx[32];
    short pp[NB];                    // pivot rows of the panel
};

// Eliminates the first w columns of P with partial pivoting among the rows with used[i] == 0
// (the first row with the largest |entry|); marks the pivots in `used`, leaves their rows in S.pp
// and their values in S.piv.  False on an exact zero (or NaN) pivot.  Ends with a barrier.
template <int NB>
__device__ bool gj_panel(double *P, int n, int w, short *used, GjPanelShared<NB> &S)
{
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5, nthr = blockDim.x, nwarps = nthr >> 5;
    unsigned long long bk = 0;
    int bi = n;
    for (int i = t; i < n; i += nthr)
        if (!used[i]) {
            const unsigned long long k = gj_key(P[gj_at<NB>(i, 0)]);
            if (k > bk) { bk = k; bi = i; }
        }
    gj_warp_max(bk, bi);
    if (lane == 0) { S.key[wid] = bk; S.idx[wid] = bi; }
    __syncthreads();
    for (int c = 0; c < w; ++c) {
        unsigned long long k = lane < nwarps ? S.key[lane] : 0ull;
        int p = lane < nwarps ? S.idx[lane] : n;
        gj_warp_max(k, p);
        if (k == 0ull) return false;                       // every warp sees the same candidates
        if (wid == 0) {
            const double piv = P[gj_at<NB>(p, c)];
            const double inv = 1.0 / piv;
            if (lane < NB) {
                const double x = lane == c ? inv : P[gj_at<NB>(p, lane)] * inv;
                S.prow[lane] = x;
            }
            if (lane == 0) {
                used[p] = 1;
                S.pp[c] = (short)p;
                S.piv[c] = piv;
            }
        }
        __syncthreads();
        // the other rows, and the candidates of column c + 1 among those not used yet
        bk = 0;
        bi = n;
        const double inv = S.prow[c];
        for (int i = t; i < n; i += nthr) {
            if (i == p) {
#pragma unroll
                for (int q = 0; q < NB; ++q) P[gj_at<NB>(i, q)] = S.prow[q];
                continue;
            }
            const double f = P[gj_at<NB>(i, c)];
#pragma unroll
            for (int q = 0; q < NB; ++q)
                if (q != c) P[gj_at<NB>(i, q)] = fma(-f, S.prow[q], P[gj_at<NB>(i, q)]);
            P[gj_at<NB>(i, c)] = -f * inv;
            if (c + 1 < w && !used[i]) {
                const unsigned long long kk = gj_key(P[gj_at<NB>(i, c + 1)]);
                if (kk > bk) { bk = kk; bi = i; }
            }
        }
        gj_warp_max(bk, bi);
        if (lane == 0) { S.key[wid] = bk; S.idx[wid] = bi; }
        __syncthreads();
    }
    return true;
}

// log|det| and sign of the panel's pivots added by warp 0 (its lane 0 holds the sums): one
// logarithm per lane, added in the pivots' order.
template <int NB>
__device__ __forceinline__ void gj_add_pivots(const GjPanelShared<NB> &S, int w, double &logabs, int &neg)
{
    const int lane = threadIdx.x & 31;
    const double piv = lane < w ? S.piv[lane] : 1.0;
    const double lg = log(fabs(piv));
    neg ^= __popc(__ballot_sync(0xffffffffu, piv < 0.0)) & 1;
    for (int c = 0; c < w; ++c) logabs += __shfl_sync(0xffffffffu, lg, c);
}

}  // namespace qmc
