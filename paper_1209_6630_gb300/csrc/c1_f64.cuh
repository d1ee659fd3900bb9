// C1 rows in FP64 (k_c1_f64 of the FP64 path, k_redo_c1 of the near-node recomputation), one CTA of
// 128 threads per (walker, electron): the active shells in chunks of 128, the exponentials spread
// flat over their primitives, the sums once per shell, the polynomials per AO.
#pragma once

#include "qmc_device.cuh"

namespace qmc {

constexpr int kCfThreads = 128;
constexpr int kCfShells = kCfThreads;                  // shells per chunk, one per thread

// Shared memory of a CTA: the active shells (for the whole electron), then one chunk's tables.
struct CfSmem {
    unsigned short *sh;            // [n_shell] active shells, ascending
    double *ex;                    // [kCfShells * kMaxPrim] exp(-gamma_p d2), by shell, in order
    double *d2;                    // [kCfShells]
    double *last;                  // [max AOs of a chunk] values (k_c1_f64), or [n_s] a row of D^-1 (k_vd_f64)
    int *ao;                       // [max AOs of a chunk] AO indices
    unsigned char *p_sh, *a_sh;    // chunk-local shell of each primitive / AO
};

__host__ __device__ inline int cf_max_ao(const SysDev &s) { return min(kCfShells * ncart(kMaxL), s.n_ao); }

__host__ __device__ inline size_t cf_smem(const SysDev &s)
{
    const size_t na = cf_max_ao(s);
    const size_t b = 8 * ((size_t)kCfShells * kMaxPrim + kCfShells) + 4 * na + 2 * (size_t)s.n_shell +
                     (size_t)kCfShells * kMaxPrim + na;
    return (b + 15) / 16 * 16;                           // (the doubles of `last` follow)
}

__device__ inline CfSmem cf_carve(const SysDev &s, unsigned char *base)
{
    const int na = cf_max_ao(s);
    CfSmem c;
    c.ex = reinterpret_cast<double *>(base);
    c.d2 = c.ex + kCfShells * kMaxPrim;
    c.ao = reinterpret_cast<int *>(c.d2 + kCfShells);
    c.sh = reinterpret_cast<unsigned short *>(c.ao + na);
    c.p_sh = reinterpret_cast<unsigned char *>(c.sh + s.n_shell);
    c.a_sh = c.p_sh + kCfShells * kMaxPrim;
    c.last = reinterpret_cast<double *>(base + cf_smem(s));
    return c;
}

// The active shells of an electron at r, ascending, into sh (the decisions of screen_electron).
static __device__ int cf_screen(const SysDev &s, double rx, double ry, double rz, unsigned short *sh_s, int *warp_s)
{
    const int t = threadIdx.x;
    const int per = (s.n_shell + kCfThreads - 1) / kCfThreads;   // <= 64, checked at load
    const int sh0 = min(t * per, s.n_shell), sh1 = min(sh0 + per, s.n_shell);
    unsigned long long mask = 0ull;
    int last_a = -1;
    bool atom_in = false;
    double d2 = 0.0;
    for (int sh = sh0; sh < sh1; ++sh) {
        const int a = s.sh_atom[sh];
        if (a != last_a) {
            last_a = a;
            d2 = sqdist_rn(rx, ry, rz, s.Q + 3 * a);
            atom_in = d2 < s.atom_R2[a];
        }
        if (atom_in && d2 < s.sh_R2[sh]) mask |= 1ull << (sh - sh0);
    }
    int total;
    int off = block_excl_scan<kCfThreads>(__popcll(mask), warp_s, &total);
    for (; mask; mask &= mask - 1) sh_s[off++] = (unsigned short)(sh0 + __ffsll((long long)mask) - 1);
    __syncthreads();
    return total;
}

// Tables of the chunk of shells from q0: returns its AO count; this thread's shell in `my` (-1:
// none), its first primitive of ex in `pofs`.  ex holds the primitives' exponentials on return.
static __device__ int cf_chunk(const SysDev &s, const CfSmem &c, int q0, int n_act, double rx, double ry, double rz,
                        int *warp_s, int &my, int &pofs)
{
    const int t = threadIdx.x;
    my = q0 + t < n_act ? c.sh[q0 + t] : -1;
    int nc = 0, np = 0, p0 = 0;
    if (my >= 0) {
        nc = ncart(s.sh_L[my]);
        np = s.sh_nprim[my];
        p0 = s.sh_pstart[my];
        const double *q = s.Q + 3 * s.sh_atom[my];
        c.d2[t] = sqdist_rn(rx, ry, rz, q);
    }
    int total;                                           // AOs in the low half, primitives in the high half
    const int off = block_excl_scan<kCfThreads>(nc | np << 16, warp_s, &total);
    pofs = off >> 16;
    for (int i = 0; i < nc; ++i) {
        c.ao[(off & 0xffff) + i] = s.sh_ao0[my] + i;
        c.a_sh[(off & 0xffff) + i] = (unsigned char)t;
    }
    for (int i = 0; i < np; ++i) {
        c.p_sh[pofs + i] = (unsigned char)t;
        reinterpret_cast<int *>(c.ex + pofs + i)[0] = p0 + i;    // the primitive, until its exponential replaces it
    }
    __syncthreads();
    const int ntp = total >> 16;
    for (int i = t; i < ntp; i += kCfThreads) {
        const int p = reinterpret_cast<const int *>(c.ex + i)[0];
        c.ex[i] = exp(-s.pg[p] * c.d2[c.p_sh[i]]);
    }
    __syncthreads();
    return total & 0xffff;
}


// C1[e][k] = sum_mu chi_mu(r) A[mu][k] into xrow, thread = MO k = t + 128 j.  The roundings are
// those that each caller has had (an ill-conditioned matrix would amplify a last bit): kRedo = false
// c (x y z) g with the terms of g rounded before they are added, true ((c x) y) z g with FMAs.
template <int NJ, bool kRedo>
__device__ __forceinline__ void c1_row_f64(const SysDev &s, const CfSmem &c, double *g_s, int *warp_s, int spin, double rx,
                                           double ry, double rz, double *__restrict__ xrow)
{
    const int t = threadIdx.x;
    const int ns = spin ? s.n_dn : s.n_up;
    const double *__restrict__ A = s.A64[spin];
    const int n_act = cf_screen(s, rx, ry, rz, c.sh, warp_s);
    double acc[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[j] = 0.0;
    const int kwarp = t & ~31;
    for (int q0 = 0; q0 < n_act; q0 += kCfShells) {
        int my, pofs;
        const int nao = cf_chunk(s, c, q0, n_act, rx, ry, rz, warp_s, my, pofs);
        if (my >= 0) {
            double g = 0.0;
            const int np = s.sh_nprim[my], p0 = s.sh_pstart[my];
            for (int p = 0; p < np; ++p)
                g = kRedo ? fma(s.pc[p0 + p], c.ex[pofs + p], g) : __dadd_rn(g, __dmul_rn(s.pc[p0 + p], c.ex[pofs + p]));
            g_s[t] = g;
        }
        __syncthreads();
        for (int m = t; m < nao; m += kCfThreads) {
            const int mu = c.ao[m], sl = c.a_sh[m];
            const double *q = s.Q + 3 * s.sh_atom[c.sh[q0 + sl]];
            const int pw = s.ao_pow[mu];
            const double x = ipow_small(rx - q[0], pw & 255), y = ipow_small(ry - q[1], (pw >> 8) & 255),
                         z = ipow_small(rz - q[2], (pw >> 16) & 255), sc = s.ao_scale[mu];
            c.last[m] = kRedo ? ((sc * x) * y) * z * g_s[sl] : sc * ((x * y) * z) * g_s[sl];
        }
        __syncthreads();
        // MO slots j whose whole warp lies beyond ns are skipped (warp-uniform)
#pragma unroll 4
        for (int m = 0; m < nao; ++m) {
            const double *__restrict__ arow = A + (size_t)c.ao[m] * ns;
            const double b = c.last[m];
            double a[NJ];
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const int k = t + kCfThreads * j;
                a[j] = (k < ns) ? __ldg(arow + k) : 0.0;
            }
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                if (kwarp + kCfThreads * j < ns) acc[j] = fma(a[j], b, acc[j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int k = t + kCfThreads * j;
        if (k < ns) xrow[k] = acc[j];
    }
}

__host__ __device__ inline size_t c1_smem(const SysDev &s) { return cf_smem(s) + 8 * (size_t)cf_max_ao(s); }

}  // namespace qmc
