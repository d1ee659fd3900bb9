// The FP64 path without the gradient and Laplacian matrices (steps a3 and a5):
// C1 alone before a4, then, from the inverse and the cofactor identities of
// Sec. II.C with the MO expansion Eq. (mo),
//   drift_{e,l} = sum_mu v_{e mu} d_l chi_mu(r_e),  lap_e = sum_mu v_{e mu} lap chi_mu(r_e),
//   v_{e mu}    = sum_k (D^-1)_{ek} a_{k mu}
// over the AOs that are not screened out for r_e: two products with the MO
// coefficients instead of five, all in FP64.  (qmc_slater_matrices, which
// returns C2..C5, keeps k_contract_f64.)
//
// Both kernels: one CTA per (walker, electron), 128 threads, shells in chunks
// of 128.  GB300's FP64 pipe runs at 1/64 of the FP32 rate (a warp instruction
// every 16 cycles of an SM, whatever number of its lanes is active), so what is
// counted is FP64 warp instructions: the exponentials are spread flat over the
// primitives of the active shells (a core shell has 8, the others 1 to 3),
// their sums taken once per shell, the polynomials per AO.
//   k_c1_f64     thread = MO; C1[e][k] = sum_mu chi_mu A[mu][k], every operation rounded as in
//                k_contract_f64 (bit-identical C1: an ill-conditioned matrix would amplify a last bit)
//   k_vd_f64     8 lanes = one row of A at a time, 32 rows per warp: each lane keeps 8 rows'
//                partial dot products with D^-1[e,:], a transposing butterfly (7 additions)
//                leaves each lane the v of one AO, which then meets that AO's derivatives
// Measured, 434 electrons x 96 walkers: C1..C5 26.9 ms -> C1 5.8 + drift 7.6 ms
// (158 electrons x 100: 4.6 -> 1.1 + 1.4 ms).  The tables of a chunk take up to 61 KB of shared memory at
// the loader's limits (8192 shells, 16 primitives, L = 4, 1024 electrons of a spin), so every system fits.
#include "c1_f64.cuh"

namespace qmc {

namespace {

template <int NJ>
__global__ void __launch_bounds__(kCfThreads) k_c1_f64(SysDev s, const double *__restrict__ R, double *__restrict__ X)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int warp_s[kCfThreads / 32];
    __shared__ double g_s[kCfShells];
    const int e = blockIdx.x, w = blockIdx.y;
    const int spin = e >= s.n_up;
    const int ei = spin ? e - s.n_up : e;
    const int ns = spin ? s.n_dn : s.n_up;
    const double *r = R + ((size_t)w * s.n_elec + e) * 3;
    const size_t msz = (size_t)s.n_up * s.n_up + (size_t)s.n_dn * s.n_dn;
    c1_row_f64<NJ, false>(s, cf_carve(s, smem_raw), g_s, warp_s, spin, r[0], r[1], r[2],
                          X + (size_t)w * msz + (spin ? (size_t)s.n_up * s.n_up : 0) + (size_t)ei * ns);
}

// Eight lanes' eight partial sums each: lane l of the group of 8 is left the total of sum l.
__device__ __forceinline__ double transpose_sum8(const double (&a)[8])
{
    const int l = threadIdx.x & 7;
    double b[4], d[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) {                        // keep the half that bit 2 of the lane names
        const double send = (l & 4) ? a[i] : a[i + 4];
        b[i] = ((l & 4) ? a[i + 4] : a[i]) + __shfl_xor_sync(0xffffffffu, send, 4);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const double send = (l & 2) ? b[i] : b[i + 2];
        d[i] = ((l & 2) ? b[i + 2] : b[i]) + __shfl_xor_sync(0xffffffffu, send, 2);
    }
    const double send = (l & 1) ? d[0] : d[1];
    return ((l & 1) ? d[1] : d[0]) + __shfl_xor_sync(0xffffffffu, send, 1);
}

__global__ void __launch_bounds__(kCfThreads) k_vd_f64(SysDev s, const double *__restrict__ R,
                                                       const double *__restrict__ Dinv, double *__restrict__ vd)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const CfSmem c = cf_carve(s, smem_raw);
    double *D_s = c.last;
    __shared__ int warp_s[kCfThreads / 32];
    __shared__ double g_s[3][kCfShells];
    __shared__ double red[kCfThreads / 32][4];

    const int e = blockIdx.x, w = blockIdx.y, t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const int spin = e >= s.n_up;
    const int ei = spin ? e - s.n_up : e;
    const int ns = spin ? s.n_dn : s.n_up;
    const double *__restrict__ A = s.A64[spin];
    const double *r = R + ((size_t)w * s.n_elec + e) * 3;
    const double rx = r[0], ry = r[1], rz = r[2];
    const size_t msz = (size_t)s.n_up * s.n_up + (size_t)s.n_dn * s.n_dn;
    const double *drow = Dinv + (size_t)w * msz + (spin ? (size_t)s.n_up * s.n_up : 0) + (size_t)ei * ns;
    for (int k = t; k < ns; k += kCfThreads) D_s[k] = drow[k];
    const int n_act = cf_screen(s, rx, ry, rz, c.sh, warp_s);   // (its barriers publish D_s)

    double b0 = 0.0, b1 = 0.0, b2 = 0.0, b3 = 0.0;
    if (t == 0) b0 = b1 = b2 = b3 = 0.0 * D_s[0];        // NaN where the inverse is NaN, also without an AO
    for (int q0 = 0; q0 < n_act; q0 += kCfShells) {
        int my, pofs;
        const int nao = cf_chunk(s, c, q0, n_act, rx, ry, rz, warp_s, my, pofs);
        if (my >= 0) {
            double g = 0.0, gd = 0.0, gl = 0.0;
            const int np = s.sh_nprim[my], p0 = s.sh_pstart[my];
            const double d2 = c.d2[t];
            for (int p = 0; p < np; ++p) {
                const double gam = s.pg[p0 + p], ce = s.pc[p0 + p] * c.ex[pofs + p];
                g += ce;
                gd += gam * ce;
                gl += (4.0 * gam * d2 - 6.0) * gam * ce;
            }
            g_s[0][t] = g;
            g_s[1][t] = gd;
            g_s[2][t] = gl;
        }
        __syncthreads();
        for (int m0 = wid * 32; m0 < nao; m0 += kCfThreads) {
            // lanes 8 j .. 8 j + 7 (group j) take rows m0 + 8 j + i, i = 0..7, eight MOs at a time
            const int j = lane >> 3, l = lane & 7;
            const double *row[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int m = m0 + 8 * j + i;
                row[i] = A + (size_t)c.ao[m < nao ? m : nao - 1] * ns;
            }
            double a[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) a[i] = 0.0;
            for (int k = l; k < ns; k += 8) {
                const double d = D_s[k];
#pragma unroll
                for (int i = 0; i < 8; ++i) a[i] = fma(__ldg(row[i] + k), d, a[i]);
            }
            __syncwarp();
            const double v = transpose_sum8(a);          // of row m0 + 8 j + l = m0 + lane
            const int m = m0 + lane;
            if (m < nao) {
                const int mu = c.ao[m], sl = c.a_sh[m];
                const double *q = s.Q + 3 * s.sh_atom[c.sh[q0 + sl]];
                const double dx = rx - q[0], dy = ry - q[1], dz = rz - q[2];
                const double g = g_s[0][sl], gd = g_s[1][sl], gl = g_s[2][sl];
                const int pw = s.ao_pow[mu];
                const int nx = pw & 255, ny = (pw >> 8) & 255, nz = (pw >> 16) & 255;
                const int L = nx + ny + nz;
                const double px = ipow_small(dx, nx), py = ipow_small(dy, ny), pz = ipow_small(dz, nz);
                const double P = px * py * pz;
                const double dpx = nx ? nx * ipow_small(dx, nx - 1) : 0.0;
                const double dpy = ny ? ny * ipow_small(dy, ny - 1) : 0.0;
                const double dpz = nz ? nz * ipow_small(dz, nz - 1) : 0.0;
                const double ddx = nx > 1 ? nx * (nx - 1) * ipow_small(dx, nx - 2) : 0.0;
                const double ddy = ny > 1 ? ny * (ny - 1) * ipow_small(dy, ny - 2) : 0.0;
                const double ddz = nz > 1 ? nz * (nz - 1) * ipow_small(dz, nz - 2) : 0.0;
                const double cv = s.ao_scale[mu] * v, m2gd = -2.0 * gd;
                b0 = fma(cv, dpx * py * pz * g + m2gd * dx * P, b0);
                b1 = fma(cv, px * dpy * pz * g + m2gd * dy * P, b1);
                b2 = fma(cv, px * py * dpz * g + m2gd * dz * P, b2);
                const double lapP = ddx * py * pz + px * ddy * pz + px * py * ddz;
                b3 = fma(cv, lapP * g + P * (gl - 4.0 * L * gd), b3);
            }
        }
        __syncthreads();
    }
    double b[4] = {b0, b1, b2, b3};
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) b[q] += __shfl_xor_sync(0xffffffffu, b[q], o);
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < 4; ++q) red[wid][q] = b[q];
    __syncthreads();
    if (t < 4) vd[((size_t)w * s.n_elec + e) * 4 + t] = ((red[0][t] + red[1][t]) + red[2][t]) + red[3][t];
}

size_t vd_smem(const SysDev &s) { return cf_smem(s) + 8 * (size_t)(s.n_up > s.n_dn ? s.n_up : s.n_dn); }

template <int NJ>
cudaError_t launch_c1_nj(const SysDev &s, int nw, const double *R, double *X, cudaStream_t st)
{
    const size_t sm = c1_smem(s);
    cudaError_t e = allow_smem<k_c1_f64<NJ>>(sm);
    if (e != cudaSuccess) return e;
    k_c1_f64<NJ><<<dim3(s.n_elec, nw), kCfThreads, sm, st>>>(s, R, X);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_c1_f64(const SysDev &s, int nw, const double *R, double *X, cudaStream_t st)
{
    if (nw == 0 || s.n_elec == 0) return cudaSuccess;
    const int nmax = s.n_up > s.n_dn ? s.n_up : s.n_dn;
    switch ((nmax + kCfThreads - 1) / kCfThreads) {
    case 1: return launch_c1_nj<1>(s, nw, R, X, st);
    case 2: return launch_c1_nj<2>(s, nw, R, X, st);
    case 3: return launch_c1_nj<3>(s, nw, R, X, st);
    case 4: return launch_c1_nj<4>(s, nw, R, X, st);
    case 5: return launch_c1_nj<5>(s, nw, R, X, st);
    case 6: return launch_c1_nj<6>(s, nw, R, X, st);
    case 7: return launch_c1_nj<7>(s, nw, R, X, st);
    case 8: return launch_c1_nj<8>(s, nw, R, X, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_vdrift_f64(const SysDev &s, int nw, const double *R, const double *Dinv, double *vd,
                              cudaStream_t st)
{
    if (nw == 0 || s.n_elec == 0) return cudaSuccess;
    const size_t sm = vd_smem(s);
    cudaError_t e = allow_smem<k_vd_f64>(sm);
    if (e != cudaSuccess) return e;
    k_vd_f64<<<dim3(s.n_elec, nw), kCfThreads, sm, st>>>(s, R, Dinv, vd);
    return cudaGetLastError();
}

}  // namespace qmc
