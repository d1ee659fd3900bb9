// Step a7: adjoint of log|Psi| with respect to the MO coefficients, FP64.
//
//   dA_s[mu][k] = sum_w g_w sum_{e in s} chi_mu(r_{w,e}) (D^-1)_{w,ek}
//
// (d log|det D| / d D_{ke} = (D^-1)_{ek} and D_{ke} = sum_mu a_{k mu} chi_mu(r_e),
// the cofactor identity behind the drift formula of Sec. II.C.)  chi is
// recomputed from R with the forward pass's exact screening decisions; the
// AO values are never stored.
//
// One cluster of C CTAs per (atom a, block of 128 MOs, spin).  It owns the rows of dA belonging to
// the atom's AOs, so no atomics are needed.  Each CTA scans its C-th of the (walker, electron)
// pairs, keeps those inside the atomic radius (same correctly rounded d2 as the forward
// screening), evaluates the atom's active shells for a batch of hits in shared memory (a warp's
// lanes at the same shell, the radial sum once per shell) and accumulates
// acc[mu] += g_w chi_mu (D^-1)_{ek} in registers (thread = MO k, four hits' loads in flight);
// at the end the cluster's partial sums are added in rank order through distributed shared
// memory.  Bound by the FP64 pipe (1/64 of the FP32 rate): the products are issued only for the
// AOs that the atom has, in groups of 5.  One CTA per atom without the split left 104 CTAs on
// 152 SMs at 158 electrons; there, with 100 walkers: 11.7 -> 1.7 ms.
#include <cooperative_groups.h>

#include "qmc_device.cuh"

namespace qmc {

namespace cg = cooperative_groups;

constexpr int kBwThreads = 128;
constexpr int kBwBatch = 128;   // hits buffered before an accumulation pass
constexpr int kBwGroup = 5;     // AOs per group of products

template <int MAXAO>
__global__ void __launch_bounds__(kBwThreads) k_backward_f64(SysDev s, int nw, const double *__restrict__ R,
                                                             const double *__restrict__ dinv,
                                                             const double *__restrict__ gw,
                                                             double *__restrict__ dA_up,
                                                             double *__restrict__ dA_dn)
{
    __shared__ int hit_w[kBwBatch + kBwThreads], hit_e[kBwBatch + kBwThreads];
    extern __shared__ __align__(16) double chi_s[];   // [kBwBatch + kBwThreads][MAXAO]; then the partial sums
    __shared__ int warp_s[kBwThreads / 32];

    cg::cluster_group cluster = cg::this_cluster();
    const int nrank = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int a = blockIdx.x / nrank, spin = blockIdx.z;      // the same for a whole cluster, so are the returns below
    const int ns = spin ? s.n_dn : s.n_up;
    const int e0 = spin ? s.n_up : 0;
    const int t = threadIdx.x;
    const int k = blockIdx.y * kBwThreads + t;
    if (blockIdx.y * kBwThreads >= ns) return;
    const int sh0 = s.atom_sh0[a], sh1 = s.atom_sh0[a + 1];
    if (sh1 == sh0) return;   // an atom without basis functions owns no rows of dA
    const int ao0 = s.sh_ao0[sh0];
    const int nao = s.sh_ao0[sh1 - 1] + ncart(s.sh_L[sh1 - 1]) - ao0;
    const double ra2 = s.atom_R2[a];
    const double *q = s.Q + 3 * a;
    const double qx = q[0], qy = q[1], qz = q[2];
    const size_t msz = (size_t)s.n_up * s.n_up + (size_t)s.n_dn * s.n_dn;
    const size_t soff = spin ? (size_t)s.n_up * s.n_up : 0;

    double acc[MAXAO];
#pragma unroll
    for (int m = 0; m < MAXAO; ++m) acc[m] = 0.0;

    const long long npair = (long long)nw * ns;
    const long long q_lo = npair * rank / nrank, q_hi = npair * (rank + 1) / nrank;
    int nbuf = 0;             // hits buffered (the same value in every thread)
    for (long long q0 = q_lo; q0 < q_hi; q0 += kBwThreads) {
        const long long qq = q0 + t;
        int w = 0, ei = 0, hit = 0;
        if (qq < q_hi) {
            w = (int)(qq / ns);
            ei = (int)(qq - (long long)w * ns);
            if (gw[w] != 0.0) {
                const double *r = R + ((size_t)w * s.n_elec + e0 + ei) * 3;
                hit = sqdist_rn(r[0], r[1], r[2], q) < ra2;
            }
        }
        int total;
        const int off = block_excl_scan<kBwThreads>(hit, warp_s, &total);
        if (hit) { hit_w[nbuf + off] = w; hit_e[nbuf + off] = ei; }
        nbuf += total;
        __syncthreads();
        if (nbuf < kBwBatch && q0 + kBwThreads < q_hi) continue;
        const int nh = nbuf;
        // AO values (times g_w) of the atom's active shells for every hit
        for (int p = t; p < nh * (sh1 - sh0); p += kBwThreads) {
            const int sh = sh0 + p / nh, h = p - (sh - sh0) * nh;
            const double *r = R + ((size_t)hit_w[h] * s.n_elec + e0 + hit_e[h]) * 3;
            const double d2s = sqdist_rn(r[0], r[1], r[2], q);
            const int m0 = s.sh_ao0[sh] - ao0, nc = ncart(s.sh_L[sh]);
            double *c = chi_s + h * MAXAO + m0;
            if (!(d2s < s.sh_R2[sh])) {
                for (int m = 0; m < nc; ++m) c[m] = 0.0;
                continue;
            }
            const double dx = r[0] - qx, dy = r[1] - qy, dz = r[2] - qz;
            const double d2 = dx * dx + dy * dy + dz * dz;
            double g = 0.0;
            const int p0 = s.sh_pstart[sh], np = s.sh_nprim[sh];
            for (int i = 0; i < np; ++i) g += s.pc[p0 + i] * exp(-s.pg[p0 + i] * d2);
            const double gv = gw[hit_w[h]];
            for (int m = 0; m < nc; ++m) {
                const int mu = ao0 + m0 + m, pw = s.ao_pow[mu];
                c[m] = gv * (s.ao_scale[mu] * ipow_small(dx, pw & 255) * ipow_small(dy, (pw >> 8) & 255) *
                             ipow_small(dz, (pw >> 16) & 255) * g);
            }
        }
        __syncthreads();
        if (k < ns) {
            const double *dcol = dinv + soff + k;
            for (int h0 = 0; h0 < nh; h0 += 4) {
                double dv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int h = min(h0 + u, nh - 1);
                    dv[u] = dcol[(size_t)hit_w[h] * msz + (size_t)hit_e[h] * ns];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (h0 + u >= nh) break;
                    const double *c = chi_s + (h0 + u) * MAXAO;
#pragma unroll
                    for (int g = 0; g < MAXAO; g += kBwGroup) {
                        if (g >= nao) break;
#pragma unroll
                        for (int m = g; m < min(g + kBwGroup, MAXAO); ++m)
                            acc[m] = fma(m < nao ? c[m] : 0.0, dv[u], acc[m]);
                    }
                }
            }
        }
        __syncthreads();
        nbuf = 0;
    }
    double *dA = spin ? dA_dn : dA_up;
    if (nrank == 1) {
        if (k < ns)
#pragma unroll
            for (int m = 0; m < MAXAO; ++m)
                if (m < nao) dA[(size_t)(ao0 + m) * ns + k] = acc[m];
        return;
    }
    // partial sums [MAXAO][128]; rank r adds rows r, r + C, ... over the ranks in order
#pragma unroll
    for (int m = 0; m < MAXAO; ++m) chi_s[m * kBwThreads + t] = acc[m];
    cluster.sync();
    if (k < ns)
        for (int m = rank; m < nao; m += nrank) {
            double x = 0.0;
            for (int r = 0; r < nrank; ++r) x += cluster.map_shared_rank(chi_s, r)[m * kBwThreads + t];
            dA[(size_t)(ao0 + m) * ns + k] = x;
        }
    cluster.sync();           // no CTA leaves while its sums are read
}

template <int MAXAO>
static cudaError_t launch_bw(const SysDev &s, int nw, const double *R, const double *dinv, const double *g,
                             double *dA_up, double *dA_dn, cudaStream_t st)
{
    const int nmax = s.n_up > s.n_dn ? s.n_up : s.n_dn;
    const int nmin = s.n_up < s.n_dn ? s.n_up : s.n_dn;
    const unsigned nblk = (nmax + kBwThreads - 1) / kBwThreads;
    // CTAs per cluster: up to 8 (the portable size), while the grid has fewer than 16 CTAs for
    // each of 152 SMs and a CTA keeps at least two scans of 128 pairs
    unsigned c = 1;
    while (c < 8 && (size_t)s.n_atom * nblk * 2 * c < 152 * 16 &&
           (long long)nw * (nmin > 0 ? nmin : nmax) >= (long long)4 * kBwThreads * c)
        c *= 2;
    const size_t sm = sizeof(double) * (size_t)(kBwBatch + kBwThreads) * MAXAO;
    cudaError_t e = cudaFuncSetAttribute(k_backward_f64<MAXAO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sm);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = c;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(s.n_atom * c, nblk, 2);
    cfg.blockDim = dim3(kBwThreads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_backward_f64<MAXAO>, s, nw, R, dinv, g, dA_up, dA_dn);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_backward_f64(const SysDev &s, int nw, const double *R, const double *dinv,
                                const double *g, double *dA_up, double *dA_dn, cudaStream_t st,
                                int max_ao_per_atom)
{
    if (max_ao_per_atom <= 16) return launch_bw<16>(s, nw, R, dinv, g, dA_up, dA_dn, st);
    if (max_ao_per_atom <= 32) return launch_bw<32>(s, nw, R, dinv, g, dA_up, dA_dn, st);
    return cudaErrorInvalidValue;
}

}  // namespace qmc
