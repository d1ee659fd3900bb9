// Steps a5-a6: drift, kinetic energy and local energy per walker, FP64.
// With a Jastrow factor (Psi = e^J Det_up Det_dn, Sec. II.C) the drift gains
// grad_e J and the kinetic term lap_e J + |grad_e J|^2 + 2 grad_e J . b_e (b_e
// the determinants' drift), J is added to log|Psi| (FP64 pair sums, each pair
// evaluated once for both of its electrons).
//
//   drift_{e,l} = sum_k (D^-1)_{ek} d_l phi_k(r_e)     (Eq. 2 with the
//   lap_e       = sum_k (D^-1)_{ek} lap phi_k(r_e)      Sec. II.C vector products;
//   T           = -1/2 sum_e lap_e                       Psi is linear in column e)
//   V_en = -sum_{e,a} Z_a / |r_e - Q_a|,  V_ee = sum_{i<j} 1 / |r_i - r_j|,
//   V_nn = sum_{a<b} Z_a Z_b / |Q_a - Q_b| (load time),  E_L = T + V (Eq. 4)
//
// A cluster of 1, 2, 4 or 8 CTAs per walker (one where the walkers fill the card); one warp per
// electron row for the dot products (rows of D^-1 and of C2..C5 are contiguous);
// warp-shuffle reductions, the CTAs' sums added in rank order through distributed shared memory.
// Measured: 1056 electrons x 37 walkers 854 -> 272 us (37 CTAs before), 158 electrons x 1 walker
// 52 -> 17 us; with the Jastrow factor, 434 electrons x 601 walkers 13.6 -> 7.2 ms.
//
// FP64 path: everything in FP64.  Mixed path (C2..C4 in FP32): the drift
// dots in FP32 (D^-1 truncated to float by integer operations), the
// Laplacian dot in FP64, and the Coulomb sums in float-float on the FP32
// pipes: differences of float-pair positions, r^2 as a float pair, 1/r from
// the FP32 reciprocal square root refined by one Newton step (relative error
// ~2^-43), sums kept as float pairs.
#include <cooperative_groups.h>
#include <math.h>

#include <type_traits>

#include "ff_math.cuh"
#include "qmc_internal.cuh"
#include "recip_f64.cuh"

namespace qmc {

namespace cg = cooperative_groups;

constexpr int kEnThreads = 256;
constexpr int kEnWarps = kEnThreads / 32;

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// x rounded toward zero to a float by integer operations (|x| in the normal
// float range or 0; used where a 2^-23 relative error is acceptable)
__device__ __forceinline__ float f32_trunc(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7ff) - 1023 + 127;
    if (ex <= 0) return 0.f;
    const unsigned int f = (unsigned int)(b >> 32 & 0x80000000u) | ((unsigned int)min(ex, 254) << 23) |
                           (unsigned int)((b >> 29) & 0x7fffffu);
    return __uint_as_float(f);
}

// 1/r for the float-pair difference (dx, dy, dz)
__device__ __forceinline__ float2 ff_inv_r(float2 dx, float2 dy, float2 dz)
{
    const float2 r2 = ff::add(ff::add(ff::mul(dx, dx), ff::mul(dy, dy)), ff::mul(dz, dz));
    const float y0 = rsqrtf(r2.x);
    const float y0s = __fmul_rn(y0, y0);
    const float2 t = make_float2(y0s, fmaf(y0, y0, -y0s));      // y0^2 exactly
    const float2 e = ff::sub(make_float2(1.f, 0.f), ff::mul(r2, t));   // 1 - r2 y0^2, small
    return ff::renorm(y0, 0.5f * y0 * e.x);                      // Newton step y0 (1 + e/2)
}

// Coulomb sums of one walker in float-float (mixed path); rs: 3N positions,
// qs: 3 n_atom nuclear positions, zs: charges, all staged in shared memory.
// Warp `wid` of `nwarps` (over the walker's CTAs).
__device__ __forceinline__ void coulomb_ff(const SysDev &s, const float2 *rs, const float2 *qs, const float *zs,
                                           int wid, int nwarps, double &ven, double &vee)
{
    const int lane = threadIdx.x & 31;
    const int N = s.n_elec;
    float2 en = make_float2(0.f, 0.f), ee = make_float2(0.f, 0.f);
    for (int e = wid; e < N; e += nwarps) {
        const float2 rx = rs[3 * e], ry = rs[3 * e + 1], rz = rs[3 * e + 2];
        for (int a = lane; a < s.n_atom; a += 32) {
            const float2 y = ff_inv_r(ff::sub(rx, qs[3 * a]), ff::sub(ry, qs[3 * a + 1]), ff::sub(rz, qs[3 * a + 2]));
            en = ff::add(en, ff::mulf(y, zs[a]));
        }
        for (int j = e + 1 + lane; j < N; j += 32)
            ee = ff::add(ee, ff_inv_r(ff::sub(rx, rs[3 * j]), ff::sub(ry, rs[3 * j + 1]), ff::sub(rz, rs[3 * j + 2])));
    }
    ven = -ff::val(en);
    vee = ff::val(ee);
}

// Drift and Laplacian of the determinants for electron e from C2..C5 (mixed path; one warp, results
// on every lane): b_l = sum_k (D^-1)_{ek} C_{1+l}[e][k], lap = sum_k (D^-1)_{ek} C5[e][k].
__device__ __forceinline__ void dets_drift_lap(const SysDev &s, const double *__restrict__ Dinv,
                                               const float *__restrict__ Cg, const CView &cv, int w, int e, int lane,
                                               size_t msz, double &b0, double &b1, double &b2, double &b3)
{
    const int spin = e >= s.n_up;
    const int ei = spin ? e - s.n_up : e;
    const int ns = spin ? s.n_dn : s.n_up;
    const size_t nu2 = (size_t)s.n_up * s.n_up;
    const size_t soff = spin ? nu2 : 0;
    const size_t nss = (size_t)ns * ns;
    const double *drow = Dinv + (size_t)w * msz + soff + (size_t)ei * ns;
    const float *grow = Cg + (size_t)w * cv.g_wstride + (spin ? cv.g_ncomp * nu2 : 0) + (size_t)ei * ns;
    const double *lrow = cv.l + (size_t)w * cv.l_wstride + (spin ? cv.l_ncomp * nu2 : 0) +
                         (size_t)cv.l_comp * nss + (size_t)ei * ns;
    float f0 = 0.f, f1 = 0.f, f2 = 0.f;
    b3 = 0.0;
    for (int k = lane; k < ns; k += 32) {
        const double d = drow[k];
        const float df = f32_trunc(d);
        f0 = fmaf(df, grow[k], f0);
        f1 = fmaf(df, grow[nss + k], f1);
        f2 = fmaf(df, grow[2 * nss + k], f2);
        b3 = fma(d, lrow[k], b3);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        f0 += __shfl_xor_sync(0xffffffffu, f0, off);
        f1 += __shfl_xor_sync(0xffffffffu, f1, off);
        f2 += __shfl_xor_sync(0xffffffffu, f2, off);
    }
    b0 = f0; b1 = f1; b2 = f2;
    b3 = warp_sum(b3);
}

// The Jastrow factor of one walker over the CTAs of its cluster: grad_e J (acc[0..2][e]) and
// lap_e J (acc[3][e]) are the sums of the ranks' arrays, J itself the sum of the returned values
// over all threads.  Each pair is evaluated once: in step d electron e meets e + d (mod N);
// within a step the partners are distinct, so their sums need only a barrier between steps, and
// every sum has a fixed order.  rank takes the steps and the atoms congruent to it.
// rj: 3N positions; acc: [4][N] in shared memory.
__device__ double jastrow_all(const SysDev &s, const double *rj, double *acc, int rank, int nrank)
{
    const int t = threadIdx.x, N = s.n_elec;
    double Jt = 0.0;
    for (int q = t; q < 4 * N; q += kEnThreads) acc[q] = 0.0;
    __syncthreads();
    for (int e0 = 0; e0 < N; e0 += kEnThreads) {
        const int e = e0 + t;
        const bool ok = e < N;
        const double rx = ok ? rj[3 * e] : 0.0, ry = ok ? rj[3 * e + 1] : 0.0, rz = ok ? rj[3 * e + 2] : 0.0;
        double g0 = 0.0, g1 = 0.0, g2 = 0.0, L = 0.0;
        for (int d = 1 + rank; d <= N / 2; d += nrank) {
            // (an even N meets its opposite electron from both sides at d = N / 2: the lower one counts)
            if (ok && !(2 * d == N && e >= d)) {
                const int j = e + d < N ? e + d : e + d - N;
                const double dx = rx - rj[3 * j], dy = ry - rj[3 * j + 1], dz = rz - rj[3 * j + 2];
                const double a = ((e < s.n_up) == (j < s.n_up)) ? s.ja_par : s.ja_anti;
                double f, lp, u;
                jastrow_term(dx * dx + dy * dy + dz * dz, a, s.jb_ee, f, lp, u);
                g0 = fma(f, dx, g0); g1 = fma(f, dy, g1); g2 = fma(f, dz, g2);
                L += lp;
                Jt += u;
                acc[j] = fma(-f, dx, acc[j]);
                acc[N + j] = fma(-f, dy, acc[N + j]);
                acc[2 * N + j] = fma(-f, dz, acc[2 * N + j]);
                acc[3 * N + j] += lp;
            }
            __syncthreads();
        }
        if (ok) {
            for (int at = rank; at < s.n_atom; at += nrank) {
                const double dx = rx - s.Q[3 * at], dy = ry - s.Q[3 * at + 1], dz = rz - s.Q[3 * at + 2];
                double f, lp, u;
                jastrow_term(dx * dx + dy * dy + dz * dz, -s.ja_en[at], s.jb_en[at], f, lp, u);
                g0 = fma(f, dx, g0); g1 = fma(f, dy, g1); g2 = fma(f, dz, g2);
                L += lp;
                Jt += u;
            }
            acc[e] += g0; acc[N + e] += g1; acc[2 * N + e] += g2; acc[3 * N + e] += L;
        }
        __syncthreads();                                       // before the next block's partners
    }
    return Jt;
}

template <typename TG>
__global__ void __launch_bounds__(kEnThreads) k_drift_energy(SysDev s, const double *__restrict__ R,
                                                             const double *__restrict__ Dinv,
                                                             const TG *__restrict__ Cg, CView cv,
                                                             const double *__restrict__ logabs2,
                                                             const double *__restrict__ sign2,
                                                             const uint32_t *__restrict__ sing,
                                                             qmc_eval_out o, int w_off, const float2 *__restrict__ Q2,
                                                             int stage)
{
    constexpr bool kMixed = std::is_same<TG, float>::value;
    // mixed: positions, nuclei, charges as floats; with a Jastrow factor (before them) positions
    // and the pair sums in FP64
    extern __shared__ __align__(16) unsigned char en_smem[];
    __shared__ double red[4][kEnWarps];
    __shared__ double total[4];
    __shared__ int s_nonfinite;
    cg::cluster_group cluster = cg::this_cluster();
    const int nrank = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int w = blockIdx.x / nrank;
    const int wg = w + w_off;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const int gw = rank * kEnWarps + wid, ngw = nrank * kEnWarps;   // warps of the walker
    const int N = s.n_elec;
    const size_t msz = (size_t)s.n_up * s.n_up + (size_t)s.n_dn * s.n_dn;
    const double *Rw = R + (size_t)w * N * 3;

    if (t == 0) s_nonfinite = 0;
    __syncthreads();
    double *acc = reinterpret_cast<double *>(en_smem);         // [4][N] (Jastrow only)
    float2 *rs = reinterpret_cast<float2 *>(acc + (s.jas ? 4 * N : 0));
    float *zs = reinterpret_cast<float *>(rs + 3 * N);         // (padded to an even count)
    float2 *qs = reinterpret_cast<float2 *>(zs + ((s.n_atom + 1) & ~1));
    double *rj = kMixed ? reinterpret_cast<double *>(qs + ((stage & 1) ? 3 * s.n_atom : 0)) : acc + 4 * N;   // [3 N]
    int bad = 0;
    for (int q = t; q < 3 * N; q += kEnThreads) {
        const double x = Rw[q];
        bad |= !isfinite(x);
        if (stage & 2) rj[q] = x;
        if constexpr (kMixed) rs[q] = ff::from_double(x);
    }
    if constexpr (kMixed) {
        if (stage & 1)
            for (int q = t; q < 3 * s.n_atom; q += kEnThreads) qs[q] = Q2[q];
        for (int a = t; a < s.n_atom; a += kEnThreads) zs[a] = (float)s.Z[a];
    }
    if (bad) s_nonfinite = 1;
    __syncthreads();

    double lap_acc = 0.0, jas_acc = 0.0;
    if (s.jas) {
        jas_acc = jastrow_all(s, (stage & 2) ? rj : Rw, acc, rank, nrank);
        cluster.sync();                                        // every rank's sums are complete
    }
    for (int e = gw; e < N; e += ngw) {
        double b0 = 0.0, b1 = 0.0, b2 = 0.0, b3 = 0.0;
        if (!kMixed || cv.vd) {  // FP64 path, C-free variant: drift and Laplacian of the determinants already formed
            const double *v = cv.vd + ((size_t)w * N + e) * 4;
            b0 = v[0]; b1 = v[1]; b2 = v[2]; b3 = v[3];
        } else if constexpr (kMixed) {
            dets_drift_lap(s, Dinv, Cg, cv, w, e, lane, msz, b0, b1, b2, b3);
        }
        if (lane == 0) {
            double g0 = 0.0, g1 = 0.0, g2 = 0.0, L = 0.0;
            if (s.jas)
                for (int r = 0; r < nrank; ++r) {
                    const double *x = cluster.map_shared_rank(acc, r);
                    g0 += x[e]; g1 += x[N + e]; g2 += x[2 * N + e]; L += x[3 * N + e];
                }
            double *dr = o.drift + ((size_t)wg * N + e) * 3;
            dr[0] = b0 + g0; dr[1] = b1 + g1; dr[2] = b2 + g2;
            // lap_e Psi / Psi with Psi = e^J Det: lap J + |grad J|^2 + 2 grad J . grad Det / Det + lap Det / Det
            lap_acc += b3 + L + (g0 * g0 + g1 * g1 + g2 * g2) + 2.0 * (g0 * b0 + g1 * b1 + g2 * b2);
        }
    }
    double ven = 0.0, vee = 0.0;
    if constexpr (kMixed) {
        coulomb_ff(s, rs, (stage & 1) ? qs : Q2, zs, gw, ngw, ven, vee);
    } else {
        for (int e = gw; e < N; e += ngw) {
            const double rx = Rw[3 * e], ry = Rw[3 * e + 1], rz = Rw[3 * e + 2];
            for (int a = lane; a < s.n_atom; a += 32) {
                const double dx = rx - s.Q[3 * a], dy = ry - s.Q[3 * a + 1], dz = rz - s.Q[3 * a + 2];
                ven -= s.Z[a] * rsqrt_f64(dx * dx + dy * dy + dz * dz);
            }
            for (int j = e + 1 + lane; j < N; j += 32) {
                const double dx = rx - Rw[3 * j], dy = ry - Rw[3 * j + 1], dz = rz - Rw[3 * j + 2];
                vee += rsqrt_f64(dx * dx + dy * dy + dz * dz);
            }
        }
    }
    if (s.jas) jas_acc = warp_sum(jas_acc);
    ven = warp_sum(ven);
    vee = warp_sum(vee);
    if (lane == 0) { red[0][wid] = lap_acc; red[1][wid] = ven; red[2][wid] = vee; red[3][wid] = jas_acc; }
    __syncthreads();
    if (t < 4) {
        double x = 0.0;
        for (int q = 0; q < kEnWarps; ++q) x += red[t][q];
        total[t] = x;
    }
    if (nrank > 1 || s.jas) cluster.sync();                    // totals, and no CTA leaves while its sums are read
    else __syncthreads();
    if (t == 0 && rank == 0) {
        double lap = 0.0, Ven = 0.0, Vee = 0.0, Jt = 0.0;
        for (int r = 0; r < nrank; ++r) {
            const double *x = cluster.map_shared_rank(total, r);
            lap += x[0]; Ven += x[1]; Vee += x[2]; Jt += x[3];
        }
        const double T = -0.5 * lap;
        const double el = T + Ven + Vee + s.vnn;
        // a spin with no electrons contributes det = 1
        const double la0 = s.n_up ? logabs2[2 * w] : 0.0, la1 = s.n_dn ? logabs2[2 * w + 1] : 0.0;
        const double sg0 = s.n_up ? sign2[2 * w] : 1.0, sg1 = s.n_dn ? sign2[2 * w + 1] : 1.0;
        uint32_t st = sing[w];
        const bool singular = (st & (QMC_STATUS_SINGULAR_UP | QMC_STATUS_SINGULAR_DN)) != 0;
        const bool finite_in = !s_nonfinite;
        if (!finite_in) st |= QMC_STATUS_NONFINITE;
        if (!singular && !(isfinite(el) && isfinite(la0) && isfinite(la1) && isfinite(Jt))) st |= QMC_STATUS_NONFINITE;
        o.logpsi[wg] = singular ? -INFINITY : la0 + la1 + Jt;     // log|Psi| = log|Det_up| + log|Det_dn| + J
        o.sign[wg] = singular ? 0.0 : sg0 * sg1;
        if (o.logabs) { o.logabs[2 * wg] = la0; o.logabs[2 * wg + 1] = la1; }
        o.e_loc[wg] = el;
        if (o.e_parts) {
            o.e_parts[4 * wg] = T; o.e_parts[4 * wg + 1] = Ven;
            o.e_parts[4 * wg + 2] = Vee; o.e_parts[4 * wg + 3] = s.vnn;
        }
        o.status[wg] = st;
    }
    if (nrank > 1) cluster.sync();                             // rank 0 has read the totals
}

template <typename TG>
static cudaError_t launch_en(const SysDev &s, int nw, const double *R, const double *Dinv, const CView &cv,
                             const double *logabs2, const double *sign2, const uint32_t *sing,
                             const qmc_eval_out &o, int w_off, cudaStream_t st, const float2 *Q2)
{
    constexpr bool kMixed = std::is_same<TG, float>::value;
    const size_t N = s.n_elec, na = s.n_atom;
    // stage bit 0: the nuclei's float pairs in shared memory, bit 1: the positions in FP64 (for the
    // Jastrow pairs); without the room they are read from global memory
    int stage = 0;
    size_t sm = (s.jas ? 8 * 4 * N : 0) + (kMixed ? sizeof(float2) * 3 * N + sizeof(float) * ((na + 1) & ~size_t(1)) : 0);
    const size_t most = 200 * 1024;
    if (kMixed && sm + sizeof(float2) * 3 * na <= most) { stage |= 1; sm += sizeof(float2) * 3 * na; }
    if (s.jas && sm + 8 * 3 * N <= most) { stage |= 2; sm += 8 * 3 * N; }
    // CTAs per walker: up to 8 (the portable cluster size) while the walkers give fewer than four
    // CTAs to each of 152 SMs and each warp keeps an electron
    unsigned c = 1;
    while (c < 8 && (size_t)nw * c < 152 * 4 && N >= (size_t)2 * kEnWarps * c) c *= 2;
    cudaError_t e = allow_smem<k_drift_energy<TG>>(sm);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = c;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nw * c);
    cfg.blockDim = dim3(kEnThreads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_drift_energy<TG>, s, R, Dinv, static_cast<const TG *>(cv.g), cv, logabs2, sign2,
                           sing, o, w_off, Q2, stage);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_drift_energy(const SysDev &s, int nw, const double *R, const double *Dinv, const CView &cv,
                                const double *logabs2, const double *sign2, const uint32_t *sing,
                                const qmc_eval_out &o, int w_off, cudaStream_t st, const float2 *Q2)
{
    if (nw == 0) return cudaSuccess;
    return cv.g_f32 ? launch_en<float>(s, nw, R, Dinv, cv, logabs2, sign2, sing, o, w_off, st, Q2)
                    : launch_en<double>(s, nw, R, Dinv, cv, logabs2, sign2, sing, o, w_off, st, nullptr);
}

}  // namespace qmc
