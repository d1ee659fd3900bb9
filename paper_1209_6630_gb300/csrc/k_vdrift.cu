// The C-free variant of steps a3 + a5 (drift and Laplacian without the
// gradient and Laplacian matrices C2..C5).  From the cofactor identities of
// Sec. II.C (the two vector products) and the MO expansion Eq. (mo):
//   drift_{e,l} = sum_k (D^-1)_{ek} d_l phi_k(r_e) = sum_mu v_{e mu} d_l chi_mu(r_e)
//   lap_e       = sum_k (D^-1)_{ek} lap phi_k(r_e) = sum_mu v_{e mu} lap chi_mu(r_e)
//   v_{e mu}    = sum_k (D^-1)_{ek} a_{k mu}              (v_e = D^-1[e,:] A^T)
// with mu over the AOs that are not screened out for r_e.  Only C1 is formed
// (for the determinant and D^-1); the product v costs sum_s N_s^2 Kbar
// multiply-adds, against 4 sum_s N_s^2 Kbar for C2..C5.
//
// k_vd_rowexp: the exponent bound E of every D^-1 row (|D^-1[e,k]| < 2^E).
// k_vd_mma (one CTA per walker tile of 128 and electron e): the union of the
// tile's active AOs for e (from the shell masks), then per AO tile of 64: v
// on the tcgen05 tensor cores as M = 128 walkers x N = 64 AOs x K = N_s MOs
// from exact BF16 slices, the split of the C1 products (k_c15_tc.cu) with
// the roles of the indices exchanged: D^-1 rows scaled by 2^-E_{w,e} (sliced
// from the FP64 inverse once per CTA into a staging image in global memory
// that every AO tile copies), A rows scaled by 2^-G_mu (sliced at load), six
// slices each, the 21 slice pairs of order <= 5 into four FP32
// accumulators (orders 0, 1, 2 exact; 3..5 together); K stages of 32 MOs
// through one stage buffer per CTA, two CTAs per SM (the staged D^-1 slices
// by one bulk copy, the B rows by cp.async), a converged warp issuing the MMAs
// through elect.sync, mbarrier commits, bounded waits.  Epilogue:
// v = 2^(E + G_mu) (acc0 + acc1 + acc2 + acc3) as a float pair (the order sums
// are exact integers in their units; the power of two is applied exactly),
// and for every active AO of the walker the gradient (FP32) and Laplacian
// (float-float, radial part once per shell) of the AO at r_e, multiplied by v
// and accumulated as float pairs on the FP32 pipes.
// Output vd[w][e] = (drift_x, drift_y, drift_z, lap_e).
#include <algorithm>

#include "ao_ff.cuh"
#include "f64_bits.cuh"
#include "qmc_internal.cuh"
#include "slices.cuh"
#include "umma.cuh"

namespace qmc {

namespace {

constexpr int kVdThreads = 256;
constexpr int kVdK = 32;                                      // MOs per stage
constexpr int kVdN = 64;                                      // AOs per tile (TMEM columns per accumulator)
constexpr uint32_t kVdPlane = TC_M * kVdK * 2;                // A: [128 rows][32 K] 16-bit, 64-byte swizzle: 8 KB
constexpr uint32_t kVdBPlane = kVdN * kVdK * 2;               // B: [64 rows][32 K]: 4 KB
constexpr uint32_t kVdBuf = kC15Slices * (kVdPlane + kVdBPlane);   // 6 A planes + 6 B planes: 72 KB
constexpr int kVdAcc = 4;
static_assert(kVdThreads == kVdN * 4, "one 16-byte chunk of a B plane per thread");

struct VdArgs {
    SysDev s;
    FfBasis fb;
    const double *R;
    const uint32_t *masks;
    int mw, nw;
    const double *Dinv;            // [nw][msz] rows = electrons
    size_t msz;
    const int *rexp;               // [nw][N] row exponents of D^-1
    const uint16_t *rslice[2];     // [6][n_ao][ns_pad]
    const int *gexp[2];            // [n_ao]
    int ns_pad[2];
    double *vd;                    // [nw][N][4]
    uint32_t *wstatus;
    unsigned long long wait_ns;
    const float *pgf, *pcf, *scf;  // FP32 exponents, coefficients [n_prim], AO scales [n_ao]
    const float *Qhi, *Qlo;        // nuclear positions as float pairs [n_atom][3]
    int e0;                        // first electron of this launch's batch
    unsigned char *astage;         // per CTA of the batch: the sliced D^-1 rows, one A image per K stage
    size_t astage_per;             // bytes per CTA
    int prows;                     // rows of a staged plane: 128, or a single tile's walkers rounded up to 8
};

__global__ void k_vd_rowexp(int nw, int n_up, int n_dn, size_t msz, const double *__restrict__ Dinv,
                            int *__restrict__ rexp)
{
    const int N = n_up + n_dn;
    const size_t row = blockIdx.x * (size_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= (size_t)nw * N) return;
    const int w = (int)(row / N), e = (int)(row - (size_t)w * N);
    const int spin = e >= n_up, ns = spin ? n_dn : n_up, ei = spin ? e - n_up : e;
    const double *d = Dinv + (size_t)w * msz + (spin ? (size_t)n_up * n_up : 0) + (size_t)ei * ns;
    // the largest magnitude by its bits, one conversion per row (rounding to FP32 keeps the order):
    // a conversion per element held the FP64 pipe (1.9 ms at 1056 electrons x 2048 walkers)
    unsigned long long m = 0;
#pragma unroll 4
    for (int k = lane; k < ns; k += 32) m = max(m, abs_bits(d[k]));
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(m >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(m >> 32) == hi ? (unsigned)m : 0u);
    if (lane == 0) rexp[row] = exp_bound((float)__hiloint2double((int)hi, (int)lo));
}

// The four order sums of 16 columns of this warp's TMEM lanes (integers in their units) added
// as float pairs: column c0 + q to out[q * ld].
__device__ __forceinline__ void vd_sums(uint32_t tmem_lanes, int c0, float2 *out, int ld)
{
    uint32_t v0[16], v1[16], v2[16], v3[16];
    tmem_ld16(tmem_lanes + (uint32_t)(0 * kVdN + c0), v0);
    tmem_ld16(tmem_lanes + (uint32_t)(1 * kVdN + c0), v1);
    tmem_ld16(tmem_lanes + (uint32_t)(2 * kVdN + c0), v2);
    tmem_ld16(tmem_lanes + (uint32_t)(3 * kVdN + c0), v3);
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        float s, e, s2, e2;
        ff::two_sum(__uint_as_float(v0[q]), __uint_as_float(v1[q]), s, e);
        ff::two_sum(s, __uint_as_float(v2[q]), s2, e2);
        e = __fadd_rn(e, e2);
        ff::two_sum(s2, __uint_as_float(v3[q]), s, e2);
        out[q * ld] = ff::renorm(s, __fadd_rn(e, e2));
    }
}

// Laplacian (float-float) and gradient (FP32) of one AO from its shell's radial part; the degrees
// 0, 1 and 2 written out (ao_ff.cuh), the same values as the general expressions below.
__device__ __forceinline__ void vd_derivs(const SysDev &s, const VdArgs &a, int mu, const FfRadial &rd, float2 &lp,
                                          float &g1, float &g2, float &g3)
{
    const int pw2 = s.ao_pow[mu], L = ao_degree(pw2);
    const float dx = rd.dx.x + rd.dx.y, dy = rd.dy.x + rd.dy.y, dz = rd.dz.x + rd.dz.y;
    const float g = rd.g.x + rd.g.y, m2gd = -2.f * (rd.gd.x + rd.gd.y);
    const float c = a.scf[mu];
    if (L <= 2) {
        const float2 cf = a.fb.sc[mu];
        if (L == 0) {
            lp = ff::mul(cf, rd.gl);
            g1 = c * (m2gd * dx);
            g2 = c * (m2gd * dy);
            g3 = c * (m2gd * dz);
            return;
        }
        int xa, xb;
        ao_axes(pw2, xa, xb);
        const float2 fa = pick3(xa, rd.dx, rd.dy, rd.dz);
        const float2 q = ff::sub(rd.gl, ff::mulf(rd.gd, (float)(4 * L)));
        const float da = pick3(xa, dx, dy, dz);
        float P = da, xA = 1.f, xB = 0.f;                  // d P / d axis a, d P / d axis b
        float2 fP = fa;
        if (L == 2) {
            const float db = pick3(xb, dx, dy, dz);
            P = da * db;
            xA = xa == xb ? 2.f * da : db;
            xB = da;
            fP = ff::mul(fa, pick3(xb, rd.dx, rd.dy, rd.dz));
        }
        lp = ff::mul(cf, xa == xb ? ff::fma2(make_float2(2.f * rd.g.x, 2.f * rd.g.y), fP, q) : ff::mul(fP, q));
        const float X0 = xa == 0 ? xA : 0.f;               // (axis b is never 0 unless a is)
        const float X1 = xa == 1 ? xA : (xb == 1 ? xB : 0.f);
        const float X2 = xa == 2 ? xA : (xb == 2 ? xB : 0.f);
        g1 = c * fmaf(__fmul_rn(m2gd, dx), P, __fmul_rn(X0, g));
        g2 = c * fmaf(__fmul_rn(m2gd, dy), P, __fmul_rn(X1, g));
        g3 = c * fmaf(__fmul_rn(m2gd, dz), P, __fmul_rn(X2, g));
        return;
    }
    float2 val;
    ff_angular(s, a.fb, mu, rd, val, lp);
    const int nx = pw2 & 255, ny = (pw2 >> 8) & 255, nz = (pw2 >> 16) & 255;
    auto ip = [](float x, int n) {
        float y = 1.f;
        for (int i = 0; i < n; ++i) y *= x;
        return y;
    };
    const float px = ip(dx, nx), py = ip(dy, ny), pz = ip(dz, nz);
    const float P = px * py * pz;
    g1 = c * ((nx ? nx * ip(dx, nx - 1) : 0.f) * py * pz * g + m2gd * dx * P);
    g2 = c * (px * (ny ? ny * ip(dy, ny - 1) : 0.f) * pz * g + m2gd * dy * P);
    g3 = c * (px * py * (nz ? nz * ip(dz, nz - 1) : 0.f) * g + m2gd * dz * P);
}

// Two CTAs per SM (256 threads, N = 64 AOs per tile, one operand stage of
// 72 KB, 256 TMEM columns each): one CTA's epilogue (the AO derivatives, the
// larger part of the work) runs while the other's copies and MMAs proceed.
__global__ void __launch_bounds__(kVdThreads, 2) k_vd_mma(VdArgs a)
{
    extern __shared__ __align__(1024) unsigned char vd_smem[];
    unsigned char *base = vd_smem + ((1024 - (smem_u32(vd_smem) & 1023)) & 1023);
    int *ao_s = reinterpret_cast<int *>(base + kVdBuf);       // [n_ao + kVdN]
    __shared__ uint32_t un_s[256];
    __shared__ int warp_s[kVdThreads / 32];
    __shared__ __align__(8) uint64_t mbar, cbar;
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort;

    const SysDev &s = a.s;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int tile = blockIdx.x, e = a.e0 + (int)blockIdx.y;
    unsigned char *ast = a.astage + ((size_t)blockIdx.y * gridDim.x + tile) * a.astage_per;
    const int N = s.n_elec;
    const int spin = e >= s.n_up, ei = spin ? e - s.n_up : e, ns = spin ? s.n_dn : s.n_up;
    const int nspad = a.ns_pad[spin];
    const int mw = a.mw;

    // union of the tile's active shells for electron e, and its AO list
    const int rv = min(TC_M, a.nw - tile * TC_M);             // walkers of this tile
    for (int j = t; j < mw; j += kVdThreads) un_s[j] = 0;
    __syncthreads();
    for (int q = t; q < rv * mw; q += kVdThreads) {           // independent loads: a word each
        const int m = q / mw, j = q - m * mw;
        const uint32_t u = a.masks[((size_t)(tile * TC_M + m) * N + e) * mw + j];
        if (u) atomicOr(&un_s[j], u);
    }
    __syncthreads();
    const int K = aos_from_mask_n(s, un_s, mw, ao_s, warp_s);
    const int nat = (K + kVdN - 1) / kVdN;
    for (int q = K + t; q < nat * kVdN; q += kVdThreads) ao_s[q] = -1;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;"
                     :: "r"(smem_u32(&tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (t == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&mbar)) : "memory");
        mbar_init(smem_u32(&cbar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const uint32_t mb = smem_u32(&mbar);
    const uint64_t kWait = a.wait_ns;
    const uint16_t *Bsl = a.rslice[spin];
    const size_t bstride = (size_t)s.n_ao * nspad;
    // K stops at the last 32 MOs that exist and the last AO tile's N at its AOs rounded up to 16 (the
    // rest is zeros): 158 electrons x 100 walkers 325 -> 294 us, 434 x 4096 22.2 -> 21.0 ms
    const int nst = (ns + kVdK - 1) / kVdK;

    // this CTA's D^-1 rows cut into six exact slices once, for every K stage (the AO tiles
    // reuse them): thread -> (row, chunk of 8 MOs), two per thread
    const uint32_t pbytes = (uint32_t)a.prows * (kVdK * 2);   // a staged plane's rows (the others feed unread lanes)
    for (int q = t; q < a.prows * 4; q += kVdThreads) {
        const int prow = q >> 2, pc = q & 3;
        const int pw = tile * TC_M + prow;
        const bool pvalid = pw < a.nw;
        const double *drow = a.Dinv + (size_t)(pvalid ? pw : 0) * a.msz + (spin ? (size_t)s.n_up * s.n_up : 0) +
                             (size_t)ei * ns;
        const int Ep = pvalid ? a.rexp[(size_t)pw * N + e] : 0;
        for (int sg = 0; sg < nst; ++sg) {
            const int k0 = sg * kVdK;
            float sl[8][kC15Slices];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int k = k0 + 8 * pc + i;
                const double d = (pvalid && k < ns) ? drow[k] : 0.0;
                slice6(ff::from_double(d), Ep, sl[i]);
            }
            unsigned char *Ad = ast + (size_t)sg * kC15Slices * pbytes;
#pragma unroll
            for (int j = 0; j < kC15Slices; ++j)
                *reinterpret_cast<uint4 *>(Ad + j * pbytes + a_off64(prow, pc)) =
                    make_uint4(bf16_pair(sl[0][j], sl[1][j]), bf16_pair(sl[2][j], sl[3][j]),
                               bf16_pair(sl[4][j], sl[5][j]), bf16_pair(sl[6][j], sl[7][j]));
        }
    }
    asm volatile("fence.proxy.async.global;" ::: "memory");   // the staging is read back by bulk copies
    __syncthreads();                                       // the block's global writes, before the copies read them
    const uint32_t cb = smem_u32(&cbar);
    int ncopy = 0;

    // epilogue role: a full tile has walker row erow (TMEM lane), columns cg * 32 .. + 32 of an AO
    // tile of 64.  A tile of at most 64 walkers hands the columns of a row to 256 / rp threads
    // (rp: the power of two that holds the rows), each a run of 64 rp / 256 of them, through
    // shared memory: the AO derivatives of one walker's column group are a serial chain, and most
    // lanes have no row there (1056 electrons x 37 walkers, with all electrons in one launch:
    // 16.8 -> 2.8 ms).
    const int lrp = 32 - __clz(rv - 1);                       // rv = 1: __clz(0) = 32
    const bool small = lrp < 7;
    const int erow = small ? t & ((1 << lrp) - 1) : (warp & 3) * 32 + lane;
    const int cg = small ? t >> lrp : warp >> 2;              // column group
    const int ncg = small ? kVdThreads >> lrp : 2;            // column groups, each of len columns
    const int len = small ? max(1, kVdN >> (8 - lrp)) : 32;
    const int ew = tile * TC_M + erow;
    const bool evalid = erow < rv;
    const int Ee = evalid ? a.rexp[(size_t)ew * N + e] : 0;
    const double *rw = a.R + ((size_t)(evalid ? ew : 0) * N + e) * 3;
    const float2 r2[3] = {ff::from_double(rw[0]), ff::from_double(rw[1]), ff::from_double(rw[2])};
    const uint32_t *my_mask = a.masks + ((size_t)(evalid ? ew : 0) * N + e) * mw;
    const uint32_t tlane = (uint32_t)((warp & 3) * 32) << 16;
    // drift and Laplacian accumulated as float pairs on the FP32 pipes (GB300's FP64 rate is 1/64
    // of FP32: FP64 sums here kept the FP64 pipe 30% busy)
    float2 b0 = make_float2(0.f, 0.f), b1 = b0, b2 = b0, lap = b0;

    int ncommit = 0;
    bool ok = true;
    unsigned char *Ab = base;
    unsigned char *Bb = base + kC15Slices * kVdPlane;
    for (int at = 0; at < nat && ok; ++at) {
        // this thread's chunk of a B row in every slice plane and stage of the tile
        const int bmu = ao_s[at * kVdN + (t >> 2)];
        const uint16_t *bsrc = Bsl + (size_t)max(bmu, 0) * nspad + 8 * (t & 3);
        const uint32_t bdst = smem_u32(Bb + a_off64(t >> 2, t & 3));
        const int ncol = min(kVdN, (K - at * kVdN + 15) / 16 * 16);              // N of the tile's MMAs
        const uint32_t idesc = umma_idesc_f16_major(TC_M, ncol, 1, 0, 0);        // BF16, A and B K-major
        for (int sg = 0; sg < nst; ++sg) {
            // the stage buffer: A (the staged D^-1 slices) and B (the rows of A of this AO tile)
            const int k0 = sg * kVdK;
            const unsigned char *As = ast + (size_t)sg * kC15Slices * pbytes;
            if (t == 0) {                                  // the staged D^-1 slices: one bulk copy
                mbar_expect_tx(cb, kC15Slices * pbytes);
                if (pbytes == kVdPlane) bulk_g2s(smem_u32(Ab), As, kC15Slices * kVdPlane, cb);
                else
                    for (int j = 0; j < kC15Slices; ++j)
                        bulk_g2s(smem_u32(Ab + j * kVdPlane), As + (size_t)j * pbytes, pbytes, cb);
            }
#pragma unroll
            for (int j = 0; j < kC15Slices; ++j)
                if ((t >> 2) < ncol) cp_async16(bdst + j * kVdBPlane, bsrc + j * bstride + k0, bmu >= 0);
            asm volatile("cp.async.commit_group;" ::: "memory");
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            ++ncopy;
            // one warp observes the bulk copy (only the MMA issue reads it); the others wait at
            // the barrier without spending issue slots the other CTA's epilogue needs
            if (warp == 0 && !mbar_wait(cb, (ncopy - 1) & 1, kWait)) s_abort = 1;
            __syncthreads();
            if (warp == 0) {                                   // converged: elect.sync per MMA
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t dA = umma_desc_sw64(smem_u32(Ab), 512);
                const uint64_t dB = umma_desc_sw64(smem_u32(Bb), 512);
#pragma unroll
                for (int kk = 0; kk < kVdK / 16; ++kk)
#pragma unroll
                    for (int d = 0; d < kC15Slices; ++d) {
                        const int acc = d < kVdAcc - 1 ? d : kVdAcc - 1;
#pragma unroll
                        for (int i = 0; i <= d; ++i) {
                            const int j = d - i;
                            const uint64_t ad = dA + ((i * kVdPlane + 32 * kk) >> 4);
                            const uint64_t bd = dB + ((j * kVdBPlane + 32 * kk) >> 4);
                            const bool first = sg == 0 && kk == 0 && i == 0 && d <= kVdAcc - 1;
                            umma_bf16_warp(tmem + acc * kVdN, ad, bd, idesc, first ? 0u : 1u);
                        }
                    }
                umma_commit_warp(mb);
            }
            ++ncommit;
            // the buffer is rewritten by the next stage: wait for these MMAs (the other CTA
            // on the SM keeps the tensor pipe busy meanwhile)
            if (warp == 0 && !mbar_wait(mb, (ncommit - 1) & 1, kWait)) s_abort = 1;
            __syncthreads();
            if (s_abort) break;
        }
        ok = !s_abort;
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // epilogue: v for 32 AOs of this walker row, then the AO derivatives at r_e
        FfRadial rd;
        int last_sh = -1;
        bool on = false;                                   // last_sh is active for this walker
        // the stage buffer is idle here: [16][256] of the threads' own columns, or [64][64 rows]
        float2 *vbuf = reinterpret_cast<float2 *>(base);
        const int vld = small ? TC_M / 2 : kVdThreads;
        if (small) {
            const int lrow = (warp & 3) * 32 + lane;       // TMEM lane
            if ((warp & 3) * 32 < rv)                      // (whole warps)
                for (int h = 0; h < 2; ++h)
                    vd_sums(tmem + tlane, (warp >> 2) * 32 + h * 16, vbuf + ((warp >> 2) * 32 + h * 16) * vld + lrow, vld);
            __syncthreads();
        }
        for (int h = 0; h < (small ? 1 : 2); ++h) {
            const int c0 = small ? cg * len : cg * 32 + h * 16;
            const float2 *vcol = small ? vbuf + c0 * vld + erow : vbuf + t;
            if (!small) vd_sums(tmem + tlane, c0, vbuf + t, vld);
            if (!evalid) continue;
            const int nq = small ? len : 16;
#pragma unroll 1
            for (int q = 0; q < nq; ++q) {
                if (c0 + q >= kVdN) break;                 // (rp <= 2: more threads than columns)
                const int mu = ao_s[at * kVdN + c0 + q];
                if (mu < 0) break;
                const int sh = s.ao_shell[mu];
                if (sh != last_sh) {
                    last_sh = sh;
                    on = (my_mask[sh >> 5] >> (sh & 31)) & 1u;
                    if (on) ff_radial(s, a.fb, sh, r2, rd);
                }
                if (!on) continue;
                const int ex = Ee + a.gexp[spin][mu];
                const float2 vr = vcol[q * vld];
                const float2 vmu = make_float2(scale_pow2(vr.x, ex), scale_pow2(vr.y, ex));   // exact scaling
                // Laplacian in float-float (the kinetic term cancels against the potential: an FP32
                // Laplacian left E_L at 2e-5 relative on 2048 walkers of 1056 electrons), the
                // gradient in FP32 from the same radial part; products with v as float pairs
                float2 lp;
                float g1, g2, g3;
                vd_derivs(s, a, mu, rd, lp, g1, g2, g3);
                b0 = ff::fma2(b0, vmu, make_float2(g1, 0.f));
                b1 = ff::fma2(b1, vmu, make_float2(g2, 0.f));
                b2 = ff::fma2(b2, vmu, make_float2(g3, 0.f));
                lap = ff::fma2(lap, vmu, lp);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // vbuf before the next tile's bulk copy
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();                                   // TMEM and vbuf read before the next tile
    }
    if (!ok) {
        if (t < TC_M && tile * TC_M + t < a.nw) atomicOr(a.wstatus + tile * TC_M + t, (uint32_t)QMC_STATUS_TIMEOUT);
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (ncopy > 0) mbar_wait(cb, (ncopy - 1) & 1, kDrainNs);        // the last bulk copy
        if (ncommit > 0) mbar_wait(mb, (ncommit - 1) & 1, kDrainNs);   // let MMAs in flight drain
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" :: "r"(tmem) : "memory");
    // the column groups' partial sums of each row, added in a fixed order
    double *red = reinterpret_cast<double *>(base);        // [groups][rows][4]; operands no longer read
    const int rows = kVdThreads / ncg;                     // 128, or rp
    double *mine = red + ((size_t)cg * rows + erow) * 4;
    mine[0] = ff::val(b0);
    mine[1] = ff::val(b1);
    mine[2] = ff::val(b2);
    mine[3] = ff::val(lap);
    __syncthreads();
    for (int q = t; q < rv * 4; q += kVdThreads) {
        const int r = q >> 2, c = q & 3;
        const int w = tile * TC_M + r;
        double x = red[(size_t)r * 4 + c];
        for (int g = 1; g < ncg; ++g) x += red[((size_t)g * rows + r) * 4 + c];
        a.vd[((size_t)w * N + e) * 4 + c] = ok ? x : __longlong_as_double(0x7ff8000000000000ll);
    }
}

}  // namespace

bool vdrift_fits(const SysDev &s)
{
    const size_t sm = 1024 + (size_t)kVdBuf + sizeof(int) * ((size_t)s.n_ao + kVdN);
    return sm <= 227 * 1024;
}

// Electrons per launch (the A staging holds one image per CTA of a batch), spread evenly over
// the launches.  The least that a workspace must hold: up to 264 from 2 walker tiles on, else
// up to 64 (one walker's scratch stays small); never smaller for more tiles, so what holds a
// walker chunk holds a shorter one.
static int vdrift_spread(int n_elec, size_t b)
{
    if ((size_t)n_elec <= b) return n_elec;
    const int nl = (int)((n_elec + b - 1) / b);
    return (n_elec + nl - 1) / nl;
}

static int vdrift_least(const SysDev &s, int tiles) { return vdrift_spread(s.n_elec, tiles >= 2 ? 264 : 64); }

static size_t vdrift_stage_per(const SysDev &s, int nw)
{
    const int nsmax = s.n_up > s.n_dn ? s.n_up : s.n_dn;
    const size_t nst = (size_t)((nsmax + 63) / 64 * 64) / kVdK;
    const size_t prows = nw >= TC_M ? TC_M : (nw + 7) / 8 * 8;
    return nst * kC15Slices * prows * (kVdK * 2);
}

// The batch that fills the card: 2432 (electron, tile) pairs are eight waves of two CTAs on
// each of 152 SMs, within 4 GiB.
static int vdrift_want(const SysDev &s, int nw)
{
    const size_t tiles = (size_t)(nw + TC_M - 1) / TC_M;
    const size_t room = (size_t(4) << 30) / (tiles * std::max(vdrift_stage_per(s, nw), size_t(1)));
    const size_t b = std::min((2432 + tiles - 1) / tiles, std::max(room, size_t(1)));
    return std::max(vdrift_least(s, (int)tiles), vdrift_spread(s.n_elec, b));
}

static size_t vdrift_head(const SysDev &s, int nw)           // the row exponents of D^-1
{
    return ((sizeof(int) * (size_t)nw * s.n_elec + 255) / 256) * 256;
}

size_t vdrift_bytes(const SysDev &s, int nw, bool want)
{
    const size_t tiles = (size_t)(nw + TC_M - 1) / TC_M;
    return vdrift_head(s, nw) +
           tiles * (size_t)(want ? vdrift_want(s, nw) : vdrift_least(s, (int)tiles)) * vdrift_stage_per(s, nw);
}

size_t vdrift_tile_bytes(const SysDev &s, int nw)
{
    const size_t tiles = (size_t)(nw + TC_M - 1) / TC_M;
    return vdrift_head(s, nw) + tiles * (size_t)vdrift_least(s, (int)tiles) * vdrift_stage_per(s, TC_M);
}

cudaError_t launch_vdrift(const SysDev &s, const FfBasis &fb, const MixedTables &mt, int nw, const double *R,
                          const uint32_t *masks, int mw, const double *Dinv, double *vd, uint32_t *wstatus,
                          void *scratch, size_t scratch_bytes, cudaStream_t st, const WaitCfg &wc)
{
    if (nw == 0) return cudaSuccess;
    if (scratch_bytes < vdrift_bytes(s, nw, false)) return cudaErrorMemoryAllocation;
    if (!vdrift_fits(s)) return cudaErrorInvalidConfiguration;
    VdArgs a;
    a.s = s; a.fb = fb; a.R = R; a.masks = masks; a.mw = mw; a.nw = nw; a.Dinv = Dinv;
    a.msz = (size_t)s.n_up * s.n_up + (size_t)s.n_dn * s.n_dn;
    a.rexp = static_cast<const int *>(scratch);
    for (int spin = 0; spin < 2; ++spin) {
        a.rslice[spin] = mt.rslice[spin];
        a.gexp[spin] = mt.gexp[spin];
        a.ns_pad[spin] = mt.ns_pad[spin];
    }
    a.vd = vd;
    a.wstatus = wstatus;
    a.pgf = mt.pgf; a.pcf = mt.pcf; a.scf = mt.scf; a.Qhi = mt.Qhi; a.Qlo = mt.Qlo;
    a.astage = static_cast<unsigned char *>(scratch) + vdrift_head(s, nw);
    a.astage_per = vdrift_stage_per(s, nw);
    a.prows = nw >= TC_M ? TC_M : (nw + 7) / 8 * 8;
    a.wait_ns = wc.limit_ns;
    const size_t rows = (size_t)nw * s.n_elec;
    k_vd_rowexp<<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(nw, s.n_up, s.n_dn, a.msz, Dinv,
                                                          static_cast<int *>(scratch));
    const size_t sm = 1024 + (size_t)kVdBuf + sizeof(int) * ((size_t)s.n_ao + kVdN);
    cudaError_t e = allow_smem<k_vd_mma>(sm);
    if (e != cudaSuccess) return e;
    const int tiles = (nw + TC_M - 1) / TC_M;
    // as many electrons per launch as the scratch holds, up to the batch that fills the card
    const size_t room = (scratch_bytes - vdrift_head(s, nw)) / (tiles * std::max(a.astage_per, size_t(1)));
    const int nb = std::min(vdrift_want(s, nw), vdrift_spread(s.n_elec, std::max(room, size_t(1))));
    for (int e0 = 0; e0 < s.n_elec; e0 += nb) {
        a.e0 = e0;
        const int ne = s.n_elec - e0 < nb ? s.n_elec - e0 : nb;
        k_vd_mma<<<dim3(tiles, ne), kVdThreads, sm, st>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace qmc
