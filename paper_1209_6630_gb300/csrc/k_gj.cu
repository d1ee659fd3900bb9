// Step a4: log|det|, sign and inverse of each Slater matrix in FP64
// (Sec. II.C: D^-1 for the drift/Laplacian vector products; Sec. IV.B: the
// inversion step, double precision).
//
// One CTA per matrix.  Gauss-Jordan elimination with partial pivoting, done
// in panels of NB = 8, 16 or 32 columns (a tile choice per system):
//   1. the n x NB panel is copied to shared memory and eliminated there,
//      column by column (pivot = largest |entry| among rows not yet used;
//      the pivots are exactly those of LU with partial pivoting);
//   2. every other column j of the matrix receives the panel's row
//      operations at once, as a rank-NB update
//        X[i][j] <- [i not a pivot row] X[i][j] + sum_c P[i][c] X[piv_c][j]
//      (P = the eliminated panel, which holds the composite row operations).
// (Matrices too few for one CTA each to fill the card: launch_gj_wide, k_gj_redo.cu.)
// The panel (gj_panel.cuh) was a third of the time with 16-way bank conflicts, a division and
// FP64 compares in every thread: 300 matrices of n = 217 7.95 -> 6.14 ms, 400 of n = 528 122 -> 116.
// Pivoting is implicit: rows never move in memory; a row map records which
// physical row was the pivot of each step.  After the last panel the array
// holds Res with X^-1[a][b] = Res[pp[a]][ipp[b]] (pp = pivot rows, ipp its
// inverse), and the kernel writes Dinv = X^-T with a tiled transpose:
//   Dinv[pp[c]][k] = Res[pp[k]][c].
// Flops: n^3 FMA = 2 n^3, the LU (2/3 n^3) plus inverse (4/3 n^3) count.
// Shared memory (n NB + 32 NB) doubles + 3n shorts: at NB = 16, ~75 KB for n = 528
// (three CTAs per SM); NB = 8 halves it at the cost of twice the panel sweeps.
#include <math.h>

#include "f64_bits.cuh"
#include "ff_math.cuh"
#include "gj_panel.cuh"
#include "qmc_internal.cuh"

namespace qmc {

constexpr int kGjThreads = 256;
constexpr int kGjWarps = kGjThreads / 32;

struct GjJobs2 {
    GjJob j[2];
};

// doubles reserved for the panel (also holds the 32 x 33 transpose tile)
__host__ __device__ __forceinline__ size_t p_region(int n, int nb)
{
    const size_t a = (size_t)n * nb;
    return a > 32 * 33 ? a : 32 * 33;
}

// bytes of the float-float panel as row pairs (at the end two 32 x 33 transpose tiles lie there)
__host__ __device__ __forceinline__ size_t gjff_p_bytes(int n, int nb)
{
    const size_t a = (size_t)((n + 1) / 2) * nb * 16;
    return a > 2 * 32 * 33 * 8 ? a : 2 * 32 * 33 * 8;
}

// ... with the pivot rows' tile [NB][32], the pivot map and the panel's row flags
__host__ __device__ __forceinline__ size_t gjff_fixed_bytes(int n, int nb)
{
    return (gjff_p_bytes(n, nb) + sizeof(float2) * nb * 32 + sizeof(short) * (2 * (size_t)n + 2) + 15) / 16 * 16;
}

template <int NB>
__global__ void __launch_bounds__(kGjThreads, NB == 32 ? 1 : 3) k_gj(GjJobs2 jobs)
{
    const GjJob &J = jobs.j[blockIdx.y];
    const int m = blockIdx.x;
    if (m >= J.count) return;
    if (J.only_redo && J.redo[m * J.redo_stride] != 1) return;   // recompute pass: flagged, not yet handled
    const int n = J.n;
    double *__restrict__ X = J.X + (size_t)m * J.x_stride;
    double *__restrict__ Dout = J.Dinv + (size_t)m * J.d_stride;

    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *P = reinterpret_cast<double *>(smem_raw);   // [n][NB], later a [32][33] tile
    double *U = P + p_region(n, NB);                      // [NB][32]
    short *used = reinterpret_cast<short *>(U + NB * 32); // [n] 1 once a row has been a pivot
    short *pp = used + n;                                 // [n] pivot row of step k
    short *rowc = pp + n;                                 // [n] panel column of a pivot row, or -1
    GjPanelShared<NB> *Sp;
    if constexpr (NB == 32) {        // in U, idle while a panel is eliminated: these panels fill the shared memory
        static_assert(NB < 32 || sizeof(GjPanelShared<NB>) <= sizeof(double) * NB * 32, "S lies in U");
        Sp = reinterpret_cast<GjPanelShared<NB> *>(U);
    } else {
        __shared__ GjPanelShared<NB> own;
        Sp = &own;
    }
    GjPanelShared<NB> &S = *Sp;

    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    for (int i = t; i < n; i += kGjThreads) { used[i] = 0; rowc[i] = -1; }
    bool sing = false;
    double logabs = 0.0;
    int neg = 0;
    __syncthreads();

    for (int jb = 0; jb < n; jb += NB) {
        const int w = min(NB, n - jb);
        for (int q = t; q < n * NB; q += kGjThreads) {
            const int i = q / NB, c = q - i * NB;
            P[gj_at<NB>(i, c)] = (c < w) ? X[(size_t)i * n + jb + c] : 0.0;
        }
        __syncthreads();
        if (!gj_panel<NB>(P, n, w, used, S)) { sing = true; break; }
        if (wid == 0) {
            gj_add_pivots<NB>(S, w, logabs, neg);
            if (lane < w) {
                pp[jb + lane] = S.pp[lane];
                rowc[S.pp[lane]] = (short)lane;
            }
        }

        // store the eliminated panel
        for (int q = t; q < n * w; q += kGjThreads) {
            const int i = q / w, c = q - i * w;
            X[(size_t)i * n + jb + c] = P[gj_at<NB>(i, c)];
        }

        // rank-w update of every other column, 32 columns at a time; the pivot
        // rows of the next chunk are read into registers while this one runs
        int c0 = 0;
        auto skip = [&](int cc0) { return cc0 >= jb && cc0 + 32 <= jb + w; };
        while (c0 < n && skip(c0)) c0 += 32;
        constexpr int UPT = NB * 32 / kGjThreads;   // U elements per thread
        double upre[UPT];
        __syncthreads();   // panel stores done before U reads of the same rows
#pragma unroll
        for (int r = 0; r < UPT; ++r) {
            const int q = t + r * kGjThreads, c = q >> 5, col = c0 + (q & 31);
            upre[r] = (c0 < n && c < w && col < n) ? X[(size_t)pp[jb + c] * n + col] : 0.0;
        }
        while (c0 < n) {
            __syncthreads();   // previous chunk done with U
#pragma unroll
            for (int r = 0; r < UPT; ++r) U[t + r * kGjThreads] = upre[r];
            __syncthreads();
            int c1 = c0 + 32;
            while (c1 < n && skip(c1)) c1 += 32;
#pragma unroll
            for (int r = 0; r < UPT; ++r) {
                const int q = t + r * kGjThreads, c = q >> 5, col = c1 + (q & 31);
                upre[r] = (c1 < n && c < w && col < n) ? X[(size_t)pp[jb + c] * n + col] : 0.0;
            }
            const int col = c0 + lane;
            const bool active = col < n && !(col >= jb && col < jb + w);
            double u[NB];
#pragma unroll
            for (int c = 0; c < NB; ++c) u[c] = U[c * 32 + lane];
            if (active) {
                int i = wid;
                for (; i + 3 * kGjWarps < n; i += 4 * kGjWarps) {
                    double x[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int ii = i + r * kGjWarps;
                        x[r] = (rowc[ii] >= 0) ? 0.0 : X[(size_t)ii * n + col];
                    }
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int ii = i + r * kGjWarps;
#pragma unroll
                        for (int c2 = 0; c2 < NB / 2; ++c2) {
                            const double2 pv = *reinterpret_cast<const double2 *>(P + gj_at<NB>(ii, 2 * c2));
                            x[r] = fma(pv.x, u[2 * c2], x[r]);
                            x[r] = fma(pv.y, u[2 * c2 + 1], x[r]);
                        }
                    }
#pragma unroll
                    for (int r = 0; r < 4; ++r) X[(size_t)(i + r * kGjWarps) * n + col] = x[r];
                }
                for (; i < n; i += kGjWarps) {
                    double x = (rowc[i] >= 0) ? 0.0 : X[(size_t)i * n + col];
#pragma unroll
                    for (int c2 = 0; c2 < NB / 2; ++c2) {
                        const double2 pv = *reinterpret_cast<const double2 *>(P + gj_at<NB>(i, 2 * c2));
                        x = fma(pv.x, u[2 * c2], x);
                        x = fma(pv.y, u[2 * c2 + 1], x);
                    }
                    X[(size_t)i * n + col] = x;
                }
            }
            c0 = c1;
        }
        __syncthreads();
        for (int c = t; c < w; c += kGjThreads) rowc[pp[jb + c]] = -1;
        __syncthreads();
    }

    if (sing) {
        const double qnan = __longlong_as_double(0x7ff8000000000000ll);
        for (size_t q = t; q < (size_t)n * n; q += kGjThreads) Dout[q] = qnan;
        if (t == 0) {
            if (J.logabs) J.logabs[(size_t)m * J.la_stride] = -INFINITY;
            if (J.sign) J.sign[(size_t)m * J.la_stride] = 0.0;
            if (J.flag) atomicOr(J.flag + m, J.flag_bit);
        }
        return;
    }
    __syncthreads();   // all panel writes to X visible to the block

    // Dinv[pp[c]][k] = Res[pp[k]][c], 32 x 32 tiles through shared memory
    double *tile = P;   // [32][33]
    for (int kb = 0; kb < n; kb += 32) {
        for (int cb = 0; cb < n; cb += 32) {
            for (int r = wid; r < 32; r += kGjWarps) {
                const int k = kb + r, c = cb + lane;
                tile[r * 33 + lane] = (k < n && c < n) ? X[(size_t)pp[k] * n + c] : 0.0;
            }
            __syncthreads();
            for (int r = wid; r < 32; r += kGjWarps) {
                const int c = cb + r, k = kb + lane;
                if (c < n && k < n) Dout[(size_t)pp[c] * n + k] = tile[lane * 33 + r];
            }
            __syncthreads();
        }
    }

    if (t == 0) {
        // sign of the row permutation k -> pp[k]: parity from its cycles
        int par = 0;
        for (int i = 0; i < n; ++i) used[i] = 0;
        for (int i = 0; i < n; ++i) {
            if (used[i]) continue;
            int len = 0, j = i;
            while (!used[j]) { used[j] = 1; j = pp[j]; ++len; }
            par ^= ((len & 1) == 0);
        }
        if (J.logabs) J.logabs[(size_t)m * J.la_stride] = logabs;
        if (J.sign) J.sign[(size_t)m * J.la_stride] = (par ^ neg) ? -1.0 : 1.0;
    }
}

template <int NB>
static cudaError_t launch_gj_nb(const GjJobs2 &js, int n_jobs, int nmax, int cmax, cudaStream_t st)
{
    const size_t sm = sizeof(double) * (p_region(nmax, NB) + NB * 32) + sizeof(short) * 3 * (size_t)nmax;
    cudaError_t e = allow_smem<k_gj<NB>>(sm);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_gj<NB>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    dim3 grid(cmax, n_jobs);
    k_gj<NB><<<grid, kGjThreads, sm, st>>>(js);
    return cudaGetLastError();
}

// Whether to spread each matrix over many CTAs (launch_gj_wide, two launches per panel) rather
// than to give it one (k_gj).  An SM's FP64 pipe takes as long for one matrix in k_gj whatever
// the others do, so the call takes ceil(T / 152) matrices' time; spread, T / 152 and the panels'
// latency and launches, 2500 / n^2 of it (the excess over T / 152 at which the two meet, read off sizes
// 32 .. 434 x 1 .. 2000 matrices; at 32 rows k_gj is as fast or faster at every T).  Measured (ms, k_gj /
// spread): n = 33: T = 4 0.126 / 0.123, 200 0.147 / 0.168; n = 48: 50 0.158 / 0.152, 200 0.193 / 0.210; n = 64:
// 4 0.225 / 0.182, 50 0.228 / 0.208, 200 0.290 / 0.278, 400 0.346 / 0.388; n = 100: 50 0.611 / 0.408, 100 0.612 /
// 0.557, 400 1.295 / 1.309; n = 160: 100 1.43 / 1.24, 700 5.75 / 5.90; n = 217: 4 3.34 / 0.76, 100 3.38 / 2.52, 200
// 6.10 / 4.65, 400 8.86 / 8.34, 700 14.7 / 14.5, 2000 40.5 / 40.0; n = 528: 4 40.2 / 4.5, 150 42.8 / 40.5, 400 116 / 103;
// n = 866: 1 176 / 7.6, 150 190 / 173.
static bool gj_wide(int n, long long T)
{
    return n > 32 && (n >= 512 || (T + 151) / 152 * 152 * n * n > T * (n * n + 2500));
}

cudaError_t launch_gj(const GjJob *jobs, int n_jobs, cudaStream_t st, int nb)
{
    GjJobs2 js;
    GjJob wide[2];
    int n_wide = 0, wmax = 0;
    long long T = 0;
    for (int q = 0; q < 2; ++q) {
        js.j[q] = jobs[q < n_jobs ? q : 0];
        if (q >= n_jobs) js.j[q].count = 0;
        const GjJob &J = js.j[q];
        // matrices of one row have no room for the spread elimination's state (a spin of one electron)
        if (J.count == 0 || J.only_redo || gj_state_bytes(J.n) > sizeof(double) * (size_t)J.n * J.n) continue;
        wide[n_wide++] = J;
        wmax = max(wmax, J.n);
        T += J.count;
    }
    if (n_wide && gj_wide(wmax, T)) {
        const cudaError_t e = launch_gj_wide(wide, n_wide, st, nb);
        if (e != cudaSuccess) return e;
        for (int q = 0; q < 2; ++q)
            if (gj_state_bytes(js.j[q].n) <= sizeof(double) * (size_t)js.j[q].n * js.j[q].n) js.j[q].count = 0;
    }
    int nmax = 0, cmax = 0;
    for (int q = 0; q < 2; ++q) {
        if (js.j[q].count == 0) continue;
        nmax = max(nmax, js.j[q].n);
        cmax = max(cmax, js.j[q].count);
    }
    if (cmax == 0) return cudaSuccess;
    switch (nb) {
    case 8: return launch_gj_nb<8>(js, n_jobs, nmax, cmax, st);
    case 16: return launch_gj_nb<16>(js, n_jobs, nmax, cmax, st);
    case 32: return launch_gj_nb<32>(js, n_jobs, nmax, cmax, st);
    default: return cudaErrorInvalidValue;
    }
}


// ---------------------------------------------------------------------------
// Float-float Gauss-Jordan (mixed path, a4 arithmetic QMC_A4_FLOAT_FLOAT).  Same elimination as k_gj, but every
// value is a pair of floats (hi + lo, ~48-bit significand) and the arithmetic
// runs on the FP32 pipes (62x the FP64 rate on this GPU).  The FP64 input X is
// left intact; the elimination works on a float-pair copy.  At the end the
// kernel measures kappa_inf = ||X||_inf ||X^-1||_inf of the result; a matrix
// above `kappa_max` (near a nodal surface of Psi, where the Slater matrix
// becomes singular) or with a non-finite result is flagged, and the caller
// recomputes the flagged matrices with the FP64 k_gj, which skips the others.
// (float-float helpers: ff_math.cuh)

// The panel holds one row per thread in registers (two where n > 512): a column step is
// two barriers, an integer REDUX search for the pivot, the pivot row scaled by its owner's warp,
// and NB float-float multiply-adds per row into registers rotated by one, so that the step's
// column is always the first and the loop needs no unrolling.  The trailing update pairs two rows
// (packed FP32 instructions: two results per issue slot, the same roundings), the eliminated
// panel lying in shared memory as row pairs {h, h', l, l'}.  Bound by the FP32 pipe: n^3 multiply-adds
// of 12 operations.  Measured (16 lanes per row of the panel and scalar updates before): 8192
// matrices of 217 rows 63.4 -> 51.6 ms, 200 of 79 rows 285 -> 207 us, 2 of 79 rows 232 -> 144 us.

// |x| as an integer that orders like it; 0 for NaN (never a pivot) and 0
__device__ __forceinline__ unsigned gjff_key(float x)
{
    const unsigned b = __float_as_uint(x) & 0x7fffffffu;
    return b > 0x7f800000u ? 0u : b;
}

// The largest key of a warp and the smallest index that has it, in every lane.
__device__ __forceinline__ void gjff_warp_max(unsigned &k, int &i)
{
    const unsigned m = __reduce_max_sync(0xffffffffu, k);
    i = (int)__reduce_min_sync(0xffffffffu, k == m ? (unsigned)i : 0x7fffffffu);
    k = m;
}

__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// (xh, xl) += (ph, pl) (uh, ul) for two rows: the product's error by FMA, TwoSum into the high
// parts, the low parts plain
__device__ __forceinline__ void gjff_step2(float2 &xh, float2 &xl, float2 ph, float2 pl, float2 uh, float2 ul)
{
    const float2 p = __fmul2_rn(ph, uh);
    float2 pe = __ffma2_rn(ph, uh, neg2(p));
    pe = __ffma2_rn(ph, ul, pe);
    pe = __ffma2_rn(pl, uh, pe);
    const float2 s = __fadd2_rn(xh, p), bb = __fadd2_rn(s, neg2(xh));
    const float2 e = __fadd2_rn(__fadd2_rn(xh, neg2(__fadd2_rn(s, neg2(bb)))), __fadd2_rn(p, neg2(bb)));
    xh = s;
    xl = __fadd2_rn(xl, __fadd2_rn(pe, e));
}

// MIN: CTAs per SM that the registers leave room for; kSmem: the work matrix lies in shared memory.
template <int NB, int THREADS, int RPT, int MIN, bool kSmem>
__global__ void __launch_bounds__(THREADS, MIN) k_gj_ff(GjJobs2 jobs, double kappa_max)
{
    constexpr int WARPS = THREADS / 32;
    const GjJob &J = jobs.j[blockIdx.y];
    const int m = blockIdx.x;
    if (m >= J.count) return;
    const int n = J.n;
    const double *__restrict__ X = J.X + (size_t)m * J.x_stride;
    double *__restrict__ Dout = J.Dinv + (size_t)m * J.d_stride;

    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *Wk;                                               // the float-pair work matrix, row stride ld
    const int ld = kSmem ? n | 1 : n;                         // (odd: a thread per row meets all banks)
    if constexpr (kSmem) Wk = reinterpret_cast<float2 *>(smem_raw + gjff_fixed_bytes(n, NB));
    else Wk = J.work + (size_t)m * J.x_stride;
    const int np = (n + 1) >> 1;                              // row pairs
    float4 *P = reinterpret_cast<float4 *>(smem_raw);         // [np][NB]
    float2 *U = reinterpret_cast<float2 *>(smem_raw + gjff_p_bytes(n, NB));   // [NB][32]
    short *pp = reinterpret_cast<short *>(U + NB * 32);
    short *rowc = pp + n;                                     // [2 np] 1 where the row is a pivot of the panel
    __shared__ unsigned red_k[WARPS];
    __shared__ int red_i[WARPS];
    __shared__ float red_f[WARPS];
    __shared__ float2 raw_s[NB], prow_s[NB];
    __shared__ float s_xnorm;

    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    // float-pair copy of X and ||X||_inf (max row sum of |x|, one warp per row)
    float rmax = 0.f;
    for (int i = wid; i < n; i += WARPS) {
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
    for (int i = t; i < 2 * np; i += THREADS) rowc[i] = 0;
    __syncthreads();
    if (t == 0) {
        float xm = 0.f;
        for (int q = 0; q < WARPS; ++q) xm = fmaxf(xm, red_f[q]);
        s_xnorm = xm;
    }
    // |det| = (mag_h + mag_l) 2^mag_e, kept by the last warp (the one with the fewest rows); the sign
    // from the parity of negative pivots
    float mag_h = 1.f, mag_l = 0.f;
    int mag_e = 0, neg = 0;
    bool sing = false;
    bool used[RPT];                                           // this thread's rows t + THREADS r
#pragma unroll
    for (int r = 0; r < RPT; ++r) used[r] = t + THREADS * r >= n;
    __syncthreads();

    for (int jb = 0; jb < n; jb += NB) {
        const int w = min(NB, n - jb);
        float2 x[RPT][NB];
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            const int i = t + THREADS * r;
            const float2 *src = Wk + (size_t)min(i, n - 1) * ld + jb;
#pragma unroll
            for (int q = 0; q < NB; ++q) x[r][q] = (i < n && q < w) ? src[q] : make_float2(0.f, 0.f);
        }
        {
            unsigned k = 0;
            int bi = n;
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                const unsigned kr = used[r] ? 0u : gjff_key(x[r][0].x);
                if (kr > k) { k = kr; bi = t + THREADS * r; }
            }
            gjff_warp_max(k, bi);
            if (lane == 0) { red_k[wid] = k; red_i[wid] = bi; }
        }
        __syncthreads();
        for (int c = 0; c < w; ++c) {
            unsigned k = lane < WARPS ? red_k[lane] : 0u;
            int p = lane < WARPS ? red_i[lane] : n;
            gjff_warp_max(k, p);
            if (k == 0u) { sing = true; break; }              // every warp sees the same candidates
            if (wid == (p & (THREADS - 1)) >> 5) {
                // the pivot row, from its owner through shared memory, scaled a column per lane
#pragma unroll
                for (int r = 0; r < RPT; ++r)
                    if (t + THREADS * r == p) {
#pragma unroll
                        for (int q = 0; q < NB; ++q) raw_s[q] = x[r][q];
                        used[r] = true;
                    }
                __syncwarp();
                const float2 pinv = ff::inv(raw_s[0]);
                if (lane < NB) prow_s[lane] = lane ? ff::mul(raw_s[lane], pinv) : pinv;
            }
            __syncthreads();
            if (wid == WARPS - 1) {
                const float2 piv = raw_s[0];
                const float2 a = piv.x < 0.f ? ff::neg(piv) : piv;
                const float2 mg = ff::mul(make_float2(mag_h, mag_l), a);
                int ex;
                frexpf(mg.x, &ex);
                mag_h = ldexpf(mg.x, -ex);
                mag_l = ldexpf(mg.y, -ex);
                mag_e += ex;
                neg ^= piv.x < 0.f;
                if (lane == 0) {
                    pp[jb + c] = (short)p;
                    rowc[p] = 1;
                }
            }
            const float2 pinv = prow_s[0];
            k = 0;
            int bi = n;
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                const int i = t + THREADS * r;
                if (i - lane >= n) break;                     // a warp without rows
                if (i == p) {
#pragma unroll
                    for (int q = 0; q + 1 < NB; ++q) x[r][q] = prow_s[q + 1];
                    x[r][NB - 1] = pinv;
                } else {
                    const float2 mf = ff::neg(x[r][0]);
#pragma unroll
                    for (int q = 0; q + 1 < NB; ++q) x[r][q] = ff::fma2(x[r][q + 1], mf, prow_s[q + 1]);
                    x[r][NB - 1] = ff::mul(mf, pinv);
                }
                const unsigned kr = (used[r] || c + 1 >= w) ? 0u : gjff_key(x[r][0].x);
                if (kr > k) { k = kr; bi = i; }
            }
            gjff_warp_max(k, bi);
            if (lane == 0) { red_k[wid] = k; red_i[wid] = bi; }
            __syncthreads();
        }
        if (sing) break;

        // the eliminated panel: part of the result, and the update's operand as row pairs (the registers
        // are w steps round: all the way, but in a short last panel)
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            const int i = t + THREADS * r;
            float *dst = reinterpret_cast<float *>(P + (size_t)(i >> 1) * NB) + (i & 1);
            if (i < n) {
#pragma unroll
                for (int q = 0; q < NB; ++q) {
                    const int col = (q + w) & (NB - 1);
                    if (col < w) Wk[(size_t)i * ld + jb + col] = x[r][q];
                    dst[4 * col] = x[r][q].x;
                    dst[4 * col + 2] = x[r][q].y;
                }
            } else if (i < 2 * np) {
#pragma unroll
                for (int q = 0; q < NB; ++q) dst[4 * q] = dst[4 * q + 2] = 0.f;
            }
        }

        int c0 = 0;
        auto skip = [&](int cc0) { return cc0 >= jb && cc0 + 32 <= jb + w; };
        while (c0 < n && skip(c0)) c0 += 32;
        constexpr int UPT = NB * 32 / THREADS > 0 ? NB * 32 / THREADS : 1;
        float2 upre[UPT];
        __syncthreads();
        auto load_u = [&](int cc0) {
#pragma unroll
            for (int r = 0; r < UPT; ++r) {
                const int q = t + r * THREADS, c = q >> 5, col = cc0 + (q & 31);
                upre[r] = (cc0 < n && c < w && col < n) ? Wk[(size_t)pp[jb + c] * ld + col] : make_float2(0.f, 0.f);
            }
        };
        load_u(c0);
        while (c0 < n) {
            __syncthreads();
#pragma unroll
            for (int r = 0; r < UPT; ++r)
                if (t + r * THREADS < NB * 32) U[t + r * THREADS] = upre[r];
            __syncthreads();
            int c1 = c0 + 32;
            while (c1 < n && skip(c1)) c1 += 32;
            load_u(c1);
            const int col = c0 + lane;
            const bool active = col < n && !(col >= jb && col < jb + w);
            float2 u[NB];
#pragma unroll
            for (int c = 0; c < NB; ++c) u[c] = U[c * 32 + lane];
            if (active) {
                auto load_pair = [&](int r, float2 &h, float2 &l) {      // rows 2 r, 2 r + 1 (0 for pivots)
                    const int i = 2 * r;
                    const float2 a = (r < np && !rowc[i]) ? Wk[(size_t)i * ld + col] : make_float2(0.f, 0.f);
                    const float2 b = (i + 1 < n && !rowc[i + 1]) ? Wk[(size_t)(i + 1) * ld + col] : make_float2(0.f, 0.f);
                    h = make_float2(a.x, b.x);
                    l = make_float2(a.y, b.y);
                };
                auto store_pair = [&](int r, float2 h, float2 l) {
                    float sh, sl;
                    ff::fast_two_sum(h.x, l.x, sh, sl);
                    Wk[(size_t)(2 * r) * ld + col] = make_float2(sh, sl);
                    if (2 * r + 1 < n) {
                        ff::fast_two_sum(h.y, l.y, sh, sl);
                        Wk[(size_t)(2 * r + 1) * ld + col] = make_float2(sh, sl);
                    }
                };
                // two row pairs at a time, the next two loaded meanwhile
                float2 nh0, nl0, nh1, nl1;
                load_pair(wid, nh0, nl0);
                load_pair(wid + WARPS, nh1, nl1);
                for (int r = wid; r < np; r += 2 * WARPS) {
                    const int r1 = r + WARPS;
                    float2 xh0 = nh0, xl0 = nl0, xh1 = nh1, xl1 = nl1;
                    load_pair(r + 2 * WARPS, nh0, nl0);
                    load_pair(r1 + 2 * WARPS, nh1, nl1);
                    const float4 *p0 = P + (size_t)r * NB, *p1 = P + (size_t)(r1 < np ? r1 : r) * NB;
#pragma unroll
                    for (int c = 0; c < NB; ++c) {
                        const float4 a0 = p0[c], a1 = p1[c];
                        const float2 uh = make_float2(u[c].x, u[c].x), ul = make_float2(u[c].y, u[c].y);
                        gjff_step2(xh0, xl0, make_float2(a0.x, a0.y), make_float2(a0.z, a0.w), uh, ul);
                        gjff_step2(xh1, xl1, make_float2(a1.x, a1.y), make_float2(a1.z, a1.w), uh, ul);
                    }
                    store_pair(r, xh0, xl0);
                    if (r1 < np) store_pair(r1, xh1, xl1);
                }
            }
            c0 = c1;
        }
        __syncthreads();
        for (int c = t; c < w; c += THREADS) rowc[pp[jb + c]] = 0;
        __syncthreads();
    }

    if (sing) {
        // a zero pivot in the float pairs: the FP64 kernel decides whether X is singular
        if (t == 0 && J.redo) J.redo[m * J.redo_stride] = 1;
        return;
    }
    __syncthreads();

    // ||X^-1||_inf (the rows of X^-1 are the rows of the result, columns permuted) and D^-1 = X^-T
    // in one pass, 32 x 32 tiles alternating between two buffers: one barrier each
    constexpr int RW = 32 / WARPS;
    float2 *tile = reinterpret_cast<float2 *>(smem_raw);      // [2][32][33] (P and U are done with)
    float imax = 0.f;
    int buf = 0;
    for (int kb = 0; kb < n; kb += 32) {
        float rs[RW];
        const float2 *row[RW];
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            const int k = kb + wid + r * WARPS;
            rs[r] = 0.f;
            row[r] = k < n ? Wk + (size_t)pp[k] * ld : nullptr;
        }
        for (int cb = 0; cb < n; cb += 32, buf ^= 32 * 33) {
            const int c = cb + lane;
            float2 v[RW];
#pragma unroll
            for (int r = 0; r < RW; ++r) v[r] = (row[r] && c < n) ? row[r][c] : make_float2(0.f, 0.f);
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                tile[buf + (wid + r * WARPS) * 33 + lane] = v[r];
                if (c < n) rs[r] += fabsf(v[r].x);
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                const int cr = cb + wid + r * WARPS, k = kb + lane;
                if (cr < n && k < n) Dout[(size_t)pp[cr] * n + k] = join_f64(tile[buf + lane * 33 + wid + r * WARPS]);
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

    // parity of the row permutation k -> pp[k]: its inversions
    int inv = 0;
    for (int i = t; i < n; i += THREADS)
        for (int j = i + 1; j < n; ++j) inv ^= pp[j] < pp[i];
    const int par = __syncthreads_count(inv) & 1;
    if (t == THREADS - 32) {
        float im = 0.f;
        for (int q = 0; q < WARPS; ++q) im = fmaxf(im, red_f[q]);
        const double kappa = (double)s_xnorm * (double)im;
        const double logabs = log((double)mag_h + (double)mag_l) + mag_e * 0.69314718055994530942;
        if (J.logabs) J.logabs[(size_t)m * J.la_stride] = logabs;
        if (J.sign) J.sign[(size_t)m * J.la_stride] = (par ^ neg) ? -1.0 : 1.0;
        if (J.redo && !(kappa <= kappa_max && isfinite(logabs))) J.redo[m * J.redo_stride] = 1;
    }
}

template <int NB, int THREADS, int RPT, int MIN, bool kSmem>
static cudaError_t launch_gj_ff_k(const GjJobs2 &js, int n_jobs, int nmax, int cmax, double kappa_max,
                                  cudaStream_t st)
{
    const size_t sm = gjff_fixed_bytes(nmax, NB) + (kSmem ? sizeof(float2) * nmax * (size_t)(nmax | 1) : 0);
    constexpr auto kern = k_gj_ff<NB, THREADS, RPT, MIN, kSmem>;
    cudaError_t e = allow_smem<kern>(sm);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    dim3 grid(cmax, n_jobs);
    kern<<<grid, THREADS, sm, st>>>(js, kappa_max);
    return cudaGetLastError();
}

// One row per thread while the rows fit a block of 64, 256 or 512, else two.  Blocks of 64 where there are
// more small matrices than two blocks of 256 on each of 152 SMs hold: a block of 256 has few threads with a row
// there, and registers for two blocks (the elimination's stage, 40000 matrices, ms: 5 rows 1.49 -> 0.55, 32 rows
// 5.55 -> 2.83; 4000 of 64 rows 1.64 -> 1.37).  Blocks of 256: the work
// matrix in shared memory where that leaves room for the matrices' CTAs (three on each of 152 SMs,
// or as many as there are: 2 matrices of 79 rows 164 -> 152 us); else with registers for two CTAs
// per SM where two hold every matrix, for three beyond (8192 matrices of 217 rows: 54.5 -> 52.0 ms;
// 2 of 79 rows: 164 -> 177 us).
template <int NB>
static cudaError_t launch_gj_ff_nb(const GjJobs2 &js, int n_jobs, int nmax, int cmax, double kappa_max,
                                   cudaStream_t st)
{
    constexpr int M2 = NB <= 16 ? 2 : 1, M3 = NB <= 16 ? 3 : 1;
    const long long T = (long long)cmax * n_jobs;
    if (nmax <= 64 && T > 304)
        return launch_gj_ff_k<NB, 64, 1, NB <= 16 ? 8 : 4, true>(js, n_jobs, nmax, cmax, kappa_max, st);
    if (nmax <= 256) {
        const size_t sm = gjff_fixed_bytes(nmax, NB) + sizeof(float2) * nmax * (size_t)(nmax | 1);
        if (sm <= 72 * 1024 || (T <= 304 && sm <= 108 * 1024) || (T <= 152 && sm <= 220 * 1024))
            return launch_gj_ff_k<NB, 256, 1, M2, true>(js, n_jobs, nmax, cmax, kappa_max, st);
        if (T <= 304) return launch_gj_ff_k<NB, 256, 1, M2, false>(js, n_jobs, nmax, cmax, kappa_max, st);
        return launch_gj_ff_k<NB, 256, 1, M3, false>(js, n_jobs, nmax, cmax, kappa_max, st);
    }
    if (nmax <= 512) return launch_gj_ff_k<NB, 512, 1, 1, false>(js, n_jobs, nmax, cmax, kappa_max, st);
    return launch_gj_ff_k<NB, 512, 2, 1, false>(js, n_jobs, nmax, cmax, kappa_max, st);
}

cudaError_t launch_gj_ff(const GjJob *jobs, int n_jobs, cudaStream_t st, int nb, double kappa_max)
{
    GjJobs2 js;
    int nmax = 0, cmax = 0;
    for (int q = 0; q < 2; ++q) {
        js.j[q] = jobs[q < n_jobs ? q : 0];
        if (q >= n_jobs) js.j[q].count = 0;
        nmax = max(nmax, js.j[q].n);
        cmax = max(cmax, js.j[q].count);
    }
    if (cmax == 0) return cudaSuccess;
    switch (nb) {
    case 8: return launch_gj_ff_nb<8>(js, n_jobs, nmax, cmax, kappa_max, st);
    case 16: return launch_gj_ff_nb<16>(js, n_jobs, nmax, cmax, kappa_max, st);
    case 32: return launch_gj_ff_nb<32>(js, n_jobs, nmax, cmax, kappa_max, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace qmc
