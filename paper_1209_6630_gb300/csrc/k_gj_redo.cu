// Step a4, mixed path: FP64 recomputation of the matrices that the
// float-float Gauss-Jordan pass flagged (near a nodal surface of Psi, where
// the Slater matrix approaches singularity; Sec. IV.B keeps the inversion in
// double precision).
//
// A 528 x 528 FP64 elimination on one SM is bound by that SM's FP64 pipe
// (~35 ms), so a single flagged matrix would dominate the stage.  Here each
// matrix is spread over many CTAs: for every panel of NB columns one
// CTA eliminates the panel (partial pivoting among rows not yet used; the
// same arithmetic, order and panel width as k_gj, so the results are
// identical) and then one CTA per block of 32, 8 or 4 columns applies the
// rank-NB update to its columns,
//   X[i][j] <- [i not a pivot of the panel] X[i][j] + sum_c P[i][c] X[piv_c][j],
// two launches per panel.  A list kernel collects the flagged matrices (up to
// kRedoMax) in a deterministic order and marks them handled (flag 2); flagged
// matrices beyond the list keep flag 1 and go through k_gj.  The update's CTAs
// walk over the (matrix, column block) items of the list, with blocks narrow
// enough to give every SM an item; with nothing flagged every CTA exits at once.
//
// launch_gj_wide runs the same kernels over all matrices of a call too few to
// fill the card with one CTA each (every SM's FP64 pipe is then in use); the
// matrices' state sits in their own D^-1 arrays until the end (from two rows on: one row has not the room).
// (Rule and times: gj_wide in k_gj.cu.)
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "c1_f64.cuh"
#include "gj_panel.cuh"
#include "qmc_device.cuh"

namespace qmc {

namespace cg = cooperative_groups;

constexpr int kRThreads = 256;
constexpr int kRWarps = kRThreads / 32;

struct RedoEntry {
    int job, m;
};

struct RedoList {
    int count;
    RedoEntry e[kRedoMax];
};

// per listed matrix: logabs, negative-pivot parity, singular flag, pivot rows
// pp[n] and the panel in which each row became a pivot (-1: not yet)
struct RedoState {
    double logabs;
    int neg, sing;
};
static_assert(sizeof(RedoState) == 16, "gj_state_bytes");

struct RedoArgs {
    GjJob j[2];
    RedoList *list;        // null: every matrix of both jobs, in order
    int n_all;             // their number
    char *state;           // kRedoMax entries of state_stride bytes
    size_t state_stride;
    int nmax;
    int e_off[2];          // first electron of each job's spin
};

__device__ __forceinline__ int rcount(const RedoArgs &a) { return a.list ? a.list->count : a.n_all; }
__device__ __forceinline__ RedoEntry rentry(const RedoArgs &a, int b)
{
    if (a.list) return a.list->e[b];
    RedoEntry en;
    en.job = b >= a.j[0].count;
    en.m = en.job ? b - a.j[0].count : b;
    return en;
}
__device__ __forceinline__ RedoState *rstate(const RedoArgs &a, int b, const RedoEntry &en)
{
    return reinterpret_cast<RedoState *>(a.list ? (void *)(a.state + (size_t)b * a.state_stride)
                                                : (void *)(a.j[en.job].Dinv + (size_t)en.m * a.j[en.job].d_stride));
}
__device__ __forceinline__ short *rpp(RedoState *st) { return reinterpret_cast<short *>(st + 1); }
__device__ __forceinline__ short *rpanel(RedoState *st, int n) { return rpp(st) + n; }

size_t redo_scratch_bytes(int nmax)
{
    const size_t stride = (gj_state_bytes(nmax) + 255) & ~size_t(255);
    return ((sizeof(RedoList) + 255) & ~size_t(255)) + kRedoMax * stride;
}

// Collect flagged matrices (flag 1) of both jobs, job 0 first, in index order.
__global__ void __launch_bounds__(1024) k_redo_list(RedoArgs a, int n_jobs)
{
    __shared__ int warp_s[32];
    __shared__ int s_base;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    if (t == 0) s_base = 0;
    __syncthreads();
    for (int job = 0; job < n_jobs; ++job) {
        const GjJob &J = a.j[job];
        for (int m0 = 0; m0 < J.count; m0 += 1024) {
            const int m = m0 + t;
            const int f = (m < J.count && J.redo[(size_t)m * J.redo_stride] == 1) ? 1 : 0;
            int x = f;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) warp_s[wid] = x;
            __syncthreads();
            int before = 0, total = 0;
            for (int q = 0; q < 32; ++q) {
                if (q < wid) before += warp_s[q];
                total += warp_s[q];
            }
            const int pos = s_base + before + x - f;
            if (f && pos < kRedoMax) {
                a.list->e[pos].job = job;
                a.list->e[pos].m = m;
                J.redo[(size_t)m * J.redo_stride] = 2;
            }
            __syncthreads();
            if (t == 0) s_base += total;
            __syncthreads();
        }
    }
    if (t == 0) a.list->count = min(s_base, kRedoMax);
}

// Eliminate panel [jb, jb + w) of every matrix (one CTA each).
template <int kRNB, int kT>                                       // kT: the most threads
__global__ void __launch_bounds__(kT) k_redo_panel(RedoArgs a, int jb)
{
    const int b = blockIdx.x;
    if (b >= rcount(a)) return;
    const RedoEntry en = rentry(a, b);
    const GjJob &J = a.j[en.job];
    const int n = J.n;
    if (jb >= n) return;
    RedoState *stt = rstate(a, b, en);
    short *pp = rpp(stt), *panel = rpanel(stt, n);
    double *__restrict__ X = J.X + (size_t)en.m * J.x_stride;
    const int nthr = kT == kRThreads ? kRThreads : blockDim.x, t = threadIdx.x, lane = t & 31, wid = t >> 5;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *P = reinterpret_cast<double *>(smem_raw);             // [n][kRNB]
    short *used = reinterpret_cast<short *>(P + (size_t)n * kRNB);  // [n]
    __shared__ GjPanelShared<kRNB> S;

    if (jb == 0) {
        for (int i = t; i < n; i += nthr) panel[i] = -1;
        if (t == 0) { stt->logabs = 0.0; stt->neg = 0; stt->sing = 0; }
        __syncthreads();
    }
    if (stt->sing) return;
    const int w = min(kRNB, n - jb);
    for (int i = t; i < n; i += nthr) used[i] = panel[i] >= 0;
    for (int q = t; q < n * kRNB; q += nthr) {
        const int i = q / kRNB, c = q - i * kRNB;
        P[gj_at<kRNB>(i, c)] = (c < w) ? X[(size_t)i * n + jb + c] : 0.0;
    }
    __syncthreads();
    const bool ok = gj_panel<kRNB>(P, n, w, used, S);
    if (wid == 0) {
        double logabs = stt->logabs;
        int neg = stt->neg;
        __syncwarp();
        if (ok) {
            gj_add_pivots<kRNB>(S, w, logabs, neg);
            if (lane < w) {
                pp[jb + lane] = S.pp[lane];
                panel[S.pp[lane]] = (short)jb;
            }
        }
        if (lane == 0) { stt->sing = !ok; stt->logabs = logabs; stt->neg = neg; }
    }
    if (ok)
        for (int q = t; q < n * w; q += nthr) {
            const int i = q / w, c = q - i * w;
            X[(size_t)i * n + jb + c] = P[gj_at<kRNB>(i, c)];
        }
}

// Rank-w update of the matrices' columns outside the panel, in blocks of 32, 8 or 4 columns: the
// widest that give each of 152 SMs two items (a block owns its columns: its pivot rows are read
// before its rows are written).
template <int kRNB>
__global__ void __launch_bounds__(kRThreads) k_redo_update(RedoArgs a, int jb)
{
    const int count = rcount(a);
    int lc = 5;
    if ((long long)count * ((a.nmax + 31) / 32) < 304) lc = (long long)count * ((a.nmax + 7) / 8) < 304 ? 2 : 3;
    const int nblk = (a.nmax + (1 << lc) - 1) >> lc, items = count * nblk;
    const int t = threadIdx.x, cols = 1 << lc;
    const int cl = t & (cols - 1), r0 = t >> lc, rstep = kRThreads >> lc;   // a thread's column and rows
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *P = reinterpret_cast<double *>(smem_raw);   // [n][kRNB]
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        const int b = it / nblk, c0 = (it - b * nblk) << lc;
        const RedoEntry en = rentry(a, b);
        const GjJob &J = a.j[en.job];
        const int n = J.n;
        if (jb >= n || c0 >= n) continue;
        const int w = min(kRNB, n - jb);
        if (c0 >= jb && c0 + cols <= jb + w) continue;    // entirely inside the panel
        RedoState *stt = rstate(a, b, en);
        if (stt->sing) continue;
        const short *pp = rpp(stt), *panel = rpanel(stt, n);
        double *__restrict__ X = J.X + (size_t)en.m * J.x_stride;
        __syncthreads();                                  // the previous item's reads of P
        for (int q = t; q < n * kRNB; q += kRThreads) {
            const int i = q / kRNB, c = q - i * kRNB;
            P[gj_at<kRNB>(i, c)] = (c < w) ? X[(size_t)i * n + jb + c] : 0.0;
        }
        const int col = c0 + cl;
        const bool active = col < n && !(col >= jb && col < jb + w);
        double u[kRNB];
#pragma unroll
        for (int c = 0; c < kRNB; ++c) u[c] = (active && c < w) ? X[(size_t)pp[jb + c] * n + col] : 0.0;
        __syncthreads();                                  // every pivot row has been read
        if (!active) continue;
        int i = r0;
        for (; i + 3 * rstep < n; i += 4 * rstep) {       // four rows: independent chains
            double x[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int ii = i + r * rstep;
                x[r] = (panel[ii] == jb) ? 0.0 : X[(size_t)ii * n + col];
            }
#pragma unroll
            for (int c2 = 0; c2 < kRNB / 2; ++c2)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const double2 pv = *reinterpret_cast<const double2 *>(P + gj_at<kRNB>(i + r * rstep, 2 * c2));
                    x[r] = fma(pv.x, u[2 * c2], x[r]);
                    x[r] = fma(pv.y, u[2 * c2 + 1], x[r]);
                }
#pragma unroll
            for (int r = 0; r < 4; ++r) X[(size_t)(i + r * rstep) * n + col] = x[r];
        }
        for (; i < n; i += rstep) {
            double x = (panel[i] == jb) ? 0.0 : X[(size_t)i * n + col];
#pragma unroll
            for (int c2 = 0; c2 < kRNB / 2; ++c2) {
                const double2 pv = *reinterpret_cast<const double2 *>(P + gj_at<kRNB>(i, 2 * c2));
                x = fma(pv.x, u[2 * c2], x);
                x = fma(pv.y, u[2 * c2 + 1], x);
            }
            X[(size_t)i * n + col] = x;
        }
    }
}

// D^-1, log|det| and sign of every matrix: Dinv[pp[c]][k] = Res[pp[k]][c], one cluster per matrix
// at a time (one CTA took 744 us for n = 528).
constexpr int kFinalCluster = 8;

__global__ void __cluster_dims__(kFinalCluster, 1, 1) __launch_bounds__(kRThreads) k_redo_final(RedoArgs a)
{
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    __shared__ double tile[32 * 33];
    __shared__ short pp[1024];
    const int count = rcount(a);
    for (int b = blockIdx.x / kFinalCluster; b < count; b += gridDim.x / kFinalCluster) {
        const RedoEntry en = rentry(a, b);
        const GjJob &J = a.j[en.job];
        const int n = J.n, m = en.m;
        const double *__restrict__ X = J.X + (size_t)m * J.x_stride;
        double *__restrict__ Dout = J.Dinv + (size_t)m * J.d_stride;
        RedoState *sp = rstate(a, b, en);
        const RedoState st0 = *sp;
        for (int i = t; i < n; i += kRThreads) pp[i] = rpp(sp)[i];
        cluster.sync();                                    // the state may lie in Dout
        if (st0.sing) {
            const double qnan = __longlong_as_double(0x7ff8000000000000ll);
            for (size_t q = (size_t)rank * kRThreads + t; q < (size_t)n * n; q += kFinalCluster * kRThreads) Dout[q] = qnan;
            if (t == 0 && rank == 0) {
                if (J.logabs) J.logabs[(size_t)m * J.la_stride] = -INFINITY;
                if (J.sign) J.sign[(size_t)m * J.la_stride] = 0.0;
                if (J.flag) atomicOr(J.flag + m, J.flag_bit);
            }
            continue;
        }
        const int nt = (n + 31) / 32;
        for (int q = rank; q < nt * nt; q += kFinalCluster) {
            const int kb = q / nt * 32, cb = (q - q / nt * nt) * 32;
            for (int r = wid; r < 32; r += kRWarps) {
                const int k = kb + r, c = cb + lane;
                tile[r * 33 + lane] = (k < n && c < n) ? X[(size_t)pp[k] * n + c] : 0.0;
            }
            __syncthreads();
            for (int r = wid; r < 32; r += kRWarps) {
                const int c = cb + r, k = kb + lane;
                if (c < n && k < n) Dout[(size_t)pp[c] * n + k] = tile[lane * 33 + r];
            }
            __syncthreads();
        }
        if (rank == 0) {
            // parity of the row permutation k -> pp[k]: its inversions
            int inv = 0;
            for (int i = t; i < n; i += kRThreads)
                for (int j = i + 1; j < n; ++j) inv ^= pp[j] < pp[i];
            const int odd = __syncthreads_count(inv) & 1;
            if (t == 0) {
                if (J.logabs) J.logabs[(size_t)m * J.la_stride] = st0.logabs;
                if (J.sign) J.sign[(size_t)m * J.la_stride] = (odd ^ st0.neg) ? -1.0 : 1.0;
            }
        }
        __syncthreads();                                   // pp is rewritten for the next matrix
    }
}

// C1 rows of every listed matrix recomputed in FP64 (exact screening, FP64 AO
// values and products): near a nodal surface the mixed-precision C1 (~2^-40
// normwise) perturbs log|det| by up to kappa times that.  Each CTA computes
// one row (blockIdx.x) of every 32nd listed matrix.
// (c1_f64.cuh: at 434 electrons x 4096 walkers, ~230 listed matrices, 8.5 -> 2.2 ms; before, every AO
// evaluated its own exponentials, a core shell's eight among the others' one to three.)
constexpr int kC1Slots = 32;   // CTAs per row; each loops over the listed matrices

template <int NJ>
__global__ void __launch_bounds__(kCfThreads) k_redo_c1(SysDev s, RedoArgs a, const double *__restrict__ R)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int warp_s[kCfThreads / 32];
    __shared__ double g_s[kCfShells];
    for (int b = blockIdx.y; b < a.list->count; b += kC1Slots) {
        const RedoEntry en = a.list->e[b];
        const GjJob &J = a.j[en.job];
        const int n = J.n, i = blockIdx.x;
        if (i >= n) continue;
        const int e = a.e_off[en.job] + i;
        const double *r = R + ((size_t)en.m * s.n_elec + e) * 3;
        __syncthreads();                                   // the previous row's tables
        c1_row_f64<NJ, true>(s, cf_carve(s, smem_raw), g_s, warp_s, e >= s.n_up, r[0], r[1], r[2],
                             J.X + (size_t)en.m * J.x_stride + (size_t)i * n);
    }
}

template <int NJ>
static cudaError_t launch_redo_c1(const SysDev &s, const RedoArgs &a, int nmax, const double *R, cudaStream_t st)
{
    const size_t sm = c1_smem(s);
    cudaError_t e = allow_smem<k_redo_c1<NJ>>(sm);
    if (e != cudaSuccess) return e;
    k_redo_c1<NJ><<<dim3(nmax, kC1Slots), kCfThreads, sm, st>>>(s, a, R);
    return cudaGetLastError();
}

static cudaError_t launch_redo_c1(const SysDev &s, const RedoArgs &a, int nmax, const double *R, cudaStream_t st)
{
    switch ((nmax + kCfThreads - 1) / kCfThreads) {
    case 1: return launch_redo_c1<1>(s, a, nmax, R, st);
    case 2: return launch_redo_c1<2>(s, a, nmax, R, st);
    case 3: return launch_redo_c1<3>(s, a, nmax, R, st);
    case 4: return launch_redo_c1<4>(s, a, nmax, R, st);
    case 5: return launch_redo_c1<5>(s, a, nmax, R, st);
    case 6: return launch_redo_c1<6>(s, a, nmax, R, st);
    case 7: return launch_redo_c1<7>(s, a, nmax, R, st);
    default: return launch_redo_c1<8>(s, a, nmax, R, st);
    }
}

template <int NB>
static cudaError_t launch_redo_panels(const RedoArgs &a, int nmax, cudaStream_t st)
{
    const size_t smp = sizeof(double) * (size_t)nmax * NB + sizeof(short) * nmax;
    const size_t smu = sizeof(double) * (size_t)nmax * NB;
    cudaError_t e;
    // the panel's steps are a chain of FP64 latencies: a thread per row, within 256 to 1024 (n = 528,
    // 33 panels of a few matrices 2.43 -> 2.00 ms; n = 866, 109 panels 4.12 -> 3.45; 512 threads 2.38 and 3.40)
    const int pthr = NB < 32 ? std::min(1024, std::max(kRThreads, (a.nmax + 127) / 128 * 128)) : kRThreads;
    constexpr auto few = k_redo_panel<NB, kRThreads>, many = k_redo_panel<NB, NB < 32 ? 1024 : kRThreads>;
    const auto panel = pthr > kRThreads ? many : few;
    if ((e = pthr > kRThreads ? allow_smem<many>(smp) : allow_smem<few>(smp)) != cudaSuccess) return e;
    if ((e = allow_smem<k_redo_update<NB>>(smu)) != cudaSuccess) return e;
    // update: two or three CTAs on each of 152 SMs walk over the items
    const unsigned ugrid = a.list ? 456 : (unsigned)std::min<long long>(456 * 8, (long long)a.n_all * ((nmax + 3) / 4));
    for (int jb = 0; jb < nmax; jb += NB) {
        panel<<<a.list ? kRedoMax : a.n_all, pthr, smp, st>>>(a, jb);
        k_redo_update<NB><<<ugrid, kRThreads, smu, st>>>(a, jb);
    }
    return cudaGetLastError();
}

static cudaError_t launch_redo_nb(const RedoArgs &a, int nmax, cudaStream_t st, int nb)
{
    switch (nb) {
    case 8: return launch_redo_panels<8>(a, nmax, st);
    case 16: return launch_redo_panels<16>(a, nmax, st);
    case 32: return launch_redo_panels<32>(a, nmax, st);
    default: return cudaErrorInvalidValue;
    }
}

static int redo_jobs(RedoArgs &a, const GjJob *jobs, int n_jobs)
{
    a.nmax = 0;
    for (int q = 0; q < 2; ++q) {
        a.j[q] = jobs[q < n_jobs ? q : 0];
        if (q >= n_jobs) a.j[q].count = 0;
        if (a.j[q].count > 0) a.nmax = max(a.nmax, a.j[q].n);
    }
    a.n_all = a.j[0].count + a.j[1].count;
    a.e_off[0] = a.e_off[1] = 0;
    a.list = nullptr;
    a.state = nullptr;
    a.state_stride = 0;
    return a.nmax;
}

// Every matrix of the jobs through the kernels above.
cudaError_t launch_gj_wide(const GjJob *jobs, int n_jobs, cudaStream_t st, int nb)
{
    RedoArgs a;
    const int nmax = redo_jobs(a, jobs, n_jobs);
    if (a.n_all == 0) return cudaSuccess;
    for (int q = 0; q < 2; ++q)
        if (a.j[q].count > 0 && gj_state_bytes(a.j[q].n) > sizeof(double) * (size_t)a.j[q].n * a.j[q].n)
            return cudaErrorInvalidValue;
    const cudaError_t e = launch_redo_nb(a, nmax, st, nb);
    if (e != cudaSuccess) return e;
    k_redo_final<<<kFinalCluster * std::min(a.n_all, 1024), kRThreads, 0, st>>>(a);
    return cudaGetLastError();
}

// nb: panel width, the same as the FP64 k_gj of this system (identical results).
// With R given, the listed matrices' C1 is first recomputed in FP64 from the
// walkers' positions (e_off: first electron of each job's spin).
cudaError_t launch_gj_redo(const GjJob *jobs, int n_jobs, void *scratch, cudaStream_t st, int nb, const SysDev *s,
                           const double *R, const int *e_off)
{
    RedoArgs a;
    const int nmax = redo_jobs(a, jobs, n_jobs);
    if (n_jobs == 0 || nmax == 0) return cudaSuccess;
    if (nmax > 1024) return cudaErrorInvalidValue;
    a.list = static_cast<RedoList *>(scratch);
    a.state = static_cast<char *>(scratch) + ((sizeof(RedoList) + 255) & ~size_t(255));
    a.state_stride = (gj_state_bytes(nmax) + 255) & ~size_t(255);
    a.e_off[0] = e_off ? e_off[0] : 0;
    a.e_off[1] = e_off ? e_off[1] : 0;
    k_redo_list<<<1, 1024, 0, st>>>(a, n_jobs);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (R && s) {
        if ((e = launch_redo_c1(*s, a, nmax, R, st)) != cudaSuccess) return e;
    }
    e = launch_redo_nb(a, nmax, st, nb);
    if (e != cudaSuccess) return e;
    k_redo_final<<<kFinalCluster * 38, kRThreads, 0, st>>>(a);   // two CTAs on each of 152 SMs
    return cudaGetLastError();
}

}  // namespace qmc
