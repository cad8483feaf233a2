// Factorisation of the large banded blocks of a grid scene (FEM slabs: 1200 DOF, band 135) and
// of what follows from the factor, when a step refactorises them.
//
// K_i's Cholesky, W = L^-1 [J^T b] and D = W^T W were one warp per block, per 32 columns, and
// per 4 x 4 entries, with every operand read from the global workspace where it was used:
// 150 ms of a 153 ms FP64 step of 16 co-rotational slabs.  Here each operand tile passes
// through shared memory once and is used for a whole register tile:
//   band_chol   a cluster of blocks per matrix.  Panels of NB columns: the diagonal tile by the
//               first block, the rows below it and the trailing update (the rows and columns
//               the panel reaches inside the envelope, at most the band) by all of them, through
//               L2, three cluster barriers a panel.  FP64: an FP64 warp instruction holds its
//               pipe for 64 cycles, so one SM needs 5.5M cycles for a slab's products; eight
//               share them.  FP32: two.
//   band_w      a block per 32 columns: the band's window of solved rows stays in shared memory
//               (a ring), a panel of L rows beside it; the products per panel are a small GEMM
//               and only the NB x NB triangle is a chain.
//   band_d      (FP64) a block per 64 x 64 tile of W^T W, from the first row on where both its
//               row and column ranges of J begin.
// 16 FP64 slabs: factor 2.6 ms, W 2.7 ms, D 4.3 ms (the FP64 pipes' bound for D is 4 ms), the
// co-rotational step 103.6 -> 14.0 ms.  64 FP32 slabs: factor 1.3 ms and W 0.6 ms (the tensor-core
// panels and Schur updates of chol.cu 3.4 ms and the lane-per-column W 2.5 ms, for these
// narrow bands: a Schur update has one to three 128 x 128 tiles a slab with K = 128); that path
// stays for wider envelopes, up to dense blocks, where its products dominate.
#include "band.h"

#include <cooperative_groups.h>

#include <algorithm>

#include "layout.h"

namespace cg = cooperative_groups;

namespace subadmm {
namespace {

template <typename F> struct BandTile;
template <> struct BandTile<float> { static constexpr int NB = 32, CL = 2; };
template <> struct BandTile<double> { static constexpr int NB = 16, CL = 8; };

__device__ __forceinline__ float rsq_of(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsq_of(double x) { return rsqrt(x); }

__device__ __forceinline__ void load4(const float *p, float *v)
{
    const float4 a = *reinterpret_cast<const float4 *>(p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void load4(const double *p, double *v)
{
    const double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

template <typename F>
size_t chol_smem(int bw)
{
    constexpr int NB = BandTile<F>::NB;
    return sizeof(F) * ((size_t)(bw + 1) * (NB + 1) + NB * (NB + 1) + NB);
}

// Right-looking Cholesky of one matrix by a cluster.  Reads of what another block wrote go to
// L2 (the cluster barrier orders them).
template <typename F>
__global__ void __launch_bounds__(kBandThreads) band_chol_kernel(const BandJob *jobs, int *status, int fail_status)
{
    constexpr int NB = BandTile<F>::NB, CL = BandTile<F>::CL, LD = NB + 1;
    constexpr bool FP64 = sizeof(F) == 8;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const BandJob &job = jobs[blockIdx.x / CL];
    volatile int *pend = job.pending;
    const bool go = *pend == 4;
    cl.sync();                                     // every block has read it before one may clear it
    if (!go) return;
    F *const K = static_cast<F *>(job.K), *const LT = static_cast<F *>(job.LT);
    const int n = job.n, tid = threadIdx.x;
    const int *const env = job.env;
    extern __shared__ __align__(16) unsigned char band_smem[];
    F *const T = reinterpret_cast<F *>(band_smem);            // diagonal tile, NB x LD
    F *const inv = T + NB * LD;                               // 1 / L_pp
    F *const Pn = inv + NB;                                   // rows below: (r - r0) x LD
    __shared__ int s_fail;
    auto at = [&](int r, int c) -> F { return c >= env[r] ? __ldcg(K + (size_t)r * n + c) : (F)0; };
    for (int k0 = 0; k0 < n; k0 += NB) {
        const int kn = min(NB, n - k0), r0 = k0 + kn;
        const int nb = job.lastr[r0 - 1] - r0 + 1;            // rows below that the panel reaches
        if (rank == 0) {
            for (int q = tid; q < NB * NB; q += kBandThreads) {
                const int i = q / NB, j = q % NB;
                T[i * LD + j] = i < kn && j <= i ? at(k0 + i, k0 + j) : (F)0;
            }
            if (tid == 0) s_fail = 0;
            __syncthreads();
            for (int k = 0; k < kn; ++k) {
                if (tid < 32) {                               // scale column k
                    const F d = T[k * LD + k];
                    const bool bad = !(d > (F)0) || !isfinite(d);
                    const F q = rsq_of(d);
                    if (tid == 0 && bad) s_fail = 1;
                    __syncwarp();
                    if (k + 1 + tid < kn) T[(k + 1 + tid) * LD + k] *= q;
                    if (tid == 0) { inv[k] = q; T[k * LD + k] = FP64 ? d * q : q; }
                }
                __syncthreads();
                const int w = kn - k - 1;                     // its triangle
                for (int t = tid; t < w * w; t += kBandThreads) {
                    const int i = t / w, j = t - i * w;
                    if (j <= i) T[(k + 1 + i) * LD + k + 1 + j] -= T[(k + 1 + i) * LD + k] * T[(k + 1 + j) * LD + k];
                }
                __syncthreads();
            }
            for (int q = tid; q < kn * NB; q += kBandThreads) {
                const int i = q / NB, j = q % NB, r = k0 + i, c = k0 + j;
                if (j > i || c < env[r]) continue;
                K[(size_t)r * n + c] = T[i * LD + j];
                if (FP64) {
                    LT[(size_t)r * n + c] = i == j ? inv[i] : T[i * LD + j];
                    if (i == j) job.idg[r] = (double)inv[i];
                }
            }
            if (s_fail && tid == 0) {
                *pend = 0;
                if (job.subflag) *job.subflag = 0;
                *status = fail_status;
            }
        }
        cl.sync();
        if (*pend != 4) return;                               // uniform over the cluster
        if (nb <= 0) { cl.sync(); continue; }
        // rows below: L_r = K_r L_kk^-T, a thread per row, in contiguous shares
        if (rank != 0) {
            for (int q = tid; q < NB * NB; q += kBandThreads) {
                const int i = q / NB, j = q % NB;
                T[i * LD + j] = i < kn && j <= i ? at(k0 + i, k0 + j) : (F)0;
            }
            if (tid < kn) inv[tid] = FP64 ? (F)__ldcg(job.idg + k0 + tid) : __ldcg(K + (size_t)(k0 + tid) * n + k0 + tid);
        }
        __syncthreads();
        const int per = (nb + CL - 1) / CL;
        for (int i = tid; i < per; i += kBandThreads) {
            const int r = r0 + rank * per + i;
            if (r >= r0 + nb) break;
            F p[NB];
            const int lo = env[r];
#pragma unroll
            for (int j = 0; j < NB; ++j) p[j] = k0 + j >= lo ? __ldcg(K + (size_t)r * n + k0 + j) : (F)0;
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                p[j] *= inv[j];
#pragma unroll
                for (int t = j + 1; t < NB; ++t) p[t] -= p[j] * T[t * LD + j];
            }
#pragma unroll
            for (int j = 0; j < NB; ++j)
                if (k0 + j >= lo) {
                    K[(size_t)r * n + k0 + j] = p[j];
                    if (FP64) LT[(size_t)r * n + k0 + j] = p[j];
                }
        }
        cl.sync();
        // trailing update: K[r][q] -= L_r . L_q over the triangle, 32 x 32 tiles dealt to the blocks,
        // 2 x 2 entries per thread
        for (int q = tid; q < nb * NB; q += kBandThreads) {
            const int i = q / NB, j = q % NB;
            Pn[i * LD + j] = at(r0 + i, k0 + j);
        }
        __syncthreads();
        const int tb = (nb + 31) / 32;
        for (int t = rank; t < tb * (tb + 1) / 2; t += CL) {
            int bi = 0;
            while ((bi + 1) * (bi + 2) / 2 <= t) ++bi;
            const int bj = t - bi * (bi + 1) / 2;
            const int i0 = 32 * bi + (tid / 16) * 2, j0 = 32 * bj + (tid % 16) * 2;
            F old[2][2], acc[2][2] = {{(F)0, (F)0}, {(F)0, (F)0}};
            bool use[2][2];
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const int r = r0 + i0 + a, c = r0 + j0 + b;
                    use[a][b] = i0 + a < nb && c <= r && c >= env[r];
                    old[a][b] = use[a][b] ? __ldcg(K + (size_t)r * n + c) : (F)0;
                }
            const F *pi = Pn + min(i0, nb - 1) * LD, *pi1 = Pn + min(i0 + 1, nb - 1) * LD;
            const F *pj = Pn + min(j0, nb - 1) * LD, *pj1 = Pn + min(j0 + 1, nb - 1) * LD;
#pragma unroll 8
            for (int k = 0; k < NB; ++k) {
                const F a0 = pi[k], a1 = pi1[k], b0 = pj[k], b1 = pj1[k];
                acc[0][0] += a0 * b0; acc[0][1] += a0 * b1;
                acc[1][0] += a1 * b0; acc[1][1] += a1 * b1;
            }
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b)
                    if (use[a][b]) K[(size_t)(r0 + i0 + a) * n + r0 + j0 + b] = old[a][b] - acc[a][b];
        }
        cl.sync();
    }
}

template <typename F>
int w_ring(int bw)                 // rows of the ring: the window and one panel, whole panels
{
    constexpr int NB = BandTile<F>::NB;
    return (bw + NB - 1) / NB * NB + 2 * NB;
}
template <typename F>
size_t w_smem(int bw)
{
    constexpr int NB = BandTile<F>::NB;
    return sizeof(F) * ((size_t)w_ring<F>(bw) * kBandCols + (size_t)NB * (w_ring<F>(bw) + 4) + NB * (kBandCols + 1) + NB);
}

// Columns c0 .. c0 + 31 of W.  Row p of column t < m starts as J[t][p] inside t's span, column m
// as b; rows above the first row that any of the columns starts in are zero.
template <typename F>
__global__ void __launch_bounds__(kBandThreads) band_w_kernel(const BandJob *jobs, const int2 *tasks, int ring)
{
    constexpr int NB = BandTile<F>::NB, RPW = NB / 8;         // rows of a panel per warp
    constexpr bool FP64 = sizeof(F) == 8;
    const int2 task = tasks[blockIdx.x];
    const BandJob &job = jobs[task.x];
    if (*job.pending != 4) return;
    const F *const L = static_cast<const F *>(FP64 ? job.LT : job.K);      // 1 / L_pp on the diagonal
    F *const W = static_cast<F *>(job.W);
    const int n = job.n, m = job.m, ldw = job.ldw, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int *const env = job.env;
    extern __shared__ __align__(16) unsigned char band_smem[];
    const int lds = ring + 4;
    F *const X = reinterpret_cast<F *>(band_smem);            // ring x 32
    F *const Ls = X + (size_t)ring * kBandCols;               // NB x lds
    F *const Ys = Ls + NB * lds;                              // NB x 33
    F *const inv = Ys + NB * (kBandCols + 1);
    const int t = task.y + lane;
    const int lo = t < m ? job.jlo[t] : t == m ? 0 : n, hi = t < m ? job.jhi[t] : t == m ? n : 0;
    int p0 = lo;
#pragma unroll
    for (int o = 16; o; o >>= 1) p0 = min(p0, __shfl_xor_sync(0xffffffffu, p0, o));
    p0 = p0 / NB * NB;
    if (t < ldw)
        for (int p = warp; p < min(p0, n); p += 8) W[(size_t)p * ldw + t] = (F)0;
    for (int k0 = p0; k0 < n; k0 += NB) {
        const int kn = min(NB, n - k0);
        const int E = max(env[k0], p0) & ~3;                  // env is nondecreasing; whole vectors
                                                              // (the rows before it count as zero)
        const int wd = k0 + NB - E;                           // columns E .. k0 + NB - 1
        for (int i = warp; i < NB; i += 8) {
            const int r = k0 + i, er = r < n ? env[r] : n;
            for (int c = lane; c < wd; c += 32) {
                const int q = E + c;
                Ls[i * lds + c] = q >= er && q < r && r < n ? L[(size_t)r * n + q] : (F)0;
            }
            if (lane == 0) inv[i] = r < n ? L[(size_t)r * n + r] : (F)0;
        }
        F acc[RPW];
#pragma unroll
        for (int i = 0; i < RPW; ++i) {
            const int p = k0 + warp * RPW + i;
            acc[i] = p >= lo && p < hi && p < n ? (F)(t == m ? job.b[p] : job.J[(size_t)t * n + p]) : (F)0;
        }
        __syncthreads();
        // acc -= L[panel][E .. k0) X
        {
            const F *lr = Ls + warp * RPW * lds;
            int x = E % ring;
            int c = 0;
            const int end = k0 - E;
            while (c < end) {                                 // (E, k0 and ring: multiples of 4)
                const int run = min(end - c, ring - x);
                const F *xp = X + (size_t)x * kBandCols + lane;
                for (int q = 0; q < run; q += 4) {
                    F xv[4], lv[RPW][4];
#pragma unroll
                    for (int z = 0; z < 4; ++z) xv[z] = xp[(q + z) * kBandCols];
#pragma unroll
                    for (int i = 0; i < RPW; ++i) load4(lr + i * lds + c + q, lv[i]);
#pragma unroll
                    for (int z = 0; z < 4; ++z)
#pragma unroll
                        for (int i = 0; i < RPW; ++i) acc[i] -= lv[i][z] * xv[z];
                }
                c += run;
                x = 0;
            }
        }
#pragma unroll
        for (int i = 0; i < RPW; ++i) Ys[(warp * RPW + i) * (kBandCols + 1) + lane] = acc[i];
        __syncthreads();
        // the panel's triangle: lanes across its rows (FP64: two columns per warp at a time)
        {
            constexpr int CW = 32 / NB, PASS = kBandCols / 8 / CW;     // columns side by side; passes
            const int r = lane % NB, ch = lane / NB;
            F y[PASS];
#pragma unroll
            for (int s = 0; s < PASS; ++s) y[s] = Ys[r * (kBandCols + 1) + warp * 4 + s * CW + ch];
            const F iv = inv[r];
            const F *lr = Ls + r * lds + (k0 - E);
#pragma unroll 4
            for (int k = 0; k < NB; ++k) {
                const F l = lr[k] ;                                   // zero for k >= r
#pragma unroll
                for (int s = 0; s < PASS; ++s) {
                    const F xk = __shfl_sync(0xffffffffu, y[s] * iv, k + ch * NB);
                    if (r > k) y[s] -= l * xk;
                }
            }
            const int x = k0 % ring;                                  // (whole panels: no wrap)
#pragma unroll
            for (int s = 0; s < PASS; ++s) X[(size_t)(x + r) * kBandCols + warp * 4 + s * CW + ch] = y[s] * iv;
        }
        __syncthreads();
        if (t < ldw)
            for (int i = warp; i < kn; i += 8) W[(size_t)(k0 + i) * ldw + t] = X[(size_t)(k0 % ring + i) * kBandCols + lane];
    }
}

// One 64 x 64 tile (rows 64 ti, columns 64 tj <= ti) of the Gram matrix of W's m + 1 columns into
// D (mirrored), c (row m) and D's zero padding.  4 x 4 entries per thread, 16 rows of W at a time.
__global__ void __launch_bounds__(kBandThreads) band_d_kernel(const BandJob *jobs, const int4 *tasks)
{
    constexpr int TT = 64, KB = 16, LD = TT + 2;
    const int4 task = tasks[blockIdx.x];
    const BandJob &job = jobs[task.x];
    if (*job.pending != 4) return;
    const double *const W = static_cast<const double *>(job.W);
    const int n = job.n, m = job.m, ldw = job.ldw, tid = threadIdx.x;
    const int i0 = task.y * TT, j0 = task.z * TT;
    __shared__ __align__(16) double A[2][KB][LD], B[2][KB][LD];
    const int ty = tid / 16, tx = tid % 16;
    double acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
    double ra[4], rb[4];
    auto fetch = [&](int p) {                      // rows p .. p + 15: 4 entries of each per thread
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = tid + q * kBandThreads, r = p + e / TT, c = e % TT;
            ra[q] = r < n && i0 + c < ldw ? W[(size_t)r * ldw + i0 + c] : 0.0;
            rb[q] = r < n && j0 + c < ldw ? W[(size_t)r * ldw + j0 + c] : 0.0;
        }
    };
    auto put = [&](int s) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = tid + q * kBandThreads;
            A[s][e / TT][e % TT] = ra[q];
            B[s][e / TT][e % TT] = rb[q];
        }
    };
    int s = 0;
    fetch(task.w);
    put(0);
    __syncthreads();
    for (int p = task.w; p < n; p += KB, s ^= 1) {
        if (p + KB < n) fetch(p + KB);
#pragma unroll
        for (int k = 0; k < KB; ++k) {
            double a[4], b[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) { a[q] = A[s][k][ty + 16 * q]; b[q] = B[s][k][tx + 16 * q]; }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[u][v] += a[u] * b[v];
        }
        if (p + KB < n) put(s ^ 1);
        __syncthreads();
    }
    double *const D = static_cast<double *>(job.D), *const cc = static_cast<double *>(job.c);
    const int ldd = job.ldd;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int r = i0 + ty + 16 * u, q = j0 + tx + 16 * v;
            if (q > r || r > m) continue;
            if (r == m) { if (q < m) cc[q] = acc[u][v]; continue; }
            D[(size_t)r * ldd + q] = acc[u][v];
            D[(size_t)q * ldd + r] = acc[u][v];
        }
    if (task.z == 0 && tid < TT && i0 + tid < m)
        for (int q = m; q < job.mpad; ++q) D[(size_t)(i0 + tid) * ldd + q] = 0.0;
}

template <typename F>
cudaError_t run(const BandPlan &P, cudaStream_t st)
{
    const size_t cs = chol_smem<F>(P.bw), ws = w_smem<F>(P.bw);
    cudaError_t e = cudaFuncSetAttribute((const void *)band_chol_kernel<F>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute((const void *)band_w_kernel<F>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(P.njobs * BandTile<F>::CL);
    cfg.blockDim = dim3(kBandThreads);
    cfg.dynamicSmemBytes = cs;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = BandTile<F>::CL;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, band_chol_kernel<F>, (const BandJob *)P.d_jobs, P.status, P.fail_status);
    if (e != cudaSuccess) return e;
    band_w_kernel<F><<<P.nw, kBandThreads, ws, st>>>(P.d_jobs, P.d_w, w_ring<F>(P.bw));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (sizeof(F) == 8 && P.nd > 0) band_d_kernel<<<P.nd, kBandThreads, 0, st>>>(P.d_jobs, P.d_d);
    return cudaGetLastError();
}

}  // namespace

cudaError_t band_plan_build(BandPlan &P, const std::vector<BandJob> &jobs,
                            const std::vector<std::vector<int>> &jlo, int bw, bool fp64, int *status,
                            int fail_status)
{
    P = BandPlan{};
    P.fp64 = fp64;
    P.njobs = (int)jobs.size();
    P.bw = bw;
    P.status = status;
    P.fail_status = fail_status;
    if (cudaError_t e = cudaGetDevice(&P.device); e != cudaSuccess) return e;
    if (jobs.empty()) return cudaSuccess;
    // tasks, the longest first (a column's work starts at its row of J)
    std::vector<std::pair<int, int2>> w;
    std::vector<std::pair<int, int4>> d;
    for (int j = 0; j < P.njobs; ++j) {
        const int n = jobs[j].n, m = jobs[j].m;
        auto first = [&](int c0, int cols) {
            int lo = n;
            for (int t = c0; t < c0 + cols && t <= m; ++t) lo = std::min(lo, t < m ? jlo[j][t] : 0);
            return lo;
        };
        for (int c = 0; c < jobs[j].ldw; c += kBandCols) w.push_back({n - first(c, kBandCols), make_int2(j, c)});
        for (int ti = 0; fp64 && ti * 64 <= m; ++ti)
            for (int tj = 0; tj <= ti; ++tj) {
                const int p = std::min(n - 1, std::max(first(64 * ti, 64), first(64 * tj, 64)) / 16 * 16);
                d.push_back({n - p, make_int4(j, ti, tj, p)});
            }
    }
    auto longer = [](const auto &a, const auto &b) { return a.first > b.first; };
    std::stable_sort(w.begin(), w.end(), longer);
    std::stable_sort(d.begin(), d.end(), longer);
    std::vector<int2> wt;
    std::vector<int4> dt;
    for (auto &x : w) wt.push_back(x.second);
    for (auto &x : d) dt.push_back(x.second);
    P.nw = (int)wt.size();
    P.nd = (int)dt.size();
    cudaError_t e = cudaMalloc((void **)&P.d_jobs, jobs.size() * sizeof(BandJob));
    if (e == cudaSuccess) e = cudaMalloc((void **)&P.d_w, wt.size() * sizeof(int2));
    if (e == cudaSuccess && P.nd) e = cudaMalloc((void **)&P.d_d, dt.size() * sizeof(int4));
    if (e == cudaSuccess) e = cudaMemcpy(P.d_jobs, jobs.data(), jobs.size() * sizeof(BandJob), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(P.d_w, wt.data(), wt.size() * sizeof(int2), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && P.nd) e = cudaMemcpy(P.d_d, dt.data(), dt.size() * sizeof(int4), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) band_plan_free(P);
    return e;
}

cudaError_t band_plan_run(const BandPlan &P, cudaStream_t st)
{
    if (P.njobs == 0) return cudaSuccess;
    return P.fp64 ? run<double>(P, st) : run<float>(P, st);
}

void band_plan_free(BandPlan &P)
{
    cudaFree(P.d_jobs);
    cudaFree(P.d_w);
    cudaFree(P.d_d);
    P = BandPlan{};
}

}  // namespace subadmm
