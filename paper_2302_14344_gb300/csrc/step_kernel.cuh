// One time step of subsystem-based ADMM (Algorithm 1) for a batch of independent scenes,
// one thread block per scene, with the whole per-step working set in shared memory.
//
// Per step and scene:
//   assemble   A_i, b_i, J_ci, e (rigid model or generic blocks)           (Eq. sdyn, Sec. II-A)
//   beta_i     Tr(A_i)/Tr(J_ci^T J_ci) or rho                               (Sec. III-D)
//   factor     K_i = A_i + beta_i J_ci^T J_ci = L_i L_i^T in FP64          (Algorithm 1, factorise)
//   map        W_i = L_i^-1 J_ci^T, g_i = L_i^-1 b_i,
//              D_i = W_i^T W_i = J_ci K_i^-1 J_ci^T, c_i = W_i^T g_i = J_ci K_i^-1 b_i
//   iterate    x_i = c_i + D_i (beta_i z_i - u_i)                           (Eq. admm-1i, x = J v)
//              y_i = beta_i x_i + u_i                                       (Eq. surrogate)
//              lambda_j by type, beta_i z_ij = y_ij + lambda_j              (Eq. admm-2j)
//              u_i = -lambda (the u-step of Eq. admm-3, simplified by Eq. surrogate)
//   recover    v_i = K_i^-1 (b_i + J_ci^T (beta_i z_i - u_i)) in FP64 for the last v-step
//   update     rigid state from v-hat                                       (Eq. ddyn)
//
// The v-step is evaluated through the per-step affine map x = c + D w instead of two
// triangular solves and two products with J per iteration: it is the same linear map,
// reassociated, so every iteration is a small dense mat-vec whose rows run in parallel.
// The u-step uses u^{l+1} = y^{l+1} - beta z^{l+1} = -lambda^{l+1} (Eq. admm-3 with
// Eq. surrogate), so each row keeps one lambda shared by its sides and w = y + 2 lambda.
//
// T is the iteration type.  T = double: the map and the iterations in FP64.  T = float (the
// mixed form): assembly stays FP64; K and its Cholesky factor are FP32 for well-conditioned
// blocks and FP64 for stiff or high-mass-ratio ones (spread of diag K above 1e3); W, g, D,
// c are formed in FP32 and the iterations run in FP32.  (In a grid scene, the FP32 factor of
// a refactorised block of >= 128 DOF is left to the blocked factorisation with tensor-core
// Schur updates that runs between the grid kernel's launches.)  When the FP32 stop test
// passes, v-hat is recovered in FP64 and the primal residual re-evaluated as
// max |J v-hat - z| in FP64; if that misses the tolerance, c is corrected by the FP64 - FP32
// difference of x at the current iterate (iterative refinement) and the iterations resume.
//
// On GB300 an FP64 warp instruction costs about 64 issue cycles of a sub-partition however
// few lanes are active, so FP64 work is kept out of the loop of the mixed form and the loops
// keep each thread's coefficients and lambda in registers for the whole step.
#pragma once
#include "layout.h"
#include "rigid_model.cuh"
#include "block_solve.cuh"
#include "band_warp.cuh"

namespace subadmm {

__device__ __forceinline__ double nanmax(double a, double b) { return (a != a || a > b) ? a : b; }

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_max(double v)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) v = nanmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// 16-byte vectors of the iteration type and residual bit patterns.  Residuals are
// non-negative, so their IEEE bit patterns order like their values and a NaN (sign bit
// cleared by fabs) orders above +inf: maxima reduce on the integer pipe.
template <typename T> struct VecOf;
template <> struct VecOf<float> { using V = float4; using U = unsigned; static constexpr int N = 4; };
template <> struct VecOf<double> { using V = double2; using U = unsigned long long; static constexpr int N = 2; };

__device__ __forceinline__ float vdot(const float4 a, const float4 b, float acc)
{
    acc = fmaf(a.x, b.x, acc); acc = fmaf(a.y, b.y, acc);
    acc = fmaf(a.z, b.z, acc); acc = fmaf(a.w, b.w, acc);
    return acc;
}
__device__ __forceinline__ double vdot(const double2 a, const double2 b, double acc)
{
    acc = fma(a.x, b.x, acc); acc = fma(a.y, b.y, acc);
    return acc;
}
__device__ __forceinline__ unsigned rbits(float v) { return __float_as_uint(v); }
__device__ __forceinline__ unsigned long long rbits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ unsigned umax(unsigned a, unsigned b) { return a > b ? a : b; }
__device__ __forceinline__ unsigned long long umax(unsigned long long a, unsigned long long b) { return a > b ? a : b; }
__device__ __forceinline__ unsigned warp_umax(unsigned v) { return __reduce_max_sync(0xffffffffu, v); }
__device__ __forceinline__ unsigned long long warp_umax(unsigned long long v)
{
    const unsigned hi = (unsigned)(v >> 32), lo = (unsigned)v;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    return ((unsigned long long)mh << 32) | ml;
}
__device__ __forceinline__ unsigned tol_bits(float, double tol) { return __float_as_uint(__double2float_rd(tol)); }
__device__ __forceinline__ unsigned long long tol_bits(double, double tol) { return rbits(tol); }
__device__ __forceinline__ unsigned inf_bits(float) { return 0x7f800000u; }
__device__ __forceinline__ unsigned long long inf_bits(double) { return 0x7ff0000000000000ull; }
template <typename T> struct VecZero;
template <> struct VecZero<float> { __device__ static float4 get() { return make_float4(0.f, 0.f, 0.f, 0.f); } };
template <> struct VecZero<double> { __device__ static double2 get() { return make_double2(0.0, 0.0); } };
// a > 0 (a NaN counts as positive), on the integer pipe
__device__ __forceinline__ bool above0(float a) { return __float_as_int(a) > 0; }
__device__ __forceinline__ bool above0(double a) { return __double_as_longlong(a) > 0; }
__device__ __forceinline__ float rsq(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsq(double x) { return rsqrt(x); }

}  // namespace subadmm
#include "own_iter.cuh"
namespace subadmm {

// Sum (a) and maxima (b, c) of three per-thread doubles over the block.
__device__ __forceinline__ void block_reduce3(double (*red)[SUBADMM_MAXWARPS], double &a,
                                              double &b, double &c)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    a = warp_sum(a); b = warp_max(b); c = warp_max(c);
    __syncthreads();
    if (lane == 0) { red[0][warp] = a; red[1][warp] = b; red[2][warp] = c; }
    __syncthreads();
    a = 0.0; b = 0.0; c = 0.0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) {
        a += red[0][q]; b = nanmax(b, red[1][q]); c = nanmax(c, red[2][q]);
    }
    __syncthreads();
}

// Phase tracer: thread 0 of a scene's block accumulates clock64 deltas per phase in
// registers and adds them to P.phase once per step (flush), so tracing stays off the
// critical path of the iterations.
struct PhaseClock {
    long long *out;
    long long t;
    long long a[8];
    __device__ __forceinline__ PhaseClock(long long *o) : out(threadIdx.x == 0 ? o : nullptr), t(0)
    {
#pragma unroll
        for (int q = 0; q < 8; ++q) a[q] = 0;
        if (out) t = clock64();
    }
    __device__ __forceinline__ void mark(int phase)
    {
        if (out) {
            const long long n = clock64();
            a[phase] += n - t;
            t = n;
        }
    }
    // attribute the time up to `when` (a clock64 value) to `phase`
    __device__ __forceinline__ void mark_at(int phase, long long when)
    {
        if (out) {
            a[phase] += when - t;
            t = when;
        }
    }
    __device__ __forceinline__ void move(int from, int to, long long cycles)
    {
        a[from] -= cycles;
        a[to] += cycles;
    }
    __device__ __forceinline__ void flush(int iters, int steps = 1)
    {
        if (out) {
            a[PHASE_ITERS] = iters;
            a[PHASE_STEPS] = steps;
#pragma unroll
            for (int q = 0; q < 8; ++q) out[q] += a[q];
        }
    }
};

// shared-memory views of one scene
template <typename T>
struct View {
    double *db;          // double region (shared memory): scene arrays
    T *tb;               // T region (shared memory): scene arrays
    double *sdb;         // per-subsystem double arrays: shared memory, or global for a
    T *stb;              // scene too large to hold them on chip; likewise for T
    T *htb;              // per-subsystem iteration arrays (D, c): shared memory unless the
                         // scene cannot hold even those
    int *row, *sub, *drow, *coff, *wbase, *mlen;   // per side-row tables
    Item *item;
    int *list;
};

template <typename T>
__device__ View<T> scene_view(const StepParams &P, const SceneDesc &S, unsigned char *raw)
{
    View<T> V;
    V.db = reinterpret_cast<double *>(raw);
    V.tb = reinterpret_cast<T *>(raw + S.t_base);
    if (S.sub_global) {
        unsigned char *w = reinterpret_cast<unsigned char *>(P.work) + S.g_base;
        V.sdb = reinterpret_cast<double *>(w);
        V.stb = reinterpret_cast<T *>(w + S.g_tbase);
    } else {
        V.sdb = V.db;
        V.stb = V.tb;
    }
    V.htb = S.hot_global ? V.stb : V.tb;
    int *ib = reinterpret_cast<int *>(raw + S.i_base);
    V.row = ib;
    V.sub = ib + S.nsr;
    V.drow = ib + 2 * S.nsr;
    V.coff = ib + 3 * S.nsr;
    V.wbase = ib + 4 * S.nsr;
    V.mlen = ib + 5 * S.nsr;
    V.item = reinterpret_cast<Item *>(ib + 6 * S.nsr);
    V.list = ib + 6 * S.nsr + 4 * S.nitem;
    return V;
}

// D row of a side-row: in the iteration arrays, or (complemented offset) the scene's copy in
// shared memory
template <typename T>
__device__ __forceinline__ const typename VecOf<T>::V *d_row(const View<T> &V, int t)
{
    const int o = V.drow[t];
    return reinterpret_cast<const typename VecOf<T>::V *>(o < 0 ? V.tb + ~o : V.htb + o);
}

// Work distribution of one scene's step: the threads of a block (block kernel: one block
// per scene) or of the whole grid (grid kernel: one scene over every SM).  Loops over
// subsystems take a warp each, loops over rows and constraints a thread each; sync() is a
// barrier over all of them.
struct BlockDist {
    // a scene's own block: its per-warp loops take the subsystems largest first, and the
    // chunks of W wait on per-subsystem flags instead of a barrier after the factor loop (a
    // scene over the whole grid has far more warps than subsystems, and its pollers would
    // load the L2 that its factorisations run through)
    static constexpr bool kSpread = true, kBig = false;
    static constexpr int kThreads = SUBADMM_THREADS;
    int tid, nthreads, warp, nwarps;
    __device__ __forceinline__ BlockDist()
        : tid(threadIdx.x), nthreads(blockDim.x), warp(threadIdx.x >> 5), nwarps(blockDim.x >> 5) {}
    __device__ __forceinline__ void sync() const { __syncthreads(); }
    __device__ __forceinline__ void fence() const { __threadfence_block(); }
};

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Barrier over the `expected` blocks of a cooperative launch.  Thread 0 of each block adds
// one to a counter that only grows (zeroed before the launch); the barrier of round r is
// complete when the counter reaches (r + 1) expected, which each block reads off its own
// arrival (arrivals of round r fall in [r expected, (r + 1) expected)).  The waiters poll
// the counter itself, so the last arrival completes the barrier with its one atomic.  A
// wait longer than limit_ns, or an error raised by another block, sets / sees the error
// flag and returns at once, here and at every later barrier, so the grid always runs to its
// end.  (`gen` is unused: kept for the scratch layout.)
static __device__ __noinline__ void grid_barrier(unsigned *count, unsigned *gen, int *err,
                                          unsigned expected, unsigned long long limit_ns)
{
    (void)gen;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned *vcount = count;
        volatile int *verr = err;
        if (!*verr) {
            __threadfence();
            const unsigned my = atomicAdd(count, 1u);
            const unsigned target = (my / expected + 1u) * expected;
            if ((int)(*vcount - target) < 0) {
                const unsigned long long t0 = global_ns();
                while ((int)(*vcount - target) < 0) {
                    if (*verr) break;
                    if (global_ns() - t0 > limit_ns) { atomicExch(err, 1); break; }
                    __nanosleep(32);
                }
            }
            __threadfence();
        }
    }
    __syncthreads();
}

// Warps are numbered block-interleaved (warp k of block b is k * blocks + b): per-subsystem
// work (one warp each, FP64-bound in the setup and the recovery) then spreads over one warp
// per block, i.e. over the SMs and their FP64 pipes, instead of filling the first blocks.
struct GridDist {
    static constexpr bool kSpread = false, kBig = false;
    static constexpr int kThreads = SUBADMM_THREADS;
    int tid, nthreads, warp, nwarps;
    unsigned *count, *gen;
    int *err;
    __device__ __forceinline__ GridDist(unsigned *c, unsigned *g, int *e)
        : tid(blockIdx.x * blockDim.x + threadIdx.x), nthreads(gridDim.x * blockDim.x),
          warp((int)(threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x),
          nwarps((gridDim.x * blockDim.x) >> 5), count(c), gen(g), err(e) {}
    __device__ __forceinline__ void sync() const
    {
        grid_barrier(count, gen, err, gridDim.x, 20000000000ull);
    }
    __device__ __forceinline__ void fence() const { __threadfence(); }
};

template <typename T, typename Dist>
__device__ void scene_tables(const StepParams &P, const SceneDesc &S, const View<T> &V,
                             const Dist &d)
{
    for (int t = d.tid; t < S.nsr; t += d.nthreads) {
        V.row[t] = 0; V.sub[t] = 0; V.drow[t] = 0; V.coff[t] = 0; V.wbase[t] = 0; V.mlen[t] = 0;
    }
    d.sync();
    for (int j = d.tid; j < S.ncon; j += d.nthreads) {
        const ConDesc &c = P.cons[S.con0 + j];
        for (int s = 0; s < c.ns; ++s) {
            const SubDesc &u = P.subs[S.sub0 + c.sub[s]];
            for (int r = 0; r < c.rows; ++r) {
                const int t = c.sr[s] + r;
                const int lr = t - u.sr0;
                V.row[t] = c.row0 + r;
                V.sub[t] = c.sub[s];
                V.drow[t] = u.ot_Dres >= 0 ? ~(u.ot_Dres + lr * u.ldd) : u.ot_D + lr * u.ldd;
                V.coff[t] = u.ot_c + lr;
                V.wbase[t] = u.sr0;
                V.mlen[t] = u.m;
            }
        }
    }
    for (int i = d.tid; i < S.nitem; i += d.nthreads) V.item[i] = P.items[S.item_g0 + i];
    for (int i = d.tid; i < S.nlist; i += d.nthreads) V.list[i] = P.lists[S.list_g0 + i];
}

// k, alpha, mu of a constraint (model kinds derive them from their drive gains)
__device__ __forceinline__ void con_params(const ConDesc &c, const double *pool, double h,
                                           double &k, double &alpha, double &mu)
{
    const double *p = pool + c.par_off;
    k = 0.0; alpha = 0.0; mu = 0.0;
    if (c.src <= SRC_CONTACT) {
        k = p[0]; alpha = p[1]; mu = p[2];
    } else if (c.src == SRC_ANGLE_PD) {
        k = p[18]; alpha = p[19] / p[18] + 0.5 * h;
    } else if (c.src == SRC_PLANE || c.src == SRC_SPHERE) {
        mu = p[22];
    }
}

// index (r, s), s <= r, of entry t of a lower triangle stored row by row
__device__ __forceinline__ void tri_index(int t, int &r, int &s)
{
    r = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while ((r + 1) * (r + 2) / 2 <= t) ++r;
    while (r * (r + 1) / 2 > t) --r;
    s = t - r * (r + 1) / 2;
}

// Profile of a subsystem's K_i and the column spans of its J rows (built by the host from
// the structure of A_i and J_i): env[p] first column of row p inside the envelope, lastr[k]
// last row whose envelope reaches column k, [jlo[t], jhi[t]) the columns of J row t.
struct SubEnv {
    const int *env, *lastr, *jlo, *jhi;
    const int *grp;        // first rows of the row groups (ngrp + 1 entries)
    int ngrp;
};

__device__ __forceinline__ SubEnv sub_env(const StepParams &P, const SubDesc &u)
{
    SubEnv e;
    e.env = P.ipool + u.env_off;
    e.lastr = e.env + u.n;
    e.jlo = e.lastr + u.n;
    e.jhi = e.jlo + u.m;
    e.grp = P.ipool + u.grp_off;
    e.ngrp = u.ngrp;
    return e;
}

// The row groups of a subsystem for one warp, 32 at a time in its lanes' registers: f(r0, r1, lo, w)
// for every group in order (rows r0 .. r1 - 1, columns lo .. lo + w - 1).  The setup's loops over
// groups and rows are chains of short passes; with their tables read as they went, each pass
// waited for two more trips to L2 (the tables of a scene whose arrays fill shared memory do not
// stay in the L1 that is left).
template <typename Fn>
__device__ __forceinline__ void for_groups(const SubEnv &e, Fn f)
{
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (int g0 = 0; g0 < e.ngrp; g0 += 32) {
        const int g = min(g0 + lane, e.ngrp - 1);
        const int r0 = e.grp[g], r1 = e.grp[g + 1], lo = e.jlo[r0], w = e.jhi[r0] - lo;
        const int cnt = min(32, e.ngrp - g0);
        for (int q = 0; q < cnt; ++q)
            f(__shfl_sync(FULL, r0, q), __shfl_sync(FULL, r1, q), __shfl_sync(FULL, lo, q), __shfl_sync(FULL, w, q));
    }
}

// Rows p of a band, 4 at a time: entries lo(p) .. hi(p) of src, converted by conv(p, q, value), into
// dst (row length n); every load of a pass before its stores
template <typename D, typename S, typename Conv>
__device__ __forceinline__ void copy_band(D *dst, const S *src, int n, const int *lo, Conv conv)
{
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (int b = 0; b < n; b += 32) {
        const int el = lo[min(b + lane, n - 1)];
        for (int h = 0; h < 32 && b + h < n; h += 4) {
            int e[4], len = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                e[i] = __shfl_sync(FULL, el, h + i);
                if (b + h + i < n) len = max(len, b + h + i - e[i] + 1);
            }
            for (int c = lane; c < (len + 31) / 32 * 32; c += 32) {
                S v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int p = b + h + i, q = e[i] + c;
                    v[i] = p < n && q <= p ? src[(size_t)p * n + q] : (S)0;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int p = b + h + i, q = e[i] + c;
                    if (p < n && q <= p) dst[(size_t)p * n + q] = conv(p, q, v[i]);
                }
            }
        }
    }
}

// A constant K_i whose factor from an earlier step is still held: in the workspace (it
// outlives the launch) or in shared memory from an earlier step of this launch.  With
// keep_factors 0 every step refactors (the same matrix; results agree to rounding).  A
// changed beta scale refactors too (K_i = A_i + beta_i J^T J changed).  A tc_phase 1 launch (the host issues it only for steps that refactor) refactors every tc
// subsystem.
__device__ __forceinline__ bool factor_kept(const StepParams &P, const SceneDesc &S,
                                            const SubDesc &u, int gsub, int step)
{
    if (P.tc_phase == 1 && u.tc) return false;
    return P.keep_factors && u.cst && (step > 0 || S.sub_global) && (P.subflag[gsub] & 1) &&
           P.beta_scale[gsub] == P.beta_used[gsub];
}

// K += beta J^T J on the lower triangle (row-major n x n), a row group at a time (rows
// with one column span [lo, lo + w)): lanes across the span's triangle entries, each summing
// its products over the group's rows with independent loads, then one update of K per
// entry and group (groups share entries, so they are added in turn)
template <typename F>
__device__ void add_jtj(F *K, int n, const double *J, const SubEnv &e, F beta)
{
    const int lane = threadIdx.x & 31;
    for_groups(e, [&](int r0, int r1, int lo, int w) {
        const double *J0 = J + (size_t)r0 * n + lo;
        for (int k = lane; k < w * (w + 1) / 2; k += 32) {
            int a, b;
            tri_index(k, a, b);
            const F old = K[(lo + a) * n + lo + b];
            F acc = (F)0;
            for (int t = 0; t < r1 - r0; ++t) acc += (F)J0[(size_t)t * n + a] * (F)J0[(size_t)t * n + b];
            K[(lo + a) * n + lo + b] = old + beta * acc;
        }
        __syncwarp();
    });
}

// Right-looking Cholesky inside the envelope, in place on the lower triangle of K (one
// warp).  Column k below the diagonal is scaled, then the triangle k < q <= r <= lastr[k]
// it reaches is updated with the lanes across its entries: a band of width w costs
// w (w + 1) / 64 warp instructions per column rather than w (on GB300 an FP64 warp
// instruction occupies its pipe however few lanes are active).  Every entry receives the
// same updates in the same order (k ascending).  INV_DIAG: the diagonal ends as 1/L_kk
// (the T factor); otherwise as L_kk with 1/L_kk in idg.  False on a non-positive pivot.
// Columns that reach at most 31 rows (narrow bands: rigid chains, spring blocks): the scaled column
// is in the lanes' registers (its entries go round by shuffles), the triangle's indices are
// worked out once, and every entry of a pass is loaded before any is stored (the compiler cannot
// move a load of K above a store to K: a 23-wide column cost nine round trips to L2, some 6k
// cycles, where it now costs one).
template <typename F, bool INV_DIAG>
__device__ bool narrow_cholesky(F *K, int n, const SubEnv &e, double *idg)
{
    constexpr int PASS = 5;                        // 32-entry slots per pass: 3 passes cover w = 30
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    unsigned char ia[3 * PASS + 1], ib[3 * PASS + 1];
#pragma unroll
    for (int s = 0; s < 3 * PASS + 1; ++s) {
        int a, b;
        tri_index(lane + 32 * s, a, b);
        ia[s] = (unsigned char)a;
        ib[s] = (unsigned char)b;
    }
    for (int k = 0; k < n; ++k) {
        const int w = e.lastr[k] - k, tri = w * (w + 1) / 2;
        const F d = K[(size_t)k * n + k];
        F l = lane < w ? K[(size_t)(k + 1 + lane) * n + k] : (F)0;
        if (!(d > (F)0) || !isfinite(d)) return false;
        F *const T0 = K + (size_t)(k + 1) * n + k + 1;
        F c[PASS];
#pragma unroll
        for (int s = 0; s < PASS; ++s) c[s] = lane + 32 * s < tri ? T0[(size_t)ia[s] * n + ib[s]] : (F)0;
        const F ilkk = rsq(d);
        l *= ilkk;
        __syncwarp();                              // every lane has read the pivot and the column
        if (lane < w) K[(size_t)(k + 1 + lane) * n + k] = l;
        if (lane == 0) {
            if (INV_DIAG) {
                K[(size_t)k * n + k] = ilkk;
            } else {
                K[(size_t)k * n + k] = d * ilkk;
                idg[k] = (double)ilkk;
            }
        }
#pragma unroll
        for (int p = 0; p < 3 * PASS + 1; p += PASS) {
            if (32 * p >= tri) break;
            if (p > 0)
#pragma unroll
                for (int s = 0; s < PASS; ++s)
                    if (p + s < 3 * PASS + 1)
                        c[s] = lane + 32 * (p + s) < tri ? T0[(size_t)ia[p + s < 3 * PASS + 1 ? p + s : 0] * n + ib[p + s < 3 * PASS + 1 ? p + s : 0]] : (F)0;
#pragma unroll
            for (int s = 0; s < PASS; ++s) {
                const int q = p + s < 3 * PASS + 1 ? p + s : 0;
                if (p + s >= 3 * PASS + 1 || 32 * (p + s) >= tri) continue;
                const F la = __shfl_sync(FULL, l, ia[q]), lb = __shfl_sync(FULL, l, ib[q]);
                if (lane + 32 * (p + s) < tri) T0[(size_t)ia[q] * n + ib[q]] = c[s] - la * lb;
            }
        }
        __syncwarp();
    }
    return true;
}

template <typename F, bool INV_DIAG>
__device__ bool env_cholesky(F *K, int n, const SubEnv &e, double *idg)
{
    const int lane = threadIdx.x & 31;
    for (int k = 0; k < n; ++k) {
        const F d = K[k * n + k];
        if (!(d > (F)0) || !isfinite(d)) return false;
        const F ilkk = rsq(d);
        const int R = e.lastr[k];
        __syncwarp();
        for (int q = k + 1 + lane; q <= R; q += 32) K[q * n + k] *= ilkk;
        if (lane == 0) {
            if (INV_DIAG) {
                K[k * n + k] = ilkk;
            } else {
                K[k * n + k] = d * ilkk;
                idg[k] = (double)ilkk;
            }
        }
        __syncwarp();
        const int w = R - k, tri = w * (w + 1) / 2;
        for (int t = lane; t < tri; t += 32) {
            int a, b;
            tri_index(t, a, b);
            const int r = k + 1 + a, q = k + 1 + b;
            K[r * n + q] -= K[r * n + k] * K[q * n + k];
        }
        __syncwarp();
    }
    return true;
}

// Columns c0 .. c0 + 31 of W = L^-1 [J^T b] (column-major, W[p ldw + t]; a lane per
// column): column t < m is row t of J, column m is b, columns m < t < ldw are padding
// (zero).  Row t of J is zero outside its span [jlo[t], jhi[t]), so column t of W is zero
// above jlo[t]: the warp starts at the first such row among its columns and reads J's span
// directly (no separate transposed fill).  Rows above that start are written as zeros only
// when `whole` (a reader that takes W whole: the tensor-core Gram kernel); the map's
// items skip them.  The diagonal of LT holds 1/L_pp.
template <typename F>
__device__ void solve_w_chunk(const F *LT, F *W, const double *J, const double *b, int n,
                              int m, int ldw, int c0, const SubEnv &e, bool whole)
{
    const int lane = threadIdx.x & 31;
    const int t = c0 + lane;
    const bool act = t <= m;                       // a column of J^T or b
    const bool pad = t > m && t < ldw;             // zero padding
    const int lo = !act ? n : (t == m ? 0 : e.jlo[t]);
    const int hi = !act ? n : (t == m ? n : e.jhi[t]);
    int p0 = lo;
#pragma unroll
    for (int o = 16; o; o >>= 1) p0 = min(p0, __shfl_xor_sync(0xffffffffu, p0, o));
    if (pad)
        for (int p = 0; p < n; ++p) W[(size_t)p * ldw + t] = (F)0;
    if (whole && act)
        for (int p = 0; p < p0; ++p) W[(size_t)p * ldw + t] = (F)0;
    F *x = W + (act ? t : c0);                     // idle lanes read column c0, write nothing
    const double *Jt = J + (size_t)(act && t < m ? t : 0) * n;
    for (int p = p0; p < n; ++p) {
        const F *Lp = LT + (size_t)p * n;
        F s0 = (F)0, s1 = (F)0, s2 = (F)0, s3 = (F)0;
        if (p >= lo && p < hi) s0 = (F)(t == m ? b[p] : Jt[p]);
        int q = max(e.env[p], p0);                 // x[q] = 0 above p0
        for (; q + 3 < p; q += 4) {
            s0 -= Lp[q] * x[(size_t)q * ldw];
            s1 -= Lp[q + 1] * x[(size_t)(q + 1) * ldw];
            s2 -= Lp[q + 2] * x[(size_t)(q + 2) * ldw];
            s3 -= Lp[q + 3] * x[(size_t)(q + 3) * ldw];
        }
        for (; q < p; ++q) s0 -= Lp[q] * x[(size_t)q * ldw];
        if (act) x[(size_t)p * ldw] = ((s0 + s1) + (s2 + s3)) * Lp[p];
    }
}

// The range of a prefix table pre[0 .. nsub] (pre[0] = 0, nondecreasing) that holds item w
// < pre[nsub]: the i with pre[i] <= w < pre[i + 1]
__device__ __forceinline__ int pre_find(const int *pre, int nsub, int w)
{
    int lo = 0, hi = nsub;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(pre + mid) <= w) lo = mid;
        else hi = mid;
    }
    return lo;
}

// x[q ldx] -= a[q lda] f for q0 <= q < q1 (warp, lanes across q).  Whole passes of 8 x 32
// entries load their a and x before writing any x (x and a may share a type, so the
// compiler could not move a load of a above a store to x, and each entry would cost a
// round trip); the remainder takes one more such pass if it is long, else one pass of 2 x 32
// or 32.  The passes are warp-uniform: a short range issues no predicated-off
// instructions (an FP64 one occupies its pipe all the same).
template <int K, typename F, typename G>
__device__ __forceinline__ void axpy_pass(F *x, int ldx, const G *a, int lda, int q, int q1, F f)
{
    G av[K];
    F xv[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int qq = q + 32 * k;
        av[k] = qq < q1 ? a[qq * lda] : (G)0;
        xv[k] = qq < q1 ? x[qq * ldx] : (F)0;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int qq = q + 32 * k;
        if (qq < q1) x[qq * ldx] = xv[k] - (F)av[k] * f;
    }
}

// (indices: q lda and q ldx stay below 2^31 for the supported sizes, n, m <= 2048)
template <typename F, typename G>
__device__ __forceinline__ void warp_axpy_neg(F *x, int ldx, const G *a, int lda, int q0, int q1,
                                              F f)
{
    const int lane = threadIdx.x & 31;
    if (q1 - q0 <= 32) {                     // one entry per lane at most
        const int q = q0 + lane;
        if (q < q1) x[q * ldx] -= (F)a[q * lda] * f;
        return;
    }
    int base = q0;
    for (; base + 256 <= q1; base += 256) axpy_pass<8>(x, ldx, a, lda, base + lane, q1, f);
    if (q1 - base > 64) {                    // a long range's remainder in one pass
        axpy_pass<8>(x, ldx, a, lda, base + lane, q1, f);
        return;
    }
    // at most 64 entries left
    if (q1 - base > 32) axpy_pass<2>(x, ldx, a, lda, base + lane, q1, f);
    else if (q1 > base) axpy_pass<1>(x, ldx, a, lda, base + lane, q1, f);
}

// y <- L^-1 y for one vector (stride ldy), column by column: lanes update the rows below p
template <typename F>
__device__ void env_forward_vec(const F *LT, F *y, int n, int ldy, const int *lastr)
{
    const int lane = threadIdx.x & 31;
    for (int p = 0; p < n; ++p) {
        const F yp = y[p * ldy] * LT[p * n + p];
        __syncwarp();
        if (lane == 0) y[p * ldy] = yp;
        warp_axpy_neg(y, ldy, LT + p, n, p + 1, lastr[p] + 1, yp);
        __syncwarp();
    }
}

__device__ __forceinline__ void load_quad(const float *p, float *v)
{
    const float4 a = *reinterpret_cast<const float4 *>(p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void load_quad(const double *p, double *v)
{
    const double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

// One work item of the map D = W^T W, c = W^T g of a subsystem (W = L^-1 [J^T b], column m
// is g; W column t is zero above row jlo[t]; D rows ldd apart, zero-padded from m to mp), for
// items spread over many threads: item k < nb (nb + 1) / 2 is the 4 x 4 block k of D's lower
// triangle (mirrored; per row p of W a thread loads 4 + 4 values for 16 FMAs); item
// nb (nb + 1) / 2 + q gives c and the zero padding of D for rows 4q .. 4q + 3.

template <typename F>
__device__ void map_item(const F *W, int n, int m, int mp, int ldd, int ldw, const int *jlo,
                         F *D, F *cc, int k, bool with_D)
{
    const int nb = (m + 3) / 4, ntri = nb * (nb + 1) / 2;
    if (k < ntri) {
        if (!with_D) return;
        int bi, bj;
        tri_index(k, bi, bj);
        const int r0 = 4 * bi, s0 = 4 * bj;
        int pr = n, ps = n;
        for (int q = 0; q < 4; ++q) {
            if (r0 + q < m) pr = min(pr, jlo[r0 + q]);
            if (s0 + q < m) ps = min(ps, jlo[s0 + q]);
        }
        F acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = (F)0;
#pragma unroll 4
        for (int p = max(pr, ps); p < n; ++p) {
            const F *Wp = W + (size_t)p * ldw;             // (16-byte aligned, as r0 and s0 are)
            F wr[4], ws[4];
            load_quad(Wp + r0, wr);
            load_quad(Wp + s0, ws);
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] += wr[a] * ws[b];
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int r = r0 + a, s = s0 + b;
                if (r < m && s < m && s <= r) {
                    D[r * ldd + s] = acc[a][b];
                    D[s * ldd + r] = acc[a][b];
                }
            }
        }
        return;
    }
    const int q0 = 4 * (k - ntri);
    for (int r = q0; r < q0 + 4 && r < m; ++r) {
        F a0 = (F)0, a1 = (F)0;
        int p = jlo[r];
        for (; p + 1 < n; p += 2) {
            a0 += W[p * ldw + r] * W[p * ldw + m];
            a1 += W[(p + 1) * ldw + r] * W[(p + 1) * ldw + m];
        }
        if (p < n) a0 += W[p * ldw + r] * W[p * ldw + m];
        cc[r] = a0 + a1;
        if (with_D)
            for (int t = m; t < mp; ++t) D[r * ldd + t] = (F)0;
    }
}

// K_i = A_i + beta_i J_i^T J_i (in the iteration type) for the blocks whose factorisation is
// left to the banded or the blocked tensor-core factorisation (step flag 4, set before the barrier that precedes this),
// a warp per row over every warp of the scene: the lower triangle from the first column of
// the envelope's tile of the row's tile row on (zeros left of the envelope: that
// factorisation reads whole tiles), then, for every row group whose span holds the row's
// column p (ascending), the group's products summed over its rows and added times beta: the
// arithmetic of add_jtj, entry by entry.
template <typename T, typename Dist>
__device__ void deferred_fill(const StepParams &P, const SceneDesc &S, const View<T> &V,
                              const Dist &d)
{
    const int lane = threadIdx.x & 31;
    for (int i = 0; i < S.nsub; ++i) {
        if (P.pending[S.sub0 + i] != 4) continue;
        const SubDesc &u = P.subs[S.sub0 + i];
        const int n = u.n;
        const SubEnv e = sub_env(P, u);
        const double *K = V.sdb + u.od_L, *J = V.sdb + u.od_J;
        // (FP64: in place, A's band is there; what lies outside the envelope is never read)
        constexpr bool COPY = sizeof(T) == 4;
        T *LT = COPY ? V.stb + u.ot_L : reinterpret_cast<T *>(V.sdb + u.od_L);
        const T beta = (T)V.db[S.od_beta + i];
        for (int p = d.warp; p < n; p += d.nwarps) {
            const int ep = e.env[p], q0 = e.env[p & ~127] & ~127;
            T *Lp = LT + (size_t)p * n;
            for (int q = q0 + lane; COPY && q <= p; q += 32) Lp[q] = q < ep ? (T)0 : (T)K[(size_t)p * n + q];
            __syncwarp();
            for (int g0 = 0; g0 < e.ngrp; g0 += 32) {
                bool cov = false;
                if (g0 + lane < e.ngrp) {
                    const int r0 = e.grp[g0 + lane];
                    cov = e.jlo[r0] <= p && p < e.jhi[r0];
                }
                for (unsigned mask = __ballot_sync(0xffffffffu, cov); mask; mask &= mask - 1) {
                    const int g = g0 + __ffs(mask) - 1;
                    const int r0 = e.grp[g], r1 = e.grp[g + 1], lo = e.jlo[r0];
                    for (int q = lo + lane; q <= p; q += 32) {
                        T acc = (T)0;
                        for (int r = r0; r < r1; ++r)
                            acc += (T)J[(size_t)r * n + p] * (T)J[(size_t)r * n + q];
                        Lp[q] += beta * acc;
                    }
                    __syncwarp();
                }
            }
        }
    }
}

// W = L^-1 [J^T b] of the subsystems whose step flag is `want` (3: factorised by the setup;
// 4: by the blocked tensor-core factorisation), in chunks of 32 columns, a warp per chunk over
// every warp of the scene, so that one large subsystem does not hold a single warp (and the
// scene) for all of its columns.  With flags still being set (want 3 in the setup, the spread
// distribution: no barrier after the factor loop) a chunk waits for its own subsystem's flag,
// and the chunks run smallest subsystem first (the largest are factorised first and take
// longest), so the chunks of the others overlap the largest factorisations.  Each warp ends
// its factor tasks before it takes a chunk, so every wait ends; it is bounded all the same (a
// wait that runs out marks the scene ST_TIMEOUT and skips the chunk).
template <typename T, typename Dist>
__device__ void w_chunks(const StepParams &P, const SceneDesc &S, const View<T> &V,
                         int *s_status, const Dist &d, int want)
{
    const int lane = threadIdx.x & 31;
    const double *sdb = V.sdb;
    T *stb = V.stb;
    {
        const int *wpre = P.ipool + S.pre_off, *ord = P.ipool + S.ord_off;
        const int total = __ldg(wpre + S.nsub);
        for (int w = d.warp; w < total; w += d.nwarps) {
            const int pos = pre_find(wpre, S.nsub, w);
            const int i = __ldg(ord + S.nsub - 1 - pos);
            int flag = 0;
            if (lane == 0 && !Dist::kSpread) {
                flag = P.pending[S.sub0 + i];     // set before the barrier above
            } else if (lane == 0) {
                volatile int *vf = &P.pending[S.sub0 + i];
                flag = *vf;
                for (long long spin = 0; flag == -1; ++spin) {
                    if (spin > (1ll << 26)) { *s_status = ST_TIMEOUT; break; }
                    __nanosleep(64);
                    flag = *vf;
                }
                d.fence();                        // the factor after its flag
            }
            flag = __shfl_sync(0xffffffffu, flag, 0);
            if (flag != want) continue;
            const SubDesc &u = P.subs[S.sub0 + i];
            const int ldw = (u.m + 1 + 3) / 4 * 4;
            const int c0 = 32 * (w - __ldg(wpre + pos));
            const bool whole = (P.tc_phase == 1 || P.tc_phase == 3) && u.tc;
            solve_w_chunk<T>(stb + u.ot_L, stb + u.ot_W, sdb + u.od_J, sdb + u.od_b, u.n, u.m,
                             ldw, c0, sub_env(P, u), whole);
        }
    }
}

// assemble .. factor .. map, and the per-step constants of the z-step
template <typename T, typename Dist>
__device__ long long scene_setup(const StepParams &P, const SceneDesc &S, const View<T> &V,
                                 int *s_status, int step, const Dist &d,
                                 unsigned char *big_smem = nullptr)
{
    const int lane = threadIdx.x & 31;
    constexpr bool MIXED = sizeof(T) == 4;
    double *db = V.db, *sdb = V.sdb;
    T *tb = V.tb, *stb = V.stb, *htb = V.htb;
    for (int i = d.warp; i < S.nsub; i += d.nwarps) {
        const SubDesc &u = P.subs[S.sub0 + i];
        const SubEnv e = sub_env(P, u);
        const bool keep = factor_kept(P, S, u, S.sub0 + i, step);
        double *J = sdb + u.od_J, *K = sdb + u.od_L;
        // J's rows are read only inside their column spans (model rows are written there,
        // explicit rows whole): zero the spans
        for_groups(e, [&](int r0, int r1, int lo, int w) {
            for (int k = lane; k < (r1 - r0) * w; k += 32)
                J[(size_t)(r0 + k / w) * u.n + lo + k % w] = 0.0;
        });
        if (u.kind == KIND_GENERIC) {
            const double *A = P.pool + u.gen_off;
            for (int q = lane; q < u.n * u.n; q += 32) K[q] = A[q];
            for (int q = lane; q < u.n; q += 32) sdb[u.od_b + q] = A[u.n * u.n + q];
            continue;
        }
        if (!keep) {
            // the band [env[p], lastr[p]] of every row holds A (both triangles)
            for (int b = 0; b < u.n; b += 32) {
                const int pl = min(b + lane, u.n - 1), lo = e.env[pl], hi = e.lastr[pl];
                for (int h = 0; h < 32 && b + h < u.n; ++h) {
                    const int q1 = __shfl_sync(0xffffffffu, hi, h);
                    for (int q = __shfl_sync(0xffffffffu, lo, h) + lane; q <= q1; q += 32)
                        K[(size_t)(b + h) * u.n + q] = 0.0;
                }
            }
        }
        if (u.kind == KIND_LINEAR) {
            // A = (2/h) M + (h/2) K_el (K_el sparse, scattered into the band);
            // b from the node state (Eq. ddyn, elastic force at the midpoint)
            __syncwarp();
            const double *mass = P.pool + u.gen_off;
            const double *f = mass + u.nb, *X0 = f + u.n, *Kval = X0 + u.n;
            const int *rowp = P.ipool + u.csr_off, *col = rowp + u.n + 1;
            const double gv[3] = {P.g0, P.g1, P.g2};
            const double *nodes = P.nodes + (size_t)u.body0 * SUBADMM_NODE;
            if (u.ne > 0) {
                // co-rotational: (2/h) M on the diagonal and b without the elastic force here;
                // the elements add (h/2) R K_e R^T and their forces in the pass below
                for (int p = lane; p < u.n; p += 32) {
                    const double m = mass[p / 3];
                    K[p * u.n + p] = (2.0 / P.h) * m;
                    sdb[u.od_b + p] = (2.0 / P.h) * m * nodes[(p / 3) * SUBADMM_NODE + 3 + p % 3] +
                                      f[p] + m * gv[p % 3];
                }
                __syncwarp();
                continue;
            }
            double *ux = sdb + u.od_v;               // x - X0 (v-hat is rewritten later)
            for (int p = lane; p < u.n; p += 32) ux[p] = nodes[(p / 3) * SUBADMM_NODE + p % 3] - X0[p];
            if (!keep) {
                for (int p = lane; p < u.n; p += 32) {
                    const int q1 = rowp[p + 1];
#pragma unroll 4
                    for (int q = rowp[p]; q < q1; ++q) K[p * u.n + col[q]] = 0.5 * P.h * Kval[q];
                }
                __syncwarp();
                for (int p = lane; p < u.n; p += 32) K[p * u.n + p] += (2.0 / P.h) * mass[p / 3];
            }
            __syncwarp();
            for (int p = lane; p < u.n; p += 32)
                sdb[u.od_b + p] = linear_b(p, mass, f, ux, Kval, rowp, col, nodes, P.h, gv);
        }
    }
    d.sync();
    // co-rotational blocks: every element's rotated stiffness and force, the elements of all
    // such blocks of the scene spread over every thread
    {
        int total = 0;
        for (int i = 0; i < S.nsub; ++i) total += P.subs[S.sub0 + i].ne;
        for (int w = d.tid; w < total; w += d.nthreads) {
            int el = w, i = 0;
            for (; i < S.nsub; ++i) {
                const int ne = P.subs[S.sub0 + i].ne;
                if (el < ne) break;
                el -= ne;
            }
            const SubDesc &u = P.subs[S.sub0 + i];
            const double *X0 = P.pool + u.gen_off + u.nb + u.n;
            corot_element(P.ipool + u.tet_off + 4 * el, P.pool + u.ke_off + 144 * (size_t)el, X0,
                          P.nodes + (size_t)u.body0 * SUBADMM_NODE, P.h, u.n, sdb + u.od_L,
                          sdb + u.od_b);
        }
    }
    // rigid bodies: diagonal A = (2/h) M and b (lane per body)
    for (int i = d.warp; i < S.nsub; i += d.nwarps) {
        const SubDesc &u = P.subs[S.sub0 + i];
        if (u.kind != KIND_RIGID) continue;
        for (int k = lane; k < u.nb; k += 32) {
            double Ad[6], bb[6];
            body_dynamics(P.bodies + (size_t)(u.body0 + k) * SUBADMM_BODY, P.h, P.g0, P.g1, P.g2,
                          Ad, bb);
            double *K = sdb + u.od_L;
            for (int d = 0; d < 6; ++d) {
                const int q = 6 * k + d;
                K[q * u.n + q] = Ad[d];
                sdb[u.od_b + q] = bb[d];
            }
        }
    }
    // constraint rows into J (FP64) and e; constraints in the host's assembly order, which
    // groups kinds by warp so a warp runs one kind's code path
    T *E = tb + S.ot_e;
    for (int a = d.tid; a < S.nasm; a += d.nthreads) {
        const int j = P.asm_order[S.asm_g0 + a];
        if (j < 0) continue;
        const ConDesc &c = P.cons[S.con0 + j];
        if (c.src <= SRC_CONTACT) {
            const double *p = P.pool + c.par_off + 3;
            for (int r = 0; r < c.rows; ++r) E[c.row0 + r] = (T)p[r];
            const double *Jp = p + c.rows;
            for (int s = 0; s < c.ns; ++s) {
                const SubDesc &u = P.subs[S.sub0 + c.sub[s]];
                for (int r = 0; r < c.rows; ++r) {
                    double *Jr = sdb + u.od_J + (c.sr[s] + r - u.sr0) * u.n;
                    for (int q = 0; q < u.n; ++q) Jr[q] = Jp[r * u.n + q];
                }
                Jp += c.rows * u.n;
            }
        } else {
            double Ja[30], Jb[30], ee[5], kk = 0.0, al = 0.0;
            model_rows(c, P.pool + c.par_off, P.bodies, P.nodes, P.h, P.gamma, Ja, Jb, ee, &kk, &al);
            for (int r = 0; r < c.rows; ++r) E[c.row0 + r] = (T)ee[r];
            {
                // a body side fills 6 columns at 6 * index, a node side 3 columns at 3 * index
                const SubDesc &u = P.subs[S.sub0 + c.sub[0]];
                const int wa = c.node_a ? 3 : 6;
                for (int r = 0; r < c.rows; ++r) {
                    double *Jr = sdb + u.od_J + (c.sr[0] + r - u.sr0) * u.n + wa * c.ba;
                    for (int q = 0; q < wa; ++q) Jr[q] = Ja[6 * r + q];
                }
            }
            if (c.side_b >= 0) {
                const SubDesc &u = P.subs[S.sub0 + c.sub[c.side_b]];
                const int wb = c.node_b ? 3 : 6;
                for (int r = 0; r < c.rows; ++r) {
                    double *Jr = sdb + u.od_J + (c.sr[c.side_b] + r - u.sr0) * u.n + wb * c.bb;
                    for (int q = 0; q < wb; ++q) Jr[q] += Jb[6 * r + q];
                }
            }
        }
    }
    // factor-ready flags of this step (see the factor loop): -1 until a subsystem is done
    for (int i = d.tid; i < S.nsub; i += d.nthreads) P.pending[S.sub0 + i] = -1;
    d.sync();
    const long long t_asm = clock64();
    // per subsystem (one warp each): beta, K = A + beta J^T J and its Cholesky factor, then
    // the map W = L^-1 [J^T b], D = W^T W, c.  The FP64 form and the stiff blocks of the mixed
    // form factorise K in FP64 (rounded into the T copy); the other mixed blocks factorise in
    // FP32, keeping the FP64 A, b and J for the recovery and refinement of v-hat.
    if constexpr (!Dist::kSpread) {
        // the large subsystems whose factor is kept, a block each: c = J K^-1 b from one solve
        // and J's spans (two solves of the vector instead of g = L^-1 b and a pass over the
        // whole of W, 3 MB a slab: 3.6M -> 0.63M SM cycles for 64 slabs); the flag 0 then
        // leaves nothing to the passes below
        for (int k = blockIdx.x; big_smem && k < S.nbig; k += gridDim.x) {
            const int i = P.ipool[S.big_off + k], gsub = S.sub0 + i;
            const SubDesc &u = P.subs[gsub];
            if (!factor_kept(P, S, u, gsub, step)) continue;
            const SubEnv e = sub_env(P, u);
            const int n = u.n;
            const double *b = sdb + u.od_b, *J = sdb + u.od_J;
            const T *LT = stb + u.ot_L;
            T *cc = htb + u.ot_c;
            BlockSolve<T> bs(big_smem, n);
            for (int p = threadIdx.x; p < n; p += Dist::kThreads) bs.x[p] = (T)b[p];
            block_solve_begin<Dist::kThreads>(LT, n, e.env, bs);
            block_forward<Dist::kThreads, T, true>(LT, nullptr, n, e.lastr, bs);
            block_backward<Dist::kThreads, T, true>(LT, nullptr, n, bs);
            for (int r = threadIdx.x; r < u.m; r += Dist::kThreads) {
                T acc = (T)0;
                for (int p = e.jlo[r]; p < e.jhi[r]; ++p) acc += (T)J[(size_t)r * n + p] * bs.x[p];
                cc[r] = acc;
            }
            if (threadIdx.x == 0) {
                if (step == 0) {
                    db[S.od_beta + i] = P.beta[gsub];
                    db[S.od_flag + i] = (P.subflag[gsub] & 2) ? 1.0 : 0.0;
                }
                P.pending[gsub] = 0;
            }
            __syncthreads();
        }
    }
    for (int k = d.warp; k < S.nsub; k += d.nwarps) {
        const int i = Dist::kSpread ? __ldg(P.ipool + S.ord_off + k) : k;   // largest first
        const SubDesc &u = P.subs[S.sub0 + i];
        const int gsub = S.sub0 + i;
        if (!Dist::kSpread && big_smem && u.n >= SUBADMM_BIG && factor_kept(P, S, u, gsub, step)) continue;
        // W's leading dimension: m + 1 columns rounded up to 4 (map_item reads 4-column blocks)
        const int n = u.n, m = u.m, ldw = (m + 1 + 3) / 4 * 4;
        const SubEnv e = sub_env(P, u);
        double *J = sdb + u.od_J, *K = sdb + u.od_L, *b = sdb + u.od_b, *idg = sdb + u.od_id;
        T *LT = stb + u.ot_L, *W = stb + u.ot_W;
        if (factor_kept(P, S, u, gsub, step)) {
            // constant K_i: only g = L^-1 b and c change (and D when the launch lost it)
            if (step == 0 && lane == 0) {
                db[S.od_beta + i] = P.beta[gsub];
                db[S.od_flag + i] = (P.subflag[gsub] & 2) ? 1.0 : 0.0;
            }
            for (int p = lane; p < n; p += 32) W[p * ldw + m] = (T)b[p];
            __syncwarp();
            env_forward_vec<T>(LT, W + m, n, ldw, e.lastr);
            // c (and D if the launch lost it) below, over every thread of the scene
            __syncwarp();
            if (lane == 0) {
                d.fence();
                *(volatile int *)&P.pending[gsub] = (step == 0 && !S.hot_global) ? 2 : 1;
            }
            __syncwarp();
            continue;
        }
        // beta_i = Tr(A_i) / Tr(J_ci^T J_ci)  (Sec. III-D)
        double beta;
        if (!MIXED) {
            double trA = 0.0, trJ = 0.0;
            for (int q = lane; q < n; q += 32) trA += K[q * n + q];
            for_groups(e, [&](int r0, int r1, int lo, int w) {      // J's rows inside their spans
                for (int k = lane; k < (r1 - r0) * w; k += 32) {
                    const double x = J[(size_t)(r0 + k / w) * n + lo + k % w];
                    trJ += x * x;
                }
            });
            trA = warp_sum(trA);
            trJ = warp_sum(trJ);
            beta = P.beta_fixed ? P.rho : (trJ > 0.0 ? trA / trJ : 1.0);
        } else {
            T trA = (T)0, trJ = (T)0;
            for (int q = lane; q < n; q += 32) trA += (T)K[q * n + q];
            for_groups(e, [&](int r0, int r1, int lo, int w) {
                for (int k = lane; k < (r1 - r0) * w; k += 32) {
                    const T jq = (T)J[(size_t)(r0 + k / w) * n + lo + k % w];
                    trJ += jq * jq;
                }
            });
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                trA += __shfl_xor_sync(0xffffffffu, trA, o);
                trJ += __shfl_xor_sync(0xffffffffu, trJ, o);
            }
            beta = (double)(P.beta_fixed ? (T)P.rho : (trJ > (T)0 ? trA / trJ : (T)1));
        }
        beta *= P.beta_scale[gsub];
        if (P.pj) beta = 0.0;                       // Projected Jacobi: K_i = A_i
        if (lane == 0) {
            db[S.od_beta + i] = beta;
            P.beta[gsub] = beta;
            P.beta_used[gsub] = P.beta_scale[gsub];
        }
        bool stiff = true;
        if (MIXED) {
            // stiffness test: the spread of K's diagonal bounds its condition number from
            // below; a stiff or high-mass-ratio block (spread > 1e3) is factorised in FP64
            const T bt = (T)beta;
            T dmax = (T)0, dmin = (T)3.0e38;
            for (int b = 0; b < n; b += 32) {
                const int p = b + lane;
                T cs = (T)0;                       // rows whose span holds column p, in order
                for_groups(e, [&](int r0, int r1, int lo, int w) {
                    if (p < lo || p >= lo + w) return;
                    for (int r = r0; r < r1; ++r) {
                        const T jr = (T)J[(size_t)r * n + p];
                        cs += jr * jr;
                    }
                });
                if (p >= n) continue;
                const T dk = (T)K[p * n + p] + bt * cs;
                dmax = dk > dmax ? dk : dmax;
                dmin = dk < dmin ? dk : dmin;
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                const T a = __shfl_xor_sync(0xffffffffu, dmax, o);
                const T c = __shfl_xor_sync(0xffffffffu, dmin, o);
                dmax = a > dmax ? a : dmax;
                dmin = c < dmin ? c : dmin;
            }
            stiff = !(dmin > (T)0) || dmax > (T)1.0e3 * dmin;
            if (lane == 0) db[S.od_flag + i] = stiff ? 1.0 : 0.0;
        }
        bool ok;
        const bool defer = (!MIXED || !stiff) && P.tc_factor && P.tc_phase == 1 && u.tc;
        if (stiff && !defer) {
            add_jtj<double>(K, n, J, e, beta);
            ok = u.bw <= kNarrowBand ? narrow_cholesky<double, false>(K, n, e, idg)
                                     : env_cholesky<double, false>(K, n, e, idg);
            if (ok) {
                copy_band(LT, K, n, e.env, [&](int p, int q, double v) { return q == p ? (T)idg[p] : (T)v; });
            }
        } else if (defer) {
            ok = true;                            // K by deferred_fill, below
        } else {
            copy_band(LT, K, n, e.env, [](int, int, double v) { return (T)v; });
            __syncwarp();
            add_jtj<T>(LT, n, J, e, (T)beta);
            ok = u.bw <= kNarrowBand ? narrow_cholesky<T, true>(LT, n, e, nullptr)
                                     : env_cholesky<T, true>(LT, n, e, nullptr);
        }
        if (u.cst && lane == 0) P.subflag[gsub] = ok ? (1 | (stiff ? 2 : 0)) : 0;
        __syncwarp();
        if (lane == 0) {
            d.fence();                            // the factor before its flag
            // 3: W, then D and c, below; 4: factor, W, D and c after this launch
            *(volatile int *)&P.pending[gsub] = ok ? (defer ? 4 : 3) : 0;
            if (!ok) *s_status = ST_NOTSPD;
        }
        __syncwarp();
    }
    // W = L^-1 [J^T b] of the subsystems factorised above (flag 3); K of the deferred ones
    if (!Dist::kSpread) d.sync();
    if (P.tc_factor && P.tc_phase == 1) deferred_fill<T>(P, S, V, d);
    w_chunks<T>(P, S, V, s_status, d, 3);
    d.sync();
    // the maps D = W^T W and c = W^T g of this step (pending >= 2: D and c, 1: c only), their
    // items (rows of c, then 4 x 4 blocks of D) spread over every thread of the scene and
    // found through the scene's prefix tables; the tensor-core Gram kernel forms them for
    // the tc subsystems in the first launch of a three-launch step
    {
        const int *cpre = P.ipool + S.pre_off + (S.nsub + 1), *dpre = cpre + (S.nsub + 1);
        const int ctot = __ldg(cpre + S.nsub), total = ctot + __ldg(dpre + S.nsub);
        for (int w = d.tid; w < total; w += d.nthreads) {
            const bool cpart = w < ctot;
            const int wl = cpart ? w : w - ctot;
            const int i = pre_find(cpart ? cpre : dpre, S.nsub, wl);
            const int pend = P.pending[S.sub0 + i];
            if (pend == 0 || (!cpart && pend < 2)) continue;
            const SubDesc &u = P.subs[S.sub0 + i];
            if (P.tc_phase == 1 && u.tc) continue;
            const int nb = (u.m + 3) / 4;
            const int k = (cpart ? nb * (nb + 1) / 2 : 0) + wl - __ldg((cpart ? cpre : dpre) + i);
            const int ldw = (u.m + 1 + 3) / 4 * 4;
            map_item<T>(stb + u.ot_W, u.n, u.m, u.mpad, u.ldd, ldw, sub_env(P, u).jlo,
                        htb + u.ot_D, htb + u.ot_c, k, pend >= 2);
        }
    }
    d.sync();
    // per-step z-step constants: 1/s, soft gain k/(1 + s alpha k), alpha, mu (per row);
    // beta and 1/beta per side-row
    T *INVS = tb + S.ot_invs, *KF = tb + S.ot_kf, *AL = tb + S.ot_al, *MU = tb + S.ot_mu;
    T *INVB = tb + S.ot_invb, *BT = tb + S.ot_b;
    const double *BETA = db + S.od_beta;
    for (int j = d.tid; j < S.ncon; j += d.nthreads) {
        const ConDesc &c = P.cons[S.con0 + j];
        if (P.pj) {
            // Projected Jacobi: 1/delta per row, delta = the sum over its sides of D's diagonal
            // entry (both tangents of a contact take the larger of theirs), soft gain
            // k/(1 + k alpha delta); beta and 1/beta per side-row are zero
            double kk, al, mu;
            con_params(c, P.pool, P.h, kk, al, mu);
            double dl[3] = {0.0, 0.0, 0.0};
            for (int r = 0; r < c.rows; ++r) {
                double dr = 0.0;
                for (int q = 0; q < c.ns; ++q) {
                    const SubDesc &u = P.subs[S.sub0 + c.sub[q]];
                    const int lr = c.sr[q] + r - u.sr0;
                    dr += (double)htb[u.ot_D + (size_t)lr * u.ldd + lr];
                }
                if (c.type == TYPE_CONTACT) dl[r] = dr;
                else {
                    INVS[c.row0 + r] = (T)(1.0 / dr);
                    KF[c.row0 + r] = (T)(c.type == TYPE_SOFT ? kk / (1.0 + kk * al * dr) : 0.0);
                }
                AL[c.row0 + r] = (T)al;
                MU[c.row0 + r] = (T)mu;
            }
            if (c.type == TYPE_CONTACT) {
                const double dt = dl[1] > dl[2] ? dl[1] : dl[2];
                INVS[c.row0] = (T)(1.0 / dl[0]);
                INVS[c.row0 + 1] = (T)(1.0 / dt);
                INVS[c.row0 + 2] = (T)(1.0 / dt);
                for (int r = 0; r < 3; ++r) KF[c.row0 + r] = (T)0;
            }
            for (int q = 0; q < c.ns; ++q)
                for (int r = 0; r < c.rows; ++r) {
                    INVB[c.sr[q] + r] = (T)0;
                    BT[c.sr[q] + r] = (T)0;
                }
            continue;
        }
        double s = 0.0;
        for (int q = 0; q < c.ns; ++q) s += 1.0 / BETA[c.sub[q]];
        double kk, al, mu;
        con_params(c, P.pool, P.h, kk, al, mu);
        const double kf = (c.type == TYPE_SOFT) ? kk / (1.0 + s * al * kk) : 0.0;
        for (int r = 0; r < c.rows; ++r) {
            INVS[c.row0 + r] = (T)(1.0 / s);
            KF[c.row0 + r] = (T)kf;
            AL[c.row0 + r] = (T)al;
            MU[c.row0 + r] = (T)mu;
        }
        for (int q = 0; q < c.ns; ++q) {
            const double be = BETA[c.sub[q]];
            for (int r = 0; r < c.rows; ++r) {
                INVB[c.sr[q] + r] = (T)(1.0 / be);
                BT[c.sr[q] + r] = (T)be;
            }
        }
    }
    d.sync();
    return t_asm;
}

// out += J^T w (FP64) over the column span of each row group (lanes across the span, each
// summing over the group's rows, then one update of out per group), in row order:
// deterministic, and O(sum of spans) instead of O(m n)
template <typename W>
__device__ __forceinline__ void add_jt(double *out, const double *J, int n, const SubEnv &e,
                                       const W *w)
{
    const int lane = threadIdx.x & 31;
    for_groups(e, [&](int r0, int r1, int lo, int sw) {
        for (int p = lo + lane; p < lo + sw; p += 32) {
            const double old = out[p];
            double acc = 0.0;
            for (int r = r0; r < r1; ++r) acc += J[(size_t)r * n + p] * (double)w[r];
            out[p] = old + acc;
        }
        __syncwarp();
    });
}

// Triangular solves with the T factor (1/L_pp on its diagonal), in place on s (warp),
// inside the envelope.
template <typename T>
__device__ __forceinline__ void warp_chol_solve(const T *LT, T *s, int n, const SubEnv &e, int bw)
{
    const int lane = threadIdx.x & 31;
    if (bw <= kNarrowBand) {
        auto inv = [LT, n](int r) { return LT[(size_t)r * n + r]; };
        warp_band_forward<T>(LT, n, e.env, s, inv);
        warp_band_backward<T>(LT, n, e.env, s, inv);
        return;
    }
    for (int p = 0; p < n; ++p) {              // L y = s (column-oriented)
        const T yp = s[p] * LT[p * n + p];
        __syncwarp();
        if (lane == 0) s[p] = yp;
        warp_axpy_neg(s, 1, LT + p, n, p + 1, e.lastr[p] + 1, yp);
        __syncwarp();
    }
    for (int p = n - 1; p >= 0; --p) {         // L^T v = y
        const T vp = s[p] * LT[p * n + p];
        __syncwarp();
        if (lane == 0) s[p] = vp;
        warp_axpy_neg(s, 1, LT + p * n, 1, e.env[p], p, vp);
        __syncwarp();
    }
}

// J^T w of one column p (FP64): the row groups that hold it in order, each summed over its rows
// before it is added (the arithmetic of add_jt); grp: the groups' first rows and column spans
template <typename W>
__device__ __forceinline__ double column_jt(double out, const double *J, int n, int p, int ngrp,
                                            const int *grp, const W *w)
{
    for (int g = 0; g < ngrp; ++g) {
        if (p < grp[3 * g + 1] || p >= grp[3 * g + 2]) continue;
        double acc = 0.0;
        for (int r = grp[3 * g]; r < grp[3 * g + 3]; ++r) acc += J[(size_t)r * n + p] * (double)w[r];
        out += acc;
    }
    return out;
}

// v-hat of one subsystem by a whole block (see recover_v): the vector and the row groups'
// spans in shared memory, the solves of block_solve.cuh.  A linear block's A is read through
// its sparse pattern (SubDesc::pat_off; 45 entries a row where the band holds 270).  1200-DOF slabs, the exit phase:
// FP32 factor with refinement 10.6M -> 2.2M SM cycles, FP64 factor 5.0M -> 1.5M.
template <typename T, int NT>
__device__ __noinline__ void block_recover_one(const StepParams &P, const SceneDesc &S, const View<T> &V,
                                               const T *w, int i, unsigned char *smem)
{
    constexpr bool MIXED = sizeof(T) == 4;
    const SubDesc &u = P.subs[S.sub0 + i];
    const int n = u.n, m = u.m, tid = threadIdx.x;
    const SubEnv e = sub_env(P, u);
    const double *J = V.sdb + u.od_J, *Lf = V.sdb + u.od_L, *b = V.sdb + u.od_b;
    double *idg = V.sdb + u.od_id, *v = V.sdb + u.od_v;
    const T *wi = w + u.sr0;
    int *grp = reinterpret_cast<int *>(smem);
    smem += block_solve_groups(e.ngrp);
    for (int g = tid; g <= e.ngrp; g += NT) {
        grp[3 * g] = e.grp[g];
        if (g < e.ngrp) { grp[3 * g + 1] = e.jlo[e.grp[g]]; grp[3 * g + 2] = e.jhi[e.grp[g]]; }
    }
    __syncthreads();
    if (!MIXED || V.db[S.od_flag + i] != 0.0) {
        BlockSolve<double> s(smem, n);
        for (int p = tid; p < n; p += NT)
            s.x[p] = column_jt(b[p], J, n, p, e.ngrp, grp, wi);
        __syncthreads();
        block_solve_begin<NT>(Lf, n, e.env, s);
        block_forward<NT, double, false>(Lf, idg, n, e.lastr, s);
        block_backward<NT, double, false>(Lf, idg, n, s);
        for (int p = tid; p < n; p += NT) v[p] = s.x[p];
        __syncthreads();
        return;
    }
    BlockSolve<T> s(smem, n);
    const T *LT = V.stb + u.ot_L;
    block_solve_begin<NT>(LT, n, e.env, s);
    double *rhs = idg, *t = V.sdb + u.od_t;
    const double beta = V.db[S.od_beta + i];
    for (int p = tid; p < n; p += NT) {
        rhs[p] = column_jt(b[p], J, n, p, e.ngrp, grp, wi);
        s.x[p] = (T)rhs[p];
    }
    __syncthreads();
    block_forward<NT, T, true>(LT, nullptr, n, e.lastr, s);
    block_backward<NT, T, true>(LT, nullptr, n, s);
    for (int p = tid; p < n; p += NT) v[p] = (double)s.x[p];
    __syncthreads();
    for (int r = tid; r < m; r += NT) {
        double acc = 0.0;
        for (int p = e.jlo[r]; p < e.jhi[r]; ++p) acc += J[(size_t)r * n + p] * v[p];
        t[r] = acc * -beta;
    }
    __syncthreads();
    const int *rowp = P.ipool + u.pat_off, *col = rowp + n + 1;
    for (int p = tid; p < n; p += NT) {
        double acc = column_jt(rhs[p], J, n, p, e.ngrp, grp, t);
        const double *Ap = Lf + (size_t)p * n;
        if (u.kind == KIND_LINEAR) {
            bool diag = false;                    // (K's pattern may leave a diagonal entry out)
            for (int q = rowp[p]; q < rowp[p + 1]; ++q) {
                const int c = col[q];
                diag = diag || c == p;
                acc -= Ap[c] * v[c];
            }
            if (!diag) acc -= Ap[p] * v[p];
        } else if (u.kind == KIND_RIGID) {
            acc -= Ap[p] * v[p];                  // A is diagonal
        } else {
            for (int q = e.env[p]; q <= e.lastr[p]; ++q) acc -= Ap[q] * v[q];
        }
        s.x[p] = (T)acc;
    }
    __syncthreads();
    block_forward<NT, T, true>(LT, nullptr, n, e.lastr, s);
    block_backward<NT, T, true>(LT, nullptr, n, s);
    for (int p = tid; p < n; p += NT) v[p] += (double)s.x[p];
    __syncthreads();
}

// v-hat of the last v-step, v = K^-1 (b + J^T w), in FP64 (warp per subsystem) into od_v.
// With an FP64 factor (FP64 form, or a stiff block of the mixed form): two triangular
// solves.  With an FP32 factor: a solve, then one step of iterative refinement with the
// residual b + J^T w - K v formed in FP64 from A (kept in od_L) and J:
// K v = A v + beta J^T (J v).
// `fast` (may be null): per-warp shared memory of fast_len T values; the FP32 solves of a
// subsystem with n <= fast_len run on a copy there instead of on the global scratch vector.
// `big_smem` (may be null): shared memory of this block in which it solves the subsystems of at
// least SUBADMM_BIG DOF, a block per subsystem; the others go to the warps, from the last
// block on (the first blocks hold the large ones).
template <typename T, typename Dist>
__device__ void recover_v(const StepParams &P, const SceneDesc &S, const View<T> &V, const T *w,
                          const Dist &d, T *fast = nullptr, int fast_len = 0,
                          unsigned char *big_smem = nullptr)
{
    constexpr bool MIXED = sizeof(T) == 4;
    const int lane = threadIdx.x & 31;
    if constexpr (Dist::kBig)                     // (grid_iter.cuh)
        for (int k = blockIdx.x; big_smem && k < S.nbig; k += gridDim.x)
            block_recover_one<T, Dist::kThreads>(P, S, V, w, P.ipool[S.big_off + k], big_smem);
    const int w0 = Dist::kSpread || !big_smem ? d.warp : d.nwarps - 1 - d.warp;
    for (int k = w0; k < S.nsub; k += d.nwarps) {
        const int i = Dist::kSpread ? __ldg(P.ipool + S.ord_off + k) : k;   // largest first
        const SubDesc &u = P.subs[S.sub0 + i];
        if (big_smem && u.n >= SUBADMM_BIG) continue;
        const int n = u.n, m = u.m;
        const SubEnv e = sub_env(P, u);
        // od_L holds the FP64 factor L (FP64 form) or A itself (mixed form)
        const double *J = V.sdb + u.od_J, *Lf = V.sdb + u.od_L, *b = V.sdb + u.od_b;
        double *idg = V.sdb + u.od_id;
        double *v = V.sdb + u.od_v;
        const T *wi = w + u.sr0;
        if (!MIXED || V.db[S.od_flag + i] != 0.0) {
            for (int p = lane; p < n; p += 32) v[p] = b[p];
            __syncwarp();
            add_jt(v, J, n, e, wi);
            if (u.bw <= kNarrowBand) {
                auto inv = [idg](int r) { return idg[r]; };
                warp_band_forward<double>(Lf, n, e.env, v, inv);
                warp_band_backward<double>(Lf, n, e.env, v, inv);
                continue;
            }
            for (int p = 0; p < n; ++p) {          // L y = rhs (column-oriented)
                const double yp = v[p] * idg[p];
                __syncwarp();
                if (lane == 0) v[p] = yp;
                warp_axpy_neg(v, 1, Lf + p, n, p + 1, e.lastr[p] + 1, yp);
                __syncwarp();
            }
            for (int p = n - 1; p >= 0; --p) {     // L^T v = y
                const double vp = v[p] * idg[p];
                __syncwarp();
                if (lane == 0) v[p] = vp;
                warp_axpy_neg(v, 1, Lf + p * n, 1, e.env[p], p, vp);
                __syncwarp();
            }
            continue;
        }
        const T *LT = V.stb + u.ot_L;
        T *s = (fast && n <= fast_len) ? fast : V.stb + u.ot_s;
        double *rhs = idg;                          // (unused by the mixed factor)
        double *t = V.sdb + u.od_t;
        const double beta = V.db[S.od_beta + i];
        for (int p = lane; p < n; p += 32) rhs[p] = b[p];
        __syncwarp();
        add_jt(rhs, J, n, e, wi);
        for (int p = lane; p < n; p += 32) s[p] = (T)rhs[p];
        __syncwarp();
        warp_chol_solve<T>(LT, s, n, e, u.bw);
        for (int p = lane; p < n; p += 32) v[p] = (double)s[p];
        __syncwarp();
        // one refinement step: r = rhs - A v - beta J^T (J v); v += K^-1 r.  Row p of A lies
        // inside the band [env[p], lastr[p]]
        for (int r = lane; r < m; r += 32) {
            double acc = 0.0;
            for (int p = e.jlo[r]; p < e.jhi[r]; ++p) acc += J[r * n + p] * v[p];
            t[r] = acc;
        }
        __syncwarp();
        for (int r = lane; r < m; r += 32) t[r] *= -beta;
        __syncwarp();
        // s = rhs - A v - beta J^T t, with J^T (-beta t) added into the FP64 rhs copy
        add_jt(rhs, J, n, e, t);
        for (int p = lane; p < n; p += 32) {
            double acc = rhs[p];
            for (int q = e.env[p]; q <= e.lastr[p]; ++q) acc -= Lf[p * n + q] * v[q];     // A v
            s[p] = (T)acc;
        }
        __syncwarp();
        warp_chol_solve<T>(LT, s, n, e, u.bw);
        for (int p = lane; p < n; p += 32) v[p] += (double)s[p];
        __syncwarp();
    }
}

// The block kernel's once-per-step phases as calls, so that the register allocation of its
// iteration loop is not shaped by the setup code's.  The parameters and the scene's descriptor stay
// where they are (parameter and shared memory): by value they took 500 bytes of every thread's
// frame, through the L1 that the setup lives on, and registers across the calls.
template <typename T>
__device__ __noinline__ long long block_setup(const StepParams &P, const SceneDesc &S, View<T> V, int *status,
                                              int step)
{
    return scene_setup<T>(P, S, V, status, step, BlockDist());
}

template <typename T>
__device__ __noinline__ void block_recover(const StepParams &P, const SceneDesc &S, View<T> V, const T *w)
{
    recover_v<T>(P, S, V, w, BlockDist());
}

// Initial z and u = -lambda of a step (Algorithm 1, before the loop): cold (zeros), warm
// from the previous step's lambda and z, or from the learned initial lambda (z from the
// previous step); y^0 = beta z^0 + u^0 and w^0 = beta z^0 - u^0.
template <typename T, typename Dist>
__device__ void init_duals(const StepParams &P, const SceneDesc &S, const View<T> &V, T *LAM,
                           T *Z, T *ZO, T *X, T *Y, T *YO, T *W0, const T *BT, bool learned,
                           const Dist &d)
{
    const double *lam = learned ? P.lam0 : P.lam;
    const bool warm = learned || P.warm_prev;
    for (int r = d.tid; r < S.nrow; r += d.nthreads) LAM[r] = warm ? (T)lam[S.row_g0 + r] : (T)0;
    for (int t = d.tid; t < S.nsr; t += d.nthreads) {
        if (V.mlen[t] == 0) continue;                 // padding side-row
        const T beta = BT[t];
        const T z = warm ? (T)P.z[S.sr_g0 + t] : (T)0;
        const T l = warm ? (T)lam[S.row_g0 + V.row[t]] : (T)0;
        Z[t] = z;
        ZO[t] = z;
        X[t] = (T)0;
        Y[t] = beta * z - l;
        YO[t] = Y[t];
        W0[t] = beta * z + l;
    }
    d.sync();
}

// One item of a Projected Jacobi iteration (the comparison solver of Sec. IV-B): the row's
// (or contact's) constraint value from the x of its sides, the relaxed Jacobi update of its
// impulse with 1/delta from INVS (soft rows: the soft law with x linearised in the row's own
// lambda; contacts: normal clamped at 0, tangents scaled onto the friction disk), w =
// lambda on every side for the next v-step, and the natural residual |d lambda| delta /
// omega, written as x - z of the first side-row (z = x on the others) so that the step's
// residuals report it; returns its bits
template <typename T, typename U>
__device__ __forceinline__ U pj_item(const Item &it, const int *ls, const T *X, const T *E,
                                     const T *INVS, const T *KF, const T *AL, const T *MU,
                                     T *LAM, T *Z, T *ZO, T *wn, T om, U mloc)
{
    const int nr = it.type == TYPE_CONTACT ? 3 : 1;
    T xr[3] = {(T)0, (T)0, (T)0}, lo[3], ln[3], id[3];
    for (int s = 0; s < it.ns; ++s)
        for (int r = 0; r < nr; ++r) xr[r] += X[ls[s] + r];
    for (int r = 0; r < nr; ++r) { lo[r] = LAM[it.row + r]; id[r] = INVS[it.row + r]; }
    if (it.type == TYPE_CONTACT) {
        T n = lo[0] - om * (xr[0] + E[it.row]) * id[0];
        n = n > (T)0 ? n : (T)0;
        T l1 = lo[1] - om * (xr[1] + E[it.row + 1]) * id[1];
        T l2 = lo[2] - om * (xr[2] + E[it.row + 2]) * id[2];
        const T lim = MU[it.row] * n, t2 = l1 * l1 + l2 * l2;
        if (t2 > lim * lim) { const T f = lim * rsq(t2); l1 *= f; l2 *= f; }
        ln[0] = n; ln[1] = l1; ln[2] = l2;
    } else if (it.type == TYPE_SOFT) {
        const T dl = (T)1 / id[0];
        const T ls_ = -KF[it.row] * (E[it.row] + AL[it.row] * (xr[0] - dl * lo[0]));
        ln[0] = lo[0] + om * (ls_ - lo[0]);
    } else {
        ln[0] = lo[0] - om * (xr[0] + E[it.row]) * id[0];
        if (it.type == TYPE_HARD) ln[0] = ln[0] > (T)0 ? ln[0] : (T)0;
    }
    for (int r = 0; r < nr; ++r) {
        LAM[it.row + r] = ln[r];
        const T res = fabs(ln[r] - lo[r]) / (om * id[r]);
        mloc = umax(mloc, rbits(res));
        for (int s = 0; s < it.ns; ++s) {
            const int t = ls[s] + r;
            const T zv = s == 0 ? X[t] - res : X[t];
            ZO[t] = zv;
            Z[t] = zv;
            wn[t] = ln[r];
        }
    }
    return mloc;
}

}  // namespace subadmm
#include "item_iter.cuh"
namespace subadmm {

// NT threads per block: SUBADMM_THREADS, or SUBADMM_WIDE for a generic variant of a class
// whose scenes take a whole SM's shared memory (one block per SM), which then uses the whole
// register file and twice the warps per scene
template <typename T, int SPLIT, bool CACHED, int NT = SUBADMM_THREADS>
__global__ void __launch_bounds__(NT, (CACHED || NT > SUBADMM_THREADS) ? 1 : 2) step_kernel(const __grid_constant__ StepParams P)
{
    static_assert(!CACHED || NT == SUBADMM_THREADS, "the register-cached map is laid out for 256 threads");
    constexpr int NW = NT / 32;
    using VT = typename VecOf<T>::V;
    using U = typename VecOf<T>::U;
    constexpr int VN = VecOf<T>::N;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ double red[4][SUBADMM_MAXWARPS];
    __shared__ U ured[NW];
    __shared__ int s_status;
    __shared__ SceneDesc s_scene;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr bool MIXED = sizeof(T) == 4;

    for (int k = blockIdx.x; k < P.nscenes; k += gridDim.x) {
        const int sc = P.scene_ids[k];
        __syncthreads();                           // (the scene before this one is done)
        for (int q = tid; q < (int)(sizeof(SceneDesc) / 4); q += NT)
            reinterpret_cast<int *>(&s_scene)[q] = reinterpret_cast<const int *>(P.scenes + sc)[q];
        __syncthreads();
        const SceneDesc &S = s_scene;
        const View<T> V = scene_view<T>(P, S, smraw);
        T *X = V.tb + S.ot_x, *Y = V.tb + S.ot_y, *Z = V.tb + S.ot_z, *LAM = V.tb + S.ot_lam;
        T *YO = V.tb + S.ot_yo, *ZO = V.tb + S.ot_zo;
        T *E = V.tb + S.ot_e, *INVB = V.tb + S.ot_invb, *BT = V.tb + S.ot_b;
        T *INVS = V.tb + S.ot_invs, *KF = V.tb + S.ot_kf, *AL = V.tb + S.ot_al;
        T *MU = V.tb + S.ot_mu;
        T *const W0 = V.tb + S.ot_w0, *const W1 = V.tb + S.ot_w1;
        // per-side-row arrays start zero (padding side-rows between subsystems stay zero)
        for (int q = tid; q < S.ot_lam - S.ot_x; q += blockDim.x) V.tb[S.ot_x + q] = (T)0;
        scene_tables<T>(P, S, V, BlockDist());
        __syncthreads();

        for (int step = 0; step < P.n_steps; ++step) {
            if (tid == 0) s_status = ST_OK;
            __syncthreads();
            PhaseClock pc(P.phase ? P.phase + 8 * sc : nullptr);
            pc.mark_at(PHASE_ASSEMBLE, block_setup<T>(P, S, V, &s_status, step));
            pc.mark(PHASE_FACTOR);
            const int status0 = s_status;
            if (status0 != ST_OK) {
                // K_i not SPD: report, leave the state untouched (the step is undefined)
                if (tid == 0) {
                    double *o = P.res + 6 * sc;
                    o[0] = o[1] = o[2] = __longlong_as_double(0x7ff8000000000000LL);
                    o[3] = 0.0; o[4] = 0.0; o[5] = (double)status0;
                }
                __syncthreads();
                continue;
            }
            // D of the subsystems that the iterations read from shared memory
            if (S.hot_global)
                for (int i = 0; i < S.nsub; ++i) {
                    const SubDesc &u = P.subs[S.sub0 + i];
                    if (u.ot_Dres < 0) continue;
                    const VT *src = reinterpret_cast<const VT *>(V.htb + u.ot_D);
                    VT *dst = reinterpret_cast<VT *>(V.tb + u.ot_Dres);
                    for (int q = tid; q < u.m * u.ldd / VN; q += NT) dst[q] = src[q];
                }
            // initial z, u = -lambda; a learned start (the launch's first step) is checked
            // after 10 iterations against the plain start's residual there, and replaced by
            // the plain start if worse
            const bool learned_mode = P.lam0 != nullptr && step == 0;
            const int skip0 = learned_mode ? P.learn_skip[2 * sc] : 0;
            bool learned = learned_mode && skip0 == 0;
            const unsigned long long ref10 = learned_mode ? P.ref10[sc] : 0ull;
            int wasted = 0, fallbacks = 0;
            __syncthreads();
            if (learned_mode && tid == 0 && skip0 > 0) P.learn_skip[2 * sc] = skip0 - 1;
            init_duals<T>(P, S, V, LAM, Z, ZO, X, Y, YO, W0, BT, learned, BlockDist());

            // ---- per-thread state of the register-cached iteration (CACHED).  The host's
            // thread map gives each thread a side-row (its lane group of SPLIT lanes) and puts
            // every projection item's side-rows on adjacent groups of one warp.  A thread keeps
            // its side-row's D chunks, c, beta, 1/beta, x and the lambda of the last iterations in
            // registers, and the constants of its item: the warp forms x, every lane of an item
            // gets its partner's x (a contact: its rows' lambda) by shuffles and projects its own row
            // (Sec. III-C), so an iteration needs one block barrier (the new w) instead of two.
            // The updates are those of grid_iter.cuh: with d = lambda' - lambda, neither y nor z is
            // formed in the loop (z only for the stop test): 2 x chunks + 6 FP64 instructions per
            // warp and iteration (+ 1 while the stop test fails), each of which holds the FP64 pipe for 64
            // cycles whatever its lanes.  Contacts' two other rows are exchanged only in the warps
            // that hold contacts, chunks beyond the warp's longest row are skipped.
            constexpr int MAXC = cached_chunks(sizeof(T), SPLIT);
            constexpr int FSI = SPLIT == 4 ? 2 : SPLIT == 2 ? 1 : 0;
            const int xg = tid / SPLIT;
            int xt = -1, xgl = tid - xg * SPLIT, flead = 0, fslot = 0, fitem = 0;
            if (CACHED) {
                const int2 fm = reinterpret_cast<const int2 *>(P.ipool + S.fmap_off[FSI])[tid];
                xt = fm.x;
                flead = fm.y & 31;
                fslot = (fm.y >> 5) & 7;
                xgl = (fm.y >> 8) & 7;
                fitem = fm.y >> 11;
            }
            VT dreg[MAXC];
            int woff[MAXC];                // each chunk's vector of w (past the row's end: its first)
            bool xv = false, ftwo = false, wcon = false, wsoft = false;
            int xrow = 0, fr = 0, ftype = 0, fpart = lane, fbase = lane, wch = 0;
            T xc = (T)0, xbt = (T)0, xib = (T)0, xe = (T)0, fa = (T)1, fmul = (T)1, fk = (T)0, fmu = (T)0;
            T xx = (T)0, xprev = (T)0, zreg = (T)0, lreg = (T)0, lreg1 = (T)0, lreg2 = (T)0;
            auto load_cache = [&]() {
                if (CACHED) {
#pragma unroll
                    for (int q = 0; q < MAXC; ++q) { dreg[q] = VecZero<T>::get(); woff[q] = 0; }
                    xv = xt >= 0 && V.mlen[xt] > 0;
                    int ch = 0;
                    if (xv) {
                        const int xnv = (V.mlen[xt] + VN - 1) / VN;
                        ch = (xnv + SPLIT - 1) / SPLIT;
                        xrow = V.row[xt];
                        xc = V.htb[V.coff[xt]];
                        xbt = BT[xt];
                        xib = INVB[xt];
                        xx = X[xt];
                        xprev = xx;
                        zreg = Z[xt];
                        lreg = LAM[xrow];
                        lreg1 = lreg2 = lreg;
                        const VT *Dr = d_row<T>(V, xt);
#pragma unroll
                        for (int q = 0; q < MAXC; ++q) {
                            const int k = xgl + q * SPLIT;
                            woff[q] = V.wbase[xt] / VN + (k < xnv ? k : 0);
                            if (k < xnv) dreg[q] = Dr[k];
                        }
                        const Item it = V.item[fitem];
                        const int nr = it.type == TYPE_CONTACT ? 3 : 1, side = fslot / nr;
                        ftype = it.type;
                        fr = fslot % nr;
                        ftwo = it.ns > 1;
                        fpart = (flead + ((ftwo ? side ^ 1 : side) * nr + fr) * SPLIT + xgl) & 31;
                        fbase = (flead + side * nr * SPLIT) & 31;
                        xe = E[xrow];
                        fmu = MU[xrow];
                        fk = INVS[xrow];
                        fa = fmul = (T)1;
                        if (ftype == TYPE_SOFT) {
                            fa = KF[xrow] * AL[xrow] / fk;
                            fmul = AL[xrow];
                            fk = KF[xrow];
                        }
                        if (sizeof(T) == 8) { fmul *= fk; xe *= fk; }
                    }
                    wch = __reduce_max_sync(0xffffffffu, ch);
                    wcon = __any_sync(0xffffffffu, xv && ftype == TYPE_CONTACT);
                    wsoft = __any_sync(0xffffffffu, xv && ftype == TYPE_SOFT);
                }
            };
            load_cache();
            // the generic variant's iterations with side-rows owned by threads (own_iter.cuh), where no
            // thread owns more than it can keep
            const bool owner = !CACHED && !P.stop_theta && !P.pj && S.max_sides <= 2 && S.nsr <= SUBADMM_OWN * (NT / SPLIT);

            int par = 0, last_par = 0, iters = 0, conv = 0, status = ST_OK;
            bool restart = false;
            double th = 0.0;
            double tolc = P.tol;
            U tolb = tol_bits(T(0), tolc > 0.0 ? tolc : 0.0);
            const bool primal_stop = !P.stop_theta && P.tol > 0.0;
            // FP64: |d| is compared with tol beta (no product); any value above the tolerance
            // stands for a residual that is
            // (blo up to infinity, exclusive: what is not finite is not counted)
            const unsigned long long blo = (unsigned long long)__double_as_longlong(P.tol * (double)xbt) + 1ull;
            const unsigned long long bspan = inf_bits(0.0) - blo;
            const U btol_over = tolb + 1;
            // the loop holds no FP64 instruction in the mixed form, not even a predicated one
            // (an FP64 warp instruction issues for ~64 cycles on GB300 whatever its predicate)
            const int rule = (P.pj ? ITEM_PJ : 0) | (P.stop_theta ? ITEM_THETA : 0) | (primal_stop ? ITEM_TOL : 0) |
                             (P.phase ? ITEM_TRACE : 0);
            // One iteration of this warp's side-rows: x = c + D w over each lane group (past a row's end
            // a zero chunk of D meets the row's own first w: what follows in shared memory may
            // be no number), the projection, the next w; with `stop` (or `all`: whole) the residual's bits
            auto iterate = [&](const VT *wb, T *wnext, bool stop, bool all, bool first) -> U {
                U res = 0;
                T acc = xgl == 0 ? xc : (T)0, a1 = (T)0;
                constexpr int QS = sizeof(T) == 4 ? 2 : 1;     // (FP32: chunks in pairs, fewer branches)
#pragma unroll
                for (int q = 0; q < MAXC; q += QS) {
                    if (q >= wch) break;
                    acc = vdot(dreg[q], wb[woff[q]], acc);
                    if (QS == 2) a1 = vdot(dreg[q + QS - 1], wb[woff[q + QS - 1]], a1);
                }
                if (QS == 2) acc += a1;
#pragma unroll
                for (int o = SPLIT / 2; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                const T xo = __shfl_sync(0xffffffffu, acc, fpart);
                // the item's sum over its sides and its lambda
                const T g = ftwo ? acc + xo : acc;
                T la;
                if (sizeof(T) == 8) la = fa * lreg - (fmul * g + xe);          // (scaled by fk)
                else if (wsoft) la = fa * lreg - (fmul * g + xe) * fk;
                else la = lreg - (g + xe) * fk;
                if (ftype == TYPE_HARD) la = above0(la) ? la : (T)0;
                if (wcon) {
                    const T l0 = __shfl_sync(0xffffffffu, la, fbase);
                    const T l1 = __shfl_sync(0xffffffffu, la, (fbase + SPLIT) & 31);
                    const T l2 = __shfl_sync(0xffffffffu, la, (fbase + 2 * SPLIT) & 31);
                    if (sizeof(T) == 4) {
                        // (no branches: they cost the warp that holds a sliding foot, which the block
                        // waits for, some 140 cycles an iteration; FP64 instructions cost more)
                        const T t2 = l1 * l1 + l2 * l2, lim = fmu * l0;
                        const T f = above0(t2 - lim * lim) ? lim * rsq(t2) : (T)1;
                        const T lc = !above0(l0) ? (T)0 : fr == 0 ? la : la * f;
                        la = ftype == TYPE_CONTACT ? lc : la;
                    } else if (ftype == TYPE_CONTACT) {
                        if (!above0(l0)) {
                            la = (T)0;
                        } else if (fr > 0) {
                            const T t2 = l1 * l1 + l2 * l2, lim = fmu * l0;
                            if (above0(t2 - lim * lim)) la = la * (lim * rsq(t2));
                        }
                    }
                }
                // w of this side-row
                const T y = xbt * acc - lreg;
                if (xv && xgl == 0) wnext[xt] = (T)2 * la + y;
                if (stop || all) {
                    // |x - z| = |d| / beta, and, if no row of the warp is above the tolerance there
                    // (FP64; always in FP32), |z - z of the iteration before|
                    const T dl = la - lreg;
                    bool over = false;
                    if (sizeof(T) == 8 && !all) {
                        over = xv && (unsigned long long)rbits(fabs(dl)) - blo < bspan;
                        if (over) res = btol_over;
                    }
                    if (sizeof(T) == 4 || !__any_sync(0xffffffffu, over)) {
                        const T dz = dl * xib, zn = acc + dz;
                        const T zo = !first ? xx + (lreg - lreg1) * xib : zreg;
                        if (xv && xgl == 0) res = umax(rbits(fabs(dz)), rbits(fabs(zn - zo)));
                    }
                }
                xprev = xx;
                xx = acc;
                lreg2 = lreg1;
                lreg1 = lreg;
                lreg = la;
                return res;
            };
            int l = 0;
            pc.mark(PHASE_ASSEMBLE);
            for (;;) {
                // a fixed iteration count: the same iteration without the tests, two at a time
                if (CACHED && !primal_stop && !learned_mode && !P.phase && l == 0) {
                    const VT *const wa = reinterpret_cast<const VT *>(W0), *const wc = reinterpret_cast<const VT *>(W1);
                    for (; l + 2 <= P.max_iters; l += 2) {
                        iterate(wa, W1, false, false, false);
                        __syncthreads();
                        iterate(wc, W0, false, false, false);
                        __syncthreads();
                    }
                    iters = l;
                    last_par = 1;
                }
                if constexpr (!CACHED) {
                    // (a learned start's iterations up to its check on their own)
                    const bool check = learned_mode && l <= 9 && P.max_iters > 9;
                    const int lend = check ? 10 : P.max_iters;
                    IterResult r;
                    if (!owner)
                        r = item_iterate<T, SPLIT, NT>(s_scene, V.htb, rule, (T)P.pj_omega, (T)P.theta_th, l, lend, par, tolb, check);
                    else if (primal_stop)
                        r = own_iterate<T, SPLIT, NT, true>(s_scene, V.htb, P.ipool + S.own_off, l, lend, P.max_iters, par, tolb, check);
                    else
                        r = own_iterate<T, SPLIT, NT, false>(s_scene, V.htb, P.ipool + S.own_off, l, lend, P.max_iters, par, tolb, check);
                    par = r.par;
                    last_par = r.last_par;
                    iters = r.l;
                    conv = r.conv;
                    if (r.conv && P.stop_theta) th = r.theta;
                    l = r.conv ? r.l - 1 : r.l;
                    pc.mark(PHASE_VSTEP);
                    pc.move(PHASE_VSTEP, PHASE_ZSTEP, r.z_cycles);
                    if (check && !conv) {
                        const U mx = (U)r.mx;
                        l = 9;
                        if (learned && r.mx > ref10) restart = true;
                        else {
                            if (!learned && tid == 0) P.ref10[sc] = r.mx;
                            if (learned && tid == 0) P.learn_skip[2 * sc + 1] = 0;     // kept: streak ends
                            if (mx >= inf_bits(T(0))) status = ST_NAN;
                            else if (primal_stop && mx <= tolb) conv = 1;
                            else { l = 10; if (l < P.max_iters) continue; }
                        }
                    }
                }
                for (; CACHED && l < P.max_iters; ++l) {
                    // x = c + D w, the projection and the next w (iterate, above)
                    const U mloc = iterate(reinterpret_cast<const VT *>(par ? W1 : W0), par ? W0 : W1, primal_stop,
                                           learned_mode && l == 9, l == 0);
                    pc.mark(PHASE_VSTEP);
                    last_par = par;
                    iters = l + 1;
                    if (!(learned_mode && l == 9)) {
                        // the stop test rides on the barrier: the number of threads whose
                        // residual is finite and above the tolerance.  A non-finite iterate
                        // stays non-finite (c is fixed for the step and w carries it to every
                        // coupled side-row), so the count drops to 0 or the limit ends the
                        // loop, and the step's FP64 residuals below report it
                        int over = 0;
                        if (primal_stop) over = __syncthreads_count(mloc > tolb && mloc < inf_bits(T(0)));
                        else __syncthreads();
                        par ^= 1;
                        pc.mark(PHASE_ZSTEP);
                        if (primal_stop && over == 0) { conv = 1; break; }
                        continue;
                    }
                    const U wmax = warp_umax(mloc);
                    if (lane == 0) ured[warp] = wmax;
                    __syncthreads();
                    U mx = 0;
#pragma unroll
                    for (int q = 0; q < NW; ++q) mx = umax(mx, ured[q]);
                    par ^= 1;
                    pc.mark(PHASE_ZSTEP);
                    if (learned && (unsigned long long)mx > ref10) { restart = true; break; }
                    if (!learned && tid == 0) P.ref10[sc] = (unsigned long long)mx;
                    if (learned && tid == 0) P.learn_skip[2 * sc + 1] = 0;       // kept: streak ends
                    if (mx >= inf_bits(T(0))) { status = ST_NAN; break; }
                    if (primal_stop && mx <= tolb) { conv = 1; break; }
                }
                if (restart) {
                    // the learned start trails the plain one after 10 iterations: restart the
                    // step from the plain start, and start plain for the next 2^streak - 1 steps
                    if (tid == 0) {
                        const int streak = min(P.learn_skip[2 * sc + 1] + 1, 5);
                        P.learn_skip[2 * sc + 1] = streak;
                        P.learn_skip[2 * sc] = (1 << streak) - 1;
                    }
                    restart = false;
                    learned = false;
                    ++fallbacks;
                    wasted += l + 1;
                    init_duals<T>(P, S, V, LAM, Z, ZO, X, Y, YO, W0, BT, false, BlockDist());
                    load_cache();
                    par = 0;
                    l = 0;
                    continue;
                }
                // the register-cached iterate: publish x, y, z, lambda and the previous y, z (after a
                // single iteration those are the initial ones, which init_duals left there)
                if (CACHED && xv && xgl == 0) {
                    X[xt] = xx;
                    Y[xt] = xbt * xx - lreg1;
                    Z[xt] = xx + (lreg - lreg1) * xib;
                    if (iters > 1) {
                        YO[xt] = xbt * xprev - lreg2;
                        ZO[xt] = xprev + (lreg1 - lreg2) * xib;
                    }
                    LAM[xrow] = lreg;
                }
                __syncthreads();
                // v-hat from the last v-step's w (ADMM), or from the last z-step's lambda
                // (Projected Jacobi: v-hat = A^-1 (b + J^T lambda) with the reported impulses)
                block_recover<T>(P, S, V, (P.pj ? par : last_par) ? W1 : W0);
                __syncthreads();
                if (MIXED && conv && primal_stop && status == ST_OK) {
                    // FP64 primal residual max |J v - z|; on a miss, refine c by the FP64 - FP32
                    // difference of x at this iterate and resume
                    double part = 0.0;
                    for (int t = tid; t < S.nsr; t += blockDim.x) {
                        if (V.mlen[t] == 0) continue;
                        const SubDesc &u = P.subs[S.sub0 + V.sub[t]];
                        const int lr = t - u.sr0, n = u.n;
                        const double *Jr = V.sdb + u.od_J + lr * n;
                        const double *v = V.sdb + u.od_v;
                        const int *jl = P.ipool + u.env_off + 2 * n;
                        double x = 0.0;
                        for (int p = jl[lr]; p < jl[u.m + lr]; ++p) x += Jr[p] * v[p];
                        part = nanmax(part, fabs(x - (double)Z[t]));
                        V.htb[V.coff[t]] += (T)(x - (double)X[t]);
                    }
                    double d0 = 0.0, d2 = 0.0;
                    block_reduce3(red, d0, part, d2);
                    if (part > P.tol && l + 1 < P.max_iters) {
                        tolc *= 0.5;
                        tolb = tol_bits(T(0), tolc);
                        if (CACHED && xv) { xc = V.htb[V.coff[xt]]; zreg = Z[xt]; }
                        conv = 0;
                        ++l;
                        continue;
                    }
                    if (part > P.tol) conv = 0;
                }
                break;
            }
            // reported residuals of the last iteration: theta, r_p = max|x - z|,
            // r_d = max beta |z^{l+1} - z^l|
            double rp, rd;
            {
                double tp = 0.0, pp = 0.0, dd = 0.0;
                for (int t = tid; t < S.nsr; t += blockDim.x) {
                    if (V.mlen[t] == 0) continue;
                    const double dy = (double)Y[t] - (double)YO[t];
                    tp += dy * dy;
                    pp = nanmax(pp, fabs((double)X[t] - (double)Z[t]));
                    dd = nanmax(dd, (double)BT[t] * fabs((double)Z[t] - (double)ZO[t]));
                }
                block_reduce3(red, tp, pp, dd);
                if (!P.stop_theta) th = tp;
                rp = pp;
                rd = dd;
            }
            // a non-finite iterate (the loop itself does not stop on one)
            if (status == ST_OK && !(isfinite(rp) && isfinite(rd))) { status = ST_NAN; conv = 0; }
            pc.mark(PHASE_EXIT);
            // v-hat out and state update of rigid bodies (Algorithm 1, after the loop)
            for (int i = warp; i < S.nsub; i += NW) {
                const SubDesc &u = P.subs[S.sub0 + i];
                const double *v = V.sdb + u.od_v;
                for (int p = lane; p < u.n; p += 32) P.vhat[u.v_off + p] = v[p];
                if (u.kind == KIND_LINEAR) {
                    double *nd = P.nodes + (size_t)u.body0 * SUBADMM_NODE;
                    for (int p = lane; p < u.n; p += 32) {
                        nd[(p / 3) * SUBADMM_NODE + p % 3] += P.h * v[p];
                        double &vel = nd[(p / 3) * SUBADMM_NODE + 3 + p % 3];
                        vel = 2.0 * v[p] - vel;
                    }
                    continue;
                }
                if (u.kind != KIND_RIGID) continue;
                for (int k = lane; k < u.nb; k += 32)
                    body_update(P.bodies + (size_t)(u.body0 + k) * SUBADMM_BODY, v + 6 * k, P.h);
            }
            __syncthreads();
            pc.mark(PHASE_RECOVER);
            pc.flush(iters);
            // warm-start state and reports
            for (int r = tid; r < S.nrow; r += blockDim.x) P.lam[S.row_g0 + r] = (double)LAM[r];
            for (int t = tid; t < S.nsr; t += blockDim.x) P.z[S.sr_g0 + t] = (double)Z[t];
            if (tid == 0) {
                double *o = P.res + 6 * sc;
                o[0] = rp; o[1] = rd; o[2] = th; o[3] = (double)iters; o[4] = (double)conv;
                o[5] = (double)status;
                long long *st = P.stats + 5 * sc;
                st[0] += iters + wasted;
                if (iters + wasted > st[1]) st[1] = iters + wasted;
                st[2] += conv ? 0 : 1;
                st[3] += 1;
                st[4] += fallbacks;
            }
            __syncthreads();
        }
    }
}

}  // namespace subadmm
