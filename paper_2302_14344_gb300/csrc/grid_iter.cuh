// One scene over the whole GPU, with one grid barrier per iteration.
//
// A step is two cooperative launches: grid_setup_kernel (assembly, beta, factors, the map D
// and c: scene_setup over the grid) and grid_iter_kernel (the ADMM loop, the recovery of
// v-hat, the state update).  The v-step x = c + D w needs the w of its own subsystem only, and
// a projection item needs the x of its own side-rows only; so a warp that holds all side-rows
// of its items (a wave: at most one side-row per lane, laid out by the host) forms their x,
// projects them and writes their next w without leaving the warp.  Only w crosses the chip:
// one barrier per iteration, where separate v- and z-steps took two and passed y, x, z and
// lambda through L2 (grid_kernel.cuh, which stays for the theta stop rule and for scenes with
// more side-rows than the grid has lanes).  Everything else of a side-row stays in its lane's
// registers for the step.
//
// With d = lambda' - lambda of the row, the updates of Sec. III-C need no y and no z:
//   equality  d = -(sum_s x_s + e) / sum 1/beta      (hard rows and contacts clamp lambda + d)
//   soft      lambda' = -k_f (e + alpha (sum_s x_s - s lambda))
//   z = x + d / beta,   next w = beta x + lambda' + d,   x - z = -d / beta
// which is fewer instructions (FP64 ones cost an issue slot of 64 cycles) and no cancellation
// of y against lambda.  z itself is formed only for the stop test and for the last iterates.
//
// Two kernels.  LONG = false (small subsystems): a wave is at most 8 rows of one vector per lane
// (shape A) or 3 wide rows of one subsystem and 3 narrow ones (shape B), its D rows stay in
// shared memory for the step, and with a fixed iteration count (no stop test to agree on) there
// is no barrier at all: every w carries the number of its iteration in the same 8-byte word
// (two words in FP64), and a warp waits for the words of its own subsystems.  That is one
// store-to-load trip through L2 where a barrier takes three (the store's fence, the arrival, the
// poll) before the load.  A slot of the two alternating buffers is written again two
// iterations later; its writer has by then read the w that each of its readers wrote after
// reading it.  LONG = true (the large beam): a warp keeps as many rows as fit in its share of
// the block's shared memory (33 MB over the chip) and streams the others through registers, a
// row ahead, the first one across the barrier; the barrier's time prefetches the next rows
// into L2 (without it 64 slabs take 23.2 us an iteration instead of 17.9).  Bound by the
// stream, some 90 MB an iteration from L2 and, for what L2 does not keep, HBM.
#pragma once

#include "grid_kernel.cuh"

namespace subadmm {

// Barrier over the blocks of the iteration kernel: round r uses counter r % 2 (zeroed before
// the step), whose low half counts arrivals and whose high half sums the blocks' flags; a block
// that reads it after its round is complete sees no arrival of round r + 2, because that needs
// its own arrival in round r + 1.  The wait is bounded like grid_barrier's.
struct IterBarrier {           // in shared memory; thread 0 alone uses what is not constant
    unsigned long long *bar;
    int *err;
    unsigned expected, round;
    unsigned seen[2];          // flags of each counter's earlier rounds
    unsigned over;             // of the last round: blocks that raised their flag
    int dead;                  // a wait ran out, here or elsewhere: no more waits

    __device__ __forceinline__ void init(GridScratch *G)
    {
        bar = G->bar;
        err = &G->err;
        expected = gridDim.x;
        round = seen[0] = seen[1] = over = 0u;
        dead = 0;
    }
    __device__ __noinline__ void wait(unsigned flag)
    {
        const unsigned r = round++;
        unsigned long long *b = bar + (r & 1);
        const unsigned target = (r / 2 + 1) * expected;
        volatile int *verr = err;
        over = 0;
        if (dead) return;
        __threadfence();
        unsigned long long v = atomicAdd(b, 1ull + ((unsigned long long)flag << 32)) + 1ull +
                               ((unsigned long long)flag << 32);
        if ((int)((unsigned)v - target) < 0) {
            const unsigned long long t0 = global_ns();
            for (unsigned k = 1;; ++k) {
                asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(b) : "memory");
                if ((int)((unsigned)v - target) >= 0) break;
                if (k % 64 == 0) {
                    if (*verr) { dead = 1; break; }
                    if (global_ns() - t0 > 20000000000ull) { atomicExch(err, 1); dead = 1; break; }
                    if (k >= 4096) __nanosleep(64);
                }
            }
        }
        __threadfence();
        over = (unsigned)(v >> 32) - seen[r & 1];
        seen[r & 1] = (unsigned)(v >> 32);
    }
    __device__ __forceinline__ unsigned sync(unsigned flag)
    {
        __syncthreads();
        if (threadIdx.x == 0) wait(flag);
        __syncthreads();
        return over;
    }
};

// the iteration kernel's work distribution (see BlockDist, GridDist)
struct IterDist {
    static constexpr bool kSpread = false, kBig = true;
    static constexpr int kThreads = SUBADMM_ITER;
    int tid, nthreads, warp, nwarps;
    IterBarrier *bar;
    __device__ __forceinline__ IterDist(IterBarrier *b)
        : tid(blockIdx.x * blockDim.x + threadIdx.x), nthreads(gridDim.x * blockDim.x),
          warp((int)(threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x),
          nwarps((gridDim.x * blockDim.x) >> 5), bar(b) {}
    __device__ __forceinline__ void sync() const { bar->sync(0); }
    __device__ __forceinline__ void fence() const { __threadfence(); }
};

// The setup of one step over the grid (tc_phase 0 or 1: scene_setup; 3: W of the subsystems
// that the blocked factorisation factorised in between)
template <typename T>
__global__ void __launch_bounds__(SUBADMM_THREADS, 2) grid_setup_kernel(StepParams P)
{
    GridScratch *G = P.grid;
    const GridDist d(&G->count, &G->gen, &G->err);
    const int sc = P.scene_ids[0];
    const SceneDesc S = P.scenes[sc];
    const View<T> V = scene_view<T>(P, S, reinterpret_cast<unsigned char *>(P.work) + S.g_scene);
    extern __shared__ __align__(128) unsigned char smem[];
    if (d.tid == 0 && P.tc_phase != 3) {
        // (nobody sets the status before scene_setup's barriers; the rest is the iteration
        // kernel's, which is not running)
        G->status = ST_OK;
        G->tsum = 0.0;
        G->pmax = G->dmax = G->chk = 0ull;
        for (int k = 0; k < 3; ++k) G->umax[k] = 0ull;
        G->bar[0] = G->bar[1] = 0ull;
    }
    if (P.tables) {
        for (int q = d.tid; q < S.ot_lam - S.ot_x; q += d.nthreads) V.tb[S.ot_x + q] = (T)0;
        scene_tables<T>(P, S, V, d);
        d.sync();
    }
    PhaseClock pc((P.phase && blockIdx.x == 0) ? P.phase + 8 * sc : nullptr);
    if (P.tc_phase == 3) w_chunks<T>(P, S, V, &G->status, d, 4);
    else pc.mark_at(PHASE_ASSEMBLE, scene_setup<T>(P, S, V, &G->status, 0, d, P.grid_big ? smem : nullptr));
    pc.mark(PHASE_FACTOR);
    pc.flush(0, 0);
}

template <typename T>
__device__ __noinline__ void iter_recover(const StepParams &P, const SceneDesc &S, const View<T> &V, const T *w,
                                          IterBarrier *bar, unsigned char *big_smem)
{
    recover_v<T>(P, S, V, w, IterDist(bar), (T *)nullptr, 0, big_smem);
}

// Sums of 8 values over the warp: value r's sum ends on lanes 4 r .. 4 r + 3 (10 shuffles and 9
// additions in place of 40 of each)
template <typename T>
__device__ __forceinline__ T reduce8(T *a)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 4; h; h >>= 1) {
        const bool up = lane & (4 * h);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < h) {
                const T send = up ? a[i] : a[i + h], keep = up ? a[i + h] : a[i];
                a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * h);
            }
    }
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
    return a[0];
}

// One w of the tagged exchange: value and tag in one 64-bit word (FP32), or the value's halves in
// two (FP64), and a vector's worth of them (32 bytes) read at once.  Each 64-bit element of an
// access is read and written whole, so a tag never comes without its value.
__device__ __forceinline__ void tag_store(void *p, float v, unsigned tag)
{
    asm volatile("{\n\t.reg .b64 a;\n\tmov.b64 a, {%1, %2};\n\tst.relaxed.gpu.global.b64 [%0], a;\n\t}"
                 ::"l"(p), "r"(__float_as_uint(v)), "r"(tag) : "memory");
}
__device__ __forceinline__ void tag_store(void *p, double v, unsigned tag)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    asm volatile("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %2};\n\t"
                 "st.relaxed.gpu.global.v2.b64 [%0], {a, b};\n\t}"
                 ::"l"(p), "r"((unsigned)b), "r"(tag), "r"((unsigned)(b >> 32)) : "memory");
}
struct TagVec { uint4 a, b; };
__device__ __forceinline__ uint4 tag_load2(const void *p)
{
    uint4 v;
    asm volatile("{\n\t.reg .b64 a, b;\n\tld.relaxed.gpu.global.v2.b64 {a, b}, [%4];\n\t"
                 "mov.b64 {%0, %1}, a;\n\tmov.b64 {%2, %3}, b;\n\t}"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ TagVec tag_load(const void *p)
{
    return TagVec{tag_load2(p), tag_load2((const char *)p + 16)};
}
// every word is of iteration `tag`, or padding (no owner; the host sets its tag to ~0)
__device__ __forceinline__ bool tag_ready(const TagVec &v, unsigned tag)
{
    return (v.a.y == tag || v.a.y == ~0u) && (v.a.w == tag || v.a.w == ~0u) &&
           (v.b.y == tag || v.b.y == ~0u) && (v.b.w == tag || v.b.w == ~0u);
}
__device__ __forceinline__ float4 tag_value(const TagVec &v, float4)
{
    return make_float4(__uint_as_float(v.a.x), __uint_as_float(v.a.z), __uint_as_float(v.b.x), __uint_as_float(v.b.z));
}
__device__ __forceinline__ double2 tag_value(const TagVec &v, double2)
{
    return make_double2(__longlong_as_double((long long)(((unsigned long long)v.a.z << 32) | v.a.x)),
                        __longlong_as_double((long long)(((unsigned long long)v.b.z << 32) | v.b.x)));
}

// A vector of a streamed D row.  A row is read once per iteration: kept out of L1, it leaves the
// 27 KB beside the D rows in shared memory to w, which every batch of rows reads (64 slabs of 686
// side-rows, FP32: 22.7 -> 17.9 us an iteration).
__device__ __forceinline__ float4 load_stream(const float4 *p)
{
    float4 v;
    asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ double2 load_stream(const double2 *p)
{
    double2 v;
    asm volatile("ld.global.L1::no_allocate.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p) : "memory");
    return v;
}

// Phase tracer of the iteration kernel (see PhaseClock): in shared memory, thread 0
struct IterClock {
    long long t, a[8];
    __device__ __forceinline__ void mark(const long long *out, int phase)
    {
        if (threadIdx.x != 0 || !out) return;
        const long long n = clock64();
        a[phase] += n - t;
        t = n;
    }
};

// residuals, state update and reports of a step (cold: kept out of the loop's registers)
template <typename T>
__device__ __noinline__ void iter_finish(const StepParams &P, const SceneDesc &S, const View<T> &V, IterBarrier *bar,
                                         IterClock *pc, long long *trace, int iters, int conv, int status,
                                         int wasted, int fallbacks)
{
    const IterDist d(bar);
    const int lane = threadIdx.x & 31, sc = P.scene_ids[0];
    GridScratch *G = P.grid;
    const T *X = V.tb + S.ot_x, *Y = V.tb + S.ot_y, *Z = V.tb + S.ot_z, *LAM = V.tb + S.ot_lam;
    const T *YO = V.tb + S.ot_yo, *ZO = V.tb + S.ot_zo, *BT = V.tb + S.ot_b;
    // reported residuals of the last iteration: theta, r_p = max|x - z|, r_d = max beta |dz|
    {
        double tp = 0.0, pp = 0.0, dd = 0.0;
        for (int t = d.tid; t < S.nsr; t += d.nthreads) {
            if (V.mlen[t] == 0) continue;
            const double dy = (double)Y[t] - (double)YO[t];
            tp += dy * dy;
            pp = nanmax(pp, fabs((double)X[t] - (double)Z[t]));
            dd = nanmax(dd, (double)BT[t] * fabs((double)Z[t] - (double)ZO[t]));
        }
        tp = warp_sum(tp);
        pp = warp_max(pp);
        dd = warp_max(dd);
        if (lane == 0) {
            if (tp != 0.0) atomicAdd(&G->tsum, tp);
            if (pp > 0.0 || pp != pp) atomicMax(&G->pmax, dbits(fabs(pp)));
            if (dd > 0.0 || dd != dd) atomicMax(&G->dmax, dbits(fabs(dd)));
        }
    }
    pc->mark(trace, PHASE_EXIT);
    // v-hat out and state update (Algorithm 1, after the loop)
    for (int i = d.warp; i < S.nsub; i += d.nwarps) {
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
    // warm-start state and reports
    for (int r = d.tid; r < S.nrow; r += d.nthreads) P.lam[S.row_g0 + r] = (double)LAM[r];
    for (int t = d.tid; t < S.nsr; t += d.nthreads) P.z[S.sr_g0 + t] = (double)Z[t];
    d.sync();
    pc->mark(trace, PHASE_RECOVER);
    if (trace && threadIdx.x == 0) {
        pc->a[PHASE_ITERS] = iters;
        pc->a[PHASE_STEPS] = 1;
        for (int q = 0; q < 8; ++q) trace[q] += pc->a[q];
    }
    if (d.tid == 0) {
        const double rp = __longlong_as_double((long long)vload(&G->pmax));
        const double rd = __longlong_as_double((long long)vload(&G->dmax));
        if (status == ST_OK && !(isfinite(rp) && isfinite(rd))) { status = ST_NAN; conv = 0; }
        if (vload(&G->err)) status = ST_TIMEOUT;
        double *o = P.res + 6 * sc;
        o[0] = rp; o[1] = rd; o[2] = vload(&G->tsum); o[3] = (double)iters; o[4] = (double)conv;
        o[5] = (double)status;
        long long *st = P.stats + 5 * sc;
        st[0] += iters + wasted;
        if (iters + wasted > st[1]) st[1] = iters + wasted;
        st[2] += conv ? 0 : 1;
        st[3] += 1;
        st[4] += fallbacks;
    }
}

template <typename T>
__device__ __noinline__ void iter_duals(const StepParams &P, const SceneDesc &S, const View<T> &V, IterBarrier *bar,
                                        bool learned)
{
    init_duals<T>(P, S, V, V.tb + S.ot_lam, V.tb + S.ot_z, V.tb + S.ot_zo, V.tb + S.ot_x, V.tb + S.ot_y,
                  V.tb + S.ot_yo, V.tb + S.ot_w0, V.tb + S.ot_b, learned, IterDist(bar));
}

template <typename T, bool LONG>
__global__ void __launch_bounds__(SUBADMM_ITER, 1) grid_iter_kernel(const __grid_constant__ StepParams P)
{
    using VT = typename VecOf<T>::V;
    using U = typename VecOf<T>::U;
    constexpr int VN = VecOf<T>::N;
    constexpr bool MIXED = sizeof(T) == 4;
    // vectors of a row per lane and segment (LONG): a row ahead of FP32 for the latency of its
    // stream (3 in place of 6: 17.9 -> 21.5 us an iteration of 64 slabs); in FP64 the three buffers
    // of 6 did not fit the registers, and 3 still cover the pipe (v-step of 16 slabs 72k -> 47k cycles,
    // the iteration 77k -> 51k)
    constexpr int CH = MIXED ? 6 : 3;
    constexpr int RV = kWideVecs<T>();             // vectors per lane of a wide row (shape B)
    static_assert(RV <= 4, "a wide row's w is gathered at once");
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(128) unsigned char smem[];
    // (what the loop does not use lives in shared memory, to spill less: 512 threads' frames do not
    // fit L1 next to the D rows.  What is left, by -Xptxas -v: some 580 bytes of spill stores a
    // thread in FP32 without LONG, 440 with, 190 and 110 in FP64; with 860-byte frames in the
    // loop a stir iteration took 13k cycles, now 8.4k)
    __shared__ SceneDesc S;
    __shared__ View<T> V;
    __shared__ IterBarrier bar;
    __shared__ IterClock pc;
    __shared__ unsigned long long s_umax[SUBADMM_ITER / 32];
    __shared__ int s_nan;
    GridScratch *G = P.grid;
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int sc = P.scene_ids[0];
    long long *const trace = P.phase && blockIdx.x == 0 ? P.phase + 8 * sc : nullptr;
    for (int q = threadIdx.x; q < (int)(sizeof(SceneDesc) / 4); q += SUBADMM_ITER)
        reinterpret_cast<int *>(&S)[q] = reinterpret_cast<const int *>(P.scenes + sc)[q];
    if (threadIdx.x == 0) {
        bar.init(G);
        s_nan = 0;
        pc.t = clock64();
        for (int q = 0; q < 8; ++q) pc.a[q] = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) V = scene_view<T>(P, S, reinterpret_cast<unsigned char *>(P.work) + S.g_scene);
    __syncthreads();
    const IterDist d(&bar);
    const bool lead = d.tid == 0;
    if (lead) G->count = 0u;                       // the setup's barrier, for the next step
    const int status0 = G->status;
    if (status0 != ST_OK) {                        // (uniform over the grid: no barrier waits)
        if (lead) {
            double *o = P.res + 6 * sc;
            o[0] = o[1] = o[2] = __longlong_as_double(0x7ff8000000000000LL);
            o[3] = 0.0; o[4] = 0.0; o[5] = (double)status0;
        }
        return;
    }
    // ---- this warp's wave: the lane's side-row and its item's constants
    const int slot = blockIdx.x * P.wave_per_block + wl;
    const bool has = wl < P.wave_per_block && slot < P.nwaves;
    WaveHead hd{0u, 0, 0, 0};
    WaveLane ln{-1, 1 << 5, lane, 0};
    if (has) {
        hd = P.wave_head[slot];
        ln = P.wave_lane[32 * slot + lane];
    }
    const int myt = ln.t;
    const bool own = myt >= 0;
    // lambda' = fa lambda - (fm sum_s x_s + e) fk before clamping (see above; soft rows: fm =
    // alpha, fk = k_f, fa = k_f alpha s; Projected Jacobi: relaxed by omega)
    T bt = (T)0, ib = (T)0, e = (T)0, fa = (T)1, fm = (T)1, fk = (T)0, mu = (T)0, c = (T)0;
    int r_len = 0, r_drow = 0, r_wb = 0;
    if (own) {
        const int row = V.row[myt];
        bt = (V.tb + S.ot_b)[myt];
        ib = (V.tb + S.ot_invb)[myt];
        e = (V.tb + S.ot_e)[row];
        mu = (V.tb + S.ot_mu)[row];
        c = V.htb[V.coff[myt]];
        const T is = (V.tb + S.ot_invs)[row], kf = (V.tb + S.ot_kf)[row], al = (V.tb + S.ot_al)[row];
        const T om = P.pj ? (T)P.pj_omega : (T)1;
        fk = om * is;
        if ((ln.meta & 3) == TYPE_SOFT) {
            fm = al;
            fk = om * kf;
            fa = kf * al / is;
            if (P.pj) fa = (T)1 - om + om * fa;
        }
        r_len = V.mlen[myt]; r_drow = V.drow[myt]; r_wb = V.wbase[myt];
    }
    // ---- D rows kept for the step in the warp's share of shared memory: all of them, a vector per
    // lane and slot (slots: row r, or RV per wide row and then one per narrow row), or the wave's
    // first rows (LONG)
    unsigned char *const share = smem + (size_t)wl * P.wave_smem;
    VT *const Ds = reinterpret_cast<VT *>(share) + lane;
    int wo[LONG ? 1 : 8];                          // each row's vector of w (shape B: RV of the wide
                                                   // rows, from 4 on one per narrow row)
    int r_res = -1;                                // LONG: offset of this lane's row in the share
    const bool wide = hd.flags & 1;
    auto load_rows = [&]() {
        if constexpr (!LONG) {
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int len = __shfl_sync(FULL, r_len, r), nv = (len + VN - 1) / VN, dr = __shfl_sync(FULL, r_drow, r);
                const int wb = __shfl_sync(FULL, r_wb, r) / VN;
                const VT *src = reinterpret_cast<const VT *>(V.htb + dr);
                if (wide && r < 3) {
#pragma unroll
                    for (int q = 0; q < RV; ++q) {
                        const bool in = lane + 32 * q < nv;
                        Ds[32 * (RV * r + q)] = in ? src[lane + 32 * q] : VecZero<T>::get();
                        if (r == 0) wo[q] = wb + (in ? lane + 32 * q : 0);
                    }
                } else if (!wide || r < 6) {
                    const bool in = lane < nv;
                    Ds[32 * (wide ? 3 * RV + r - 3 : r)] = in ? src[lane] : VecZero<T>::get();
                    const int o = wb + (in ? lane : 0);
                    if (!wide) wo[r] = o;
                    else if (r >= 3) wo[4 + r - 3] = o;
                }
            }
        } else {
            int off = 0;
            for (int k = 0; k < hd.nrows; ++k) {
                const int nv = (__shfl_sync(FULL, r_len, k) + VN - 1) / VN, dr = __shfl_sync(FULL, r_drow, k);
                if (off + nv * 16 > P.wave_smem) break;
                const VT *src = reinterpret_cast<const VT *>(V.htb + dr);
                VT *dst = reinterpret_cast<VT *>(share + off);
                for (int q = lane; q < nv; q += 32) dst[q] = src[q];
                if (lane == k) r_res = off;
                off += nv * 16;
            }
        }
        __syncwarp();
    };
    load_rows();
    // initial z, u = -lambda; a learned start is checked after 10 iterations against the plain
    // start's residual there, and replaced by the plain start if worse
    const bool learned_mode = P.lam0 != nullptr;
    bool learned = learned_mode;
    int fallbacks = 0, wasted = 0;
    if (learned_mode) {
        const int skip0 = vload(&P.learn_skip[2 * sc]);
        learned = skip0 == 0;
        d.sync();                                  // every block has read it
        if (lead && skip0 > 0) P.learn_skip[2 * sc] = skip0 - 1;
    }
    iter_duals<T>(P, S, V, &bar, learned);
    // x, lambda and z of the last iterations (lam1, lam2: one and two iterations ago)
    T x = (T)0, xp = (T)0, lam = (T)0, lam1 = (T)0, lam2 = (T)0, z = (T)0;
    auto load_duals = [&]() {
        lam = own ? (V.tb + S.ot_lam)[V.row[myt]] : (T)0;
        lam1 = lam2 = lam;
        z = own ? (V.tb + S.ot_z)[myt] : (T)0;
    };
    load_duals();
    VT cur[LONG ? CH : 1];                         // LONG: the row (or its segment) that is used next
    auto fetch = [&](VT *dst, const VT *row, int nv, int seg) {
#pragma unroll
        for (int q = 0; q < CH; ++q) {
            const int k = (seg * CH + q) * 32 + lane;
            dst[q] = k < nv ? row[k] : VecZero<T>::get();
        }
    };
    auto fetch_row = [&](VT *dst, int r, int nv, int seg) {       // D row of lane r's side-row
        const int res = __shfl_sync(FULL, r_res, r), dr = __shfl_sync(FULL, r_drow, r);
        if (res >= 0) {
            fetch(dst, reinterpret_cast<const VT *>(share + res), nv, seg);
            return;
        }
        const VT *row = reinterpret_cast<const VT *>(V.htb + dr);
#pragma unroll
        for (int q = 0; q < CH; ++q) {
            const int k = (seg * CH + q) * 32 + lane;
            dst[q] = VecZero<T>::get();
            if (k < nv) dst[q] = load_stream(row + k);
        }
    };
    auto fetch_first = [&]() {
        if constexpr (LONG)
            if (hd.nrows > 0) fetch_row(cur, 0, (__shfl_sync(FULL, r_len, 0) + VN - 1) / VN, 0);
    };
    fetch_first();
    // the tagged exchange: this launch's tags follow the last launch's (the count of iterations
    // so far is kept with the buffers, so that a replayed launch does not find its old tags)
    const bool tagged = !LONG && P.wave_tag != nullptr;
    unsigned char *const tw = reinterpret_cast<unsigned char *>(P.wave_tag) + 16;
    const unsigned tag0 = tagged ? *P.wave_tag : 0u;
    const unsigned tstride = (unsigned)S.nsr * 2u * (unsigned)sizeof(T);
    bool tag_dead = false;
    if (tagged) {
        d.sync();                                  // every block has read the count
        if (own) tag_store(tw + (size_t)myt * 2 * sizeof(T), (V.tb + S.ot_w0)[myt], tag0);
        if (lead) *P.wave_tag = (tag0 + (unsigned)P.max_iters + 1u) & 0x7fffffffu;
    }

    int conv = 0, status = ST_OK, iters = 0;
    double tolc = P.tol;
    const bool primal_stop = P.tol > 0.0;
    int l = 0;
    int par = 0;                                   // w of iteration l in W1 if set, else in W0
    pc.mark(trace, PHASE_ASSEMBLE);
    for (;;) {
        bool restart = false;
        const U tolb = tol_bits(T(0), tolc > 0.0 ? tolc : 0.0);
        for (; l < P.max_iters; ++l) {
            // ---- v-step through the affine map: x = c + D w of the wave's side-rows
            T dot = (T)0;
            if constexpr (!LONG) {
                // up to four vectors of w (those in `want`) at once, waited for if tagged
                auto gather = [&](const int *o, unsigned want, VT *out) {
                    if (!tagged) {
                        const VT *wv = reinterpret_cast<const VT *>(V.tb + (par ? S.ot_w1 : S.ot_w0));
#pragma unroll
                        for (int q = 0; q < 4; ++q) out[q] = want >> q & 1 ? wv[o[q]] : VecZero<T>::get();
                        return;
                    }
                    const unsigned tag = (tag0 + (unsigned)l) & 0x7fffffffu;
                    const unsigned char *src = tw + (l & 1) * tstride;
                    unsigned long long t0 = 0;
                    for (unsigned spin = 0;; ++spin) {
                        bool ok = true;
                        TagVec tv[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (want >> q & 1) tv[q] = tag_load(src + (size_t)o[q] * 32);
                            else tv[q].a = tv[q].b = make_uint4(0u, tag, 0u, tag);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            ok = ok && tag_ready(tv[q], tag);
                            out[q] = tag_value(tv[q], VT());
                        }
                        if (__all_sync(FULL, ok) || tag_dead) break;
                        if (spin % 256 == 255) {   // bounded: 2 s, or an error elsewhere
                            const unsigned long long now = global_ns();
                            if (t0 == 0) t0 = now;
                            bool out_of_time = now - t0 > 2000000000ull;
                            if (out_of_time && lane == 0) atomicExch(&G->err, 1);
                            tag_dead = __any_sync(FULL, out_of_time || vload(&G->err));
                        }
                    }
                };
                T acc[8];
#pragma unroll
                for (int r = 0; r < 8; ++r) acc[r] = (T)0;
                VT wr[4], cw = VecZero<T>::get();
                if (wide) {
                    // 3 wide rows of one subsystem, RV vectors of w, then 3 narrow rows
                    gather(wo, (1u << RV) - 1u, wr);
#pragma unroll
                    for (int r = 0; r < 3; ++r)
#pragma unroll
                        for (int q = 0; q < RV; ++q) acc[r] = vdot(Ds[32 * (RV * r + q)], wr[q], acc[r]);
                    if (hd.nrows > 3) {
                        gather(wo + 4, hd.starts >> 3 & 7u, wr);
#pragma unroll
                        for (int r = 0; r < 3; ++r) {
                            if (hd.starts >> (3 + r) & 1) cw = wr[r];
                            acc[3 + r] = vdot(Ds[32 * (3 * RV + r)], cw, (T)0);
                        }
                    }
                } else {
#pragma unroll
                    for (int h = 0; h < 8; h += 4) {
                        if (h && hd.nrows <= h) break;
                        gather(wo + h, hd.starts >> h & 15u, wr);
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            if (hd.starts >> (h + r) & 1) cw = wr[r];
                            acc[h + r] = vdot(Ds[32 * (h + r)], cw, (T)0);
                        }
                    }
                }
                const T s = reduce8(acc);
                dot = __shfl_sync(FULL, s, (lane << 2) & 31);
            } else {
                const T *w = V.tb + (par ? S.ot_w1 : S.ot_w0);
                for (unsigned left = hd.starts; left; left &= left - 1) {
                    const int k0 = __ffs(left) - 1;
                    const unsigned rest = left & (left - 1);
                    const int cnt = (rest ? __ffs(rest) - 1 : hd.nrows) - k0;
                    const int nv = (__shfl_sync(FULL, r_len, k0) + VN - 1) / VN;
                    const VT *wv = reinterpret_cast<const VT *>(w + __shfl_sync(FULL, r_wb, k0));
                    const int segs = (nv + 32 * CH - 1) / (32 * CH);
                    T acc[8];
#pragma unroll
                    for (int r = 0; r < 8; ++r) acc[r] = (T)0;
                    for (int seg = 0; seg < segs; ++seg) {
                        VT wr[CH];
                        fetch(wr, wv, nv, seg);
#pragma unroll
                        for (int r = 0; r < 8; ++r) {
                            if (r >= cnt) break;
                            // the next row (or segment, or batch) on its way while this one is used
                            VT nxt[CH];
                            int kn = k0 + r + 1, sn = seg, nvn = nv;
                            if (r + 1 == cnt && seg + 1 < segs) { kn = k0; sn = seg + 1; }
                            else if (r + 1 == cnt) {
                                sn = 0;
                                nvn = kn < hd.nrows ? (__shfl_sync(FULL, r_len, kn) + VN - 1) / VN : 0;
                            }
                            if (nvn > 0) fetch_row(nxt, kn, nvn, sn);
                            T a = acc[r];
#pragma unroll
                            for (int q = 0; q < CH; ++q) a = vdot(cur[q], wr[q], a);
                            acc[r] = a;
                            if (nvn > 0)
#pragma unroll
                                for (int q = 0; q < CH; ++q) cur[q] = nxt[q];
                        }
                    }
                    const T s = reduce8(acc);
                    const T v = __shfl_sync(FULL, s, ((lane - k0) << 2) & 31);
                    if (lane >= k0 && lane < k0 + cnt) dot = v;
                }
            }
            const T xn = dot + c;
            pc.mark(trace, PHASE_VSTEP);
            // ---- z-step (Sec. III-C) of the wave's items and the u-step, u = -lambda
            const int type = ln.meta & 3, fr = (ln.meta >> 2) & 3, ns = ln.meta >> 5;
            T g = (T)0;
            for (int s = 0; s < hd.flags >> 8; ++s) {
                const int b = s < 6 ? (ln.base >> (5 * s)) & 31 : (ln.base2 >> (5 * (s - 6))) & 31;
                const T xs = __shfl_sync(FULL, xn, b + fr);
                if (s < ns) g += xs;
            }
            T la = fa * lam - (fm * g + e) * fk;
            if (type == TYPE_HARD) la = la > (T)0 ? la : (T)0;
            if (hd.flags & 2) {
                const int b = ln.base & 31;
                const T l0 = __shfl_sync(FULL, la, b), l1 = __shfl_sync(FULL, la, (b + 1) & 31);
                const T l2 = __shfl_sync(FULL, la, (b + 2) & 31);
                if (type == TYPE_CONTACT) {
                    if (!(l0 > (T)0)) {
                        // open, or (not a number) carried on
                        la = l0 <= (T)0 ? (T)0 : fr == 0 ? l0 : la;
                    } else if (fr > 0) {
                        const T t2 = l1 * l1 + l2 * l2, lim = mu * l0;
                        if (t2 > lim * lim) la = la * (lim * rsq(t2));
                    }
                }
            }
            const T dl = la - lam;
            U mloc = 0;
            // (a learned start's check after 10 iterations needs the z of the ninth, too)
            if (primal_stop || (learned_mode && l <= 9)) {
                const T zn = xn + dl * ib;
                if (own) mloc = umax(rbits(fabs(dl * ib)), rbits(fabs(zn - z)));
                z = zn;
            }
            if (own) {
                const T wn = P.pj ? la : bt * xn + (la + dl);
                if (tagged) tag_store(tw + ((l + 1) & 1) * tstride + (size_t)myt * 2 * sizeof(T), wn,
                                      (tag0 + (unsigned)l + 1u) & 0x7fffffffu);
                else (V.tb + (par ? S.ot_w0 : S.ot_w1))[myt] = wn;
                if (LONG && r_res < 0)             // D rows of the next iteration towards L2
                    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;"
                                 ::"l"(V.htb + r_drow), "r"((r_len + VN - 1) / VN * 16) : "memory");
            }
            xp = x;
            x = xn;
            lam2 = lam1;
            lam1 = lam;
            lam = la;
            fetch_first();
            iters = l + 1;
            par ^= 1;
            if (tagged) {
                pc.mark(trace, PHASE_ZSTEP);
                continue;
            }
            if (!(learned_mode && l == 9)) {
                // the stop test rides on the barrier: blocks with a residual above the tolerance
                // in the flags' low half, blocks with one that is not finite in the high half
                // (such a step ends at once; with a fixed count the step's residuals find it)
                unsigned over = 0;
                if (primal_stop) {
                    if (mloc >= inf_bits(T(0))) s_nan = 1;
                    over = __syncthreads_or(mloc > tolb) ? 1u : 0u;
                    if (s_nan) over |= 0x10000u;
                }
                over = bar.sync(over);
                pc.mark(trace, PHASE_ZSTEP);
                if (primal_stop) {
                    if (over >> 16) { status = ST_NAN; break; }
                    if (over == 0) { conv = 1; break; }
                }
                continue;
            }
            mloc = warp_umax(mloc);
            if (lane == 0) s_umax[wl] = (unsigned long long)mloc;
            __syncthreads();
            if (threadIdx.x == 0) {
                unsigned long long mb = 0ull;
                for (int k = 0; k < SUBADMM_ITER / 32; ++k) mb = umax(mb, s_umax[k]);
                if (mb) atomicMax(&G->umax[fallbacks], mb);
            }
            const unsigned long long ref10 = vload(&P.ref10[sc]);
            d.sync();
            const U mx = (U)vload(&G->umax[fallbacks]);
            pc.mark(trace, PHASE_ZSTEP);
            if (learned && (unsigned long long)mx > ref10) { restart = true; break; }
            if (!learned && lead) P.ref10[sc] = (unsigned long long)mx;
            if (learned && lead) P.learn_skip[2 * sc + 1] = 0;
            if (mx >= inf_bits(T(0))) { status = ST_NAN; break; }
            if (primal_stop && mx <= tolb) { conv = 1; break; }
        }
        if (restart) {
            // the learned start trails the plain one after 10 iterations: restart the step from
            // the plain start, and start plain for the next 2^streak - 1 steps
            if (lead) {
                const int streak = min(P.learn_skip[2 * sc + 1] + 1, 5);
                P.learn_skip[2 * sc + 1] = streak;
                P.learn_skip[2 * sc] = (1 << streak) - 1;
            }
            learned = false;
            ++fallbacks;
            wasted += l + 1;
            iter_duals<T>(P, S, V, &bar, false);
            load_duals();
            x = xp = (T)0;
            par = 0;
            l = 0;
            continue;
        }
        // publish x, y, z, lambda of the last iteration and y, z of the one before (after a
        // single iteration those are the initial ones, which init_duals left there), and, after
        // a tagged exchange, the w of the last v-step and the next one
        if (own) {
            (V.tb + S.ot_x)[myt] = x;
            (V.tb + S.ot_y)[myt] = bt * x - lam1;
            if (iters > 1) (V.tb + S.ot_yo)[myt] = bt * xp - lam2;
            const bool writes = ln.meta & 16;
            if (P.pj) {
                const T res = fabs(lam - lam1) / ((ln.meta & 3) == TYPE_SOFT ? (T)P.pj_omega * (V.tb + S.ot_invs)[V.row[myt]] : fk);
                (V.tb + S.ot_z)[myt] = (V.tb + S.ot_zo)[myt] = writes ? x - res : x;
            } else {
                (V.tb + S.ot_z)[myt] = x + (lam - lam1) * ib;
                if (iters > 1) (V.tb + S.ot_zo)[myt] = xp + (lam1 - lam2) * ib;
            }
            if (writes) (V.tb + S.ot_lam)[V.row[myt]] = lam;
            if (tagged) {
                if (iters > 1) (V.tb + (par ? S.ot_w0 : S.ot_w1))[myt] = P.pj ? lam1 : bt * xp + (lam1 + (lam1 - lam2));
                (V.tb + (par ? S.ot_w1 : S.ot_w0))[myt] = P.pj ? lam : bt * x + (lam + (lam - lam1));
            }
        }
        if (lead) G->chk = 0ull;
        if (tagged) d.sync();
        // v-hat from the last v-step's w (ADMM), or from the last z-step's lambda (Projected
        // Jacobi: v-hat = A^-1 (b + J^T lambda) with the impulses it reports); the D rows in
        // shared memory give way to the block solves
        iter_recover<T>(P, S, V, V.tb + ((P.pj ? par : par ^ 1) ? S.ot_w1 : S.ot_w0), &bar, P.grid_big ? smem : nullptr);
        d.sync();
        if (MIXED && conv && primal_stop && status == ST_OK) {
            // FP64 primal residual max |J v - z|; on a miss, refine c by the FP64 - FP32
            // difference of x at this iterate and resume
            const T *X = V.tb + S.ot_x, *Z = V.tb + S.ot_z;
            double part = 0.0;
            for (int t = d.tid; t < S.nsr; t += d.nthreads) {
                if (V.mlen[t] == 0) continue;
                const SubDesc &u = P.subs[S.sub0 + V.sub[t]];
                const int lr = t - u.sr0, n = u.n;
                const double *Jr = V.sdb + u.od_J + (size_t)lr * n;
                const double *v = V.sdb + u.od_v;
                const int *jl = P.ipool + u.env_off + 2 * n;
                double xd = 0.0;
                for (int p = jl[lr]; p < jl[u.m + lr]; ++p) xd += Jr[p] * v[p];
                part = nanmax(part, fabs(xd - (double)Z[t]));
                V.htb[V.coff[t]] += (T)(xd - (double)X[t]);
            }
            part = warp_max(part);
            if (lane == 0 && part > 0.0) atomicMax(&G->chk, dbits(part));
            d.sync();
            part = __longlong_as_double((long long)vload(&G->chk));
            if (part > P.tol && l + 1 < P.max_iters) {
                tolc *= 0.5;
                conv = 0;
                ++l;
                if (own) { c = V.htb[V.coff[myt]]; z = Z[myt]; }
                d.sync();                          // every block has read chk
                load_rows();
                fetch_first();
                continue;
            }
            if (part > P.tol) conv = 0;
        }
        break;
    }
    iter_finish<T>(P, S, V, &bar, &pc, trace, iters, conv, status, wasted, fallbacks);
}

}  // namespace subadmm
