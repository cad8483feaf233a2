// Triangular solves with one factor by a whole block (the grid kernel's large subsystems).
//
// A single-vector solve is a chain of n steps.  One warp walking it column by column pays a
// round trip to memory per column (the factor lives in the global workspace): 3.0M SM cycles
// per solve of a 1200-DOF slab.  Here the chain runs over panels of 32 rows: one warp solves
// the panel's 32 x 32 triangle from shared memory (32 dependent shuffle + FMA steps; its rows
// are scaled by 1 / L_pp as they are stored, so that no product is left on the chain), and all
// warps apply the panel to the rows (columns) that the envelope lets it reach.  Both the
// next triangle and the panel's rows are on their way while a triangle is solved, and the
// whole band is prefetched into L2 at the start (the iterations evict it).  The vector and the
// envelope stay in shared memory.  Four such solves and the FP64 refinement between them, for 64
// slabs: 10.6M -> 2.2M cycles per step.
#pragma once
#include "layout.h"

namespace subadmm {

// shared memory of a block solve: the vector, two diagonal tiles, the envelope
template <typename F>
struct BlockSolve {
    F *x;          // n
    F *tile;       // 2 x kPanel x kTileLd
    int *env;      // n
    __device__ __forceinline__ BlockSolve(unsigned char *smem, int n)
    {
        x = reinterpret_cast<F *>(smem);
        tile = x + (n + 1) / 2 * 2;
        env = reinterpret_cast<int *>(tile + 2 * kPanel * kTileLd);
    }
};

// the envelope into shared memory, and the rows of L inside it on their way into L2
template <int NT, typename F>
__device__ __forceinline__ void block_solve_begin(const F *L, int n, const int *env, const BlockSolve<F> &s)
{
    for (int r = threadIdx.x; r < n; r += NT) {
        const int lo = env[r];
        s.env[r] = lo;
        const char *p = reinterpret_cast<const char *>(L + (size_t)r * n + lo);
        const char *end = reinterpret_cast<const char *>(L + (size_t)r * n + r);
        for (; p <= end; p += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
    }
    __syncthreads();
}

// A panel's diagonal tile (lower triangle inside the envelope, zeros elsewhere), in registers
// (fetch) and then in shared memory (put): 1 / L_pp on the diagonal, the entries below it
// times the 1 / L_pp of their row (forward) or column (COLS, backward).  INVD: the diagonal of
// L holds 1 / L_pp, otherwise idg does.
template <int NT, typename F, bool INVD, bool COLS>
struct PanelTile {
    static constexpr int PER = kPanel * kPanel / NT, NW = NT / 32;
    F v[PER], inv[COLS ? 1 : PER];
    __device__ __forceinline__ F inverse(const F *L, const double *idg, int n, int r) const
    {
        if (r >= n) return (F)0;
        return INVD ? L[(size_t)r * n + r] : (F)idg[r];
    }
    __device__ __forceinline__ void fetch(const F *L, const double *idg, int n, int k0, const int *env)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int r = k0 + warp + NW * i, c = k0 + lane;
            v[i] = r < n && c < r && c >= env[r] ? L[(size_t)r * n + c] : (F)0;
            if (!COLS) inv[i] = inverse(L, idg, n, r);
        }
        if (COLS) inv[0] = inverse(L, idg, n, k0 + lane);
    }
    __device__ __forceinline__ void put(F *tile) const
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int r = warp + NW * i;
            const F q = inv[COLS ? 0 : i];
            tile[r * kTileLd + lane] = r == lane ? q : v[i] * q;
        }
    }
};

// x <- L^-1 x (x in shared memory, complete on entry and on return; block_solve_begin done;
// every thread of a block of NT threads)
template <int NT, typename F, bool INVD>
__device__ __noinline__ void block_forward(const F *L, const double *idg, int n, const int *lastr,
                                           BlockSolve<F> s)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr bool WIDE = sizeof(F) == 4;       // FP32: 8 lanes per row; FP64: a thread per row
    constexpr int PRE = !WIDE ? 1 : NT == 256 ? 6 : 3;           // (an FP64 add costs as much as a product)
    constexpr int ROWS = WIDE ? 4 * (NT / 32) : NT;  // rows per pass
    F *x = s.x;
    const int *env = s.env;
    PanelTile<NT, F, INVD, false> pt;
    pt.fetch(L, idg, n, 0, env);
    pt.put(s.tile);
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < n; k0 += kPanel, buf ^= 1) {
        const F *tile = s.tile + buf * kPanel * kTileLd;
        const int r0 = k0 + kPanel;                       // first row below the panel
        const int R = r0 <= n ? lastr[r0 - 1] : n - 1;
        // this thread's part of the rows below and of the next triangle
        F pre[PRE][WIDE ? 4 : kPanel];
        if (r0 < n) {
#pragma unroll
            for (int i = 0; i < PRE; ++i) {
                const int r = WIDE ? r0 + i * ROWS + warp * 4 + (lane >> 3) : r0 + (int)threadIdx.x;
                const int lo = r <= R ? env[r] : n;
#pragma unroll
                for (int j = 0; j < (WIDE ? 4 : kPanel); ++j) {
                    const int c = k0 + (WIDE ? (lane & 7) + 8 * j : j);
                    pre[i][j] = c >= lo ? L[(size_t)r * n + c] : (F)0;
                }
            }
            pt.fetch(L, idg, n, r0, env);
        }
        if (warp == 0) {
            F xi = k0 + lane < n ? x[k0 + lane] * tile[lane * kTileLd + lane] : (F)0;
#pragma unroll
            for (int j = 0; j < kPanel; ++j) {
                const F y = __shfl_sync(0xffffffffu, xi, j);
                if (lane > j) xi -= tile[lane * kTileLd + j] * y;
            }
            if (k0 + lane < n) x[k0 + lane] = xi;
        }
        __syncthreads();
        if (r0 >= n) break;
        pt.put(s.tile + (buf ^ 1) * kPanel * kTileLd);
        if (WIDE) {
            F y[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) y[j] = x[k0 + (lane & 7) + 8 * j];
            auto finish = [&](int r, F acc) {
#pragma unroll
                for (int o = 4; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if ((lane & 7) == 0 && r <= R) x[r] -= acc;
            };
#pragma unroll
            for (int i = 0; i < PRE; ++i) {
                if (r0 + i * ROWS > R) break;
                F acc = (F)0;
#pragma unroll
                for (int j = 0; j < 4; ++j) acc += pre[i][j] * y[j];
                finish(r0 + i * ROWS + warp * 4 + (lane >> 3), acc);
            }
            for (int rb = r0 + PRE * ROWS; rb <= R; rb += ROWS) {
                const int r = rb + warp * 4 + (lane >> 3), lo = r <= R ? env[r] : n;
                F acc = (F)0;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c = k0 + (lane & 7) + 8 * j;
                    if (c >= lo) acc += L[(size_t)r * n + c] * y[j];
                }
                finish(r, acc);
            }
        } else {
            for (int rb = r0; rb <= R; rb += ROWS) {
                const int r = rb + threadIdx.x;
                if (r <= R) {
                    F acc = x[r];
                    if (rb == r0) {
#pragma unroll
                        for (int j = 0; j < kPanel; ++j) acc -= pre[0][WIDE ? 0 : j] * x[k0 + j];
                    } else {
                        for (int c = max(k0, env[r]); c < r0; ++c) acc -= L[(size_t)r * n + c] * x[c];
                    }
                    x[r] = acc;
                }
            }
        }
        __syncthreads();
    }
    __syncthreads();
}

// x <- L^-T x, the panels from the last to the first; a thread per column that the panel
// reaches (coalesced along the rows of L)
template <int NT, typename F, bool INVD>
__device__ __noinline__ void block_backward(const F *L, const double *idg, int n, BlockSolve<F> s)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    F *x = s.x;
    const int *env = s.env;
    PanelTile<NT, F, INVD, true> pt;
    int k0 = (n - 1) / kPanel * kPanel, buf = 0;
    pt.fetch(L, idg, n, k0, env);
    pt.put(s.tile);
    __syncthreads();
    for (; k0 >= 0; k0 -= kPanel, buf ^= 1) {
        const F *tile = s.tile + buf * kPanel * kTileLd;
        const int kn = min(kPanel, n - k0);
        const int q0 = env[k0] + (int)threadIdx.x;        // env is nondecreasing
        F pre[kPanel];
#pragma unroll
        for (int j = 0; j < kPanel; ++j)
            pre[j] = j < kn && q0 < k0 && q0 >= env[k0 + j] ? L[(size_t)(k0 + j) * n + q0] : (F)0;
        if (k0 > 0) pt.fetch(L, idg, n, k0 - kPanel, env);
        if (warp == 0) {
            F xi = k0 + lane < n ? x[k0 + lane] * tile[lane * kTileLd + lane] : (F)0;
#pragma unroll
            for (int j = kPanel - 1; j >= 0; --j) {
                const F y = __shfl_sync(0xffffffffu, xi, j);
                if (lane < j) xi -= tile[j * kTileLd + lane] * y;
            }
            if (k0 + lane < n) x[k0 + lane] = xi;
        }
        __syncthreads();
        if (k0 > 0) pt.put(s.tile + (buf ^ 1) * kPanel * kTileLd);
        if (q0 < k0) {
            F acc = x[q0];
#pragma unroll
            for (int j = 0; j < kPanel; ++j)
                if (j < kn) acc -= pre[j] * x[k0 + j];
            x[q0] = acc;
        }
        for (int q = q0 + NT; q < k0; q += NT) {
            F acc = x[q];
            for (int j = 0; j < kn; ++j)
                if (q >= env[k0 + j]) acc -= L[(size_t)(k0 + j) * n + q] * x[k0 + j];
            x[q] = acc;
        }
        __syncthreads();
    }
}

}  // namespace subadmm
