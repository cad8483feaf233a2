// One warp on a narrow band (at most 31 columns left of the diagonal: rigid chains have 11, the
// spring blocks 23): single-vector solves.
#pragma once
#include "layout.h"

namespace subadmm {

constexpr int kNarrowBand = 31;

// x <- L^-1 x and x <- L^-T x, in place (lanes hold rows k .. k + 31 of the window in registers).
// Row (column) r belongs to lane r % 32, which keeps its x while the 31 entries that reach it
// go by: a step is a product, a shuffle and an FMA (180 cycles in FP64, 35 in FP32), where the
// vector in memory took an axpy through L1 per column (1.2k cycles).  The entries of L are
// loaded eight steps ahead.  inv(r) = 1 / L_rr.
template <typename F, typename Inv>
__device__ __noinline__ void warp_band_forward(const F *L, int n, const int *env, F *x, Inv inv)
{
    constexpr int B = 8;
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    auto xat = [&](int r) -> F { return r < n ? x[r] : (F)0; };
    auto eat = [&](int r) -> int { return r < n ? env[r] : n; };
    int r = lane, e0 = eat(r), e1 = eat(r + 32), e2 = eat(r + 64);
    F xi = xat(r), xn = xat(r + 32);
    F a[B], iv;
    auto fetch = [&](F *o, F &v, int k0, int row, int ea, int eb) {
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const int k = k0 + j, q = row >= k ? row : row + 32, e = row >= k ? ea : eb;
            o[j] = q > k && q < n && k >= e ? L[(size_t)q * n + k] : (F)0;
        }
        v = row < k0 + B && row < n ? inv(row) : (F)0;
    };
    fetch(a, iv, 0, r, e0, e1);
    for (int k0 = 0; k0 < n; k0 += B) {
        const bool turn = r < k0 + B;                 // this lane's row ends in this batch
        const int rn = turn ? r + 32 : r;
        F an[B], ivn, yo = (F)0;
        fetch(an, ivn, k0 + B, rn, turn ? e1 : e0, turn ? e2 : e1);
        const F xnn = turn ? xat(rn + 32) : xn;
        const int e3 = turn ? eat(rn + 64) : e2;
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const F y = __shfl_sync(FULL, xi * iv, (k0 + j) & 31);
            if (r == k0 + j) { yo = y; xi = xn; }
            else xi -= a[j] * y;
        }
        if (turn) {
            if (r < n) x[r] = yo;
            e0 = e1; e1 = e2; e2 = e3;
        }
        r = rn;
        xn = xnn;
#pragma unroll
        for (int j = 0; j < B; ++j) a[j] = an[j];
        iv = ivn;
    }
    __syncwarp();
}

template <typename F, typename Inv>
__device__ __noinline__ void warp_band_backward(const F *L, int n, const int *env, F *x, Inv inv)
{
    constexpr int B = 8;
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    auto xat = [&](int c) -> F { return c >= 0 ? x[c] : (F)0; };
    // steps run over k = top, top - 1, ..; a lane's column is the largest c <= k with c % 32 == lane
    const int top = (n + B - 1) / B * B - 1;
    int c = top - ((top - lane) & 31);
    F xi = c < n ? xat(c) : (F)0, xn = xat(c - 32);
    F a[B], iv;
    auto fetch = [&](F *o, F &v, int k0, int col) {
        const int ke = k0 - (lane & (B - 1));          // lane j holds env of step j
        const int ev = ke >= 0 && ke < n ? env[ke] : n;
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const int k = k0 - j, q = col <= k ? col : col - 32, e = __shfl_sync(FULL, ev, j);
            o[j] = q < k && q >= e && k < n && k >= 0 ? L[(size_t)k * n + q] : (F)0;
        }
        v = col > k0 - B && col >= 0 && col < n ? inv(col) : (F)0;
    };
    fetch(a, iv, top, c);
    for (int k0 = top; k0 >= 0; k0 -= B) {
        const bool turn = c > k0 - B;
        const int cn = turn ? c - 32 : c;
        F an[B], ivn, yo = (F)0;
        fetch(an, ivn, k0 - B, cn);
        const F xnn = turn ? xat(cn - 32) : xn;
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const F y = __shfl_sync(FULL, xi * iv, (k0 - j) & 31);
            if (c == k0 - j) { yo = y; xi = xn; }
            else xi -= a[j] * y;
        }
        if (turn && c >= 0 && c < n) x[c] = yo;
        c = cn;
        xn = xnn;
#pragma unroll
        for (int j = 0; j < B; ++j) a[j] = an[j];
        iv = ivn;
    }
    __syncwarp();
}

}  // namespace subadmm
