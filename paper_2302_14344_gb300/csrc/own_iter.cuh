// The generic iteration of the block kernel with side-rows owned by threads.
//
// A thread (SPLIT lanes) keeps the constants, lambda and tables of up to SUBADMM_OWN side-rows in
// registers for the whole step: x = c + D w of its rows, a barrier, then the projection of its
// own rows from the x of their partners (each side of an interface projects the row itself).  Only
// x and w pass through shared memory, and lambda of contact rows, for their siblings; z and y are
// formed only where a stop test or the last two iterates need them (the updates are those of
// grid_iter.cuh).  The item loop that this replaces gathered and scattered y, z, lambda and the
// tables of every item in every iteration, 16 FP64 instructions a row where 6 do.
//
// A call of its own: the step kernel around it holds 0.8 KB of frames per thread, and with the
// shared memory full the L1 is too small for any spill inside the loop (the loop inline spilled
// its rows' state and took 7.2k cycles an iteration on the batched scenes, the item loop 7.6k; this
// takes 4.4k).  Offsets from the block's shared memory, not pointers, so that its accesses are
// shared-memory instructions.
#pragma once
#include "layout.h"

namespace subadmm {

// of own_iterate and item_iterate (item_iter.cuh)
struct IterResult {
    int l;                     // iterations run so far
    int conv;                  // 1: the stop test held in iteration l - 1
    int par, last_par;         // which w the next iteration reads, which one the last one read
    unsigned long long mx;     // asked for: the largest residual's bits of the last iteration
    double theta;              // theta of the last iteration (its stop rule)
    long long z_cycles;        // traced: cycles of the z-steps
};

// Iterations l .. lend - 1 of the scene whose descriptor and shared arrays these are (map: see
// SceneDesc::own_off); par: which of
// the two w holds iteration l's.  STOP: ends when no residual is above tolb.  max_iters: the step's
// limit (its last two iterations keep z and y).
template <typename T, int SPLIT, int NT, bool STOP>
__device__ __noinline__ IterResult own_iterate(const SceneDesc &S, const T *htb, const int *map, int l, int lend, int max_iters,
                                              int par, typename VecOf<T>::U tolb, bool want_max)
{
    using VT = typename VecOf<T>::V;
    using U = typename VecOf<T>::U;
    constexpr int VN = VecOf<T>::N, groups = NT / SPLIT, OWN = SUBADMM_OWN;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ U red[NT / 32];
    T *const tb = reinterpret_cast<T *>(smraw + S.t_base);
    const int *const ib = reinterpret_cast<const int *>(smraw + S.i_base);
    const int nsr = S.nsr;
    const int xg = threadIdx.x / SPLIT, xgl = threadIdx.x - xg * SPLIT;
    T *const X = tb + S.ot_x, *const LAM = tb + S.ot_lam;
    const T *const E = tb + S.ot_e;
    const int w0 = S.ot_w0, w1 = S.ot_w1;
    struct Own {
        int d;                 // D row: offset in shared memory's T region, or in htb
        int w;                 // first side-row of its subsystem
        int nv, row, other;    // vectors of the row (0: none); its constraint row; the same row's
                               // side-row on the other side (-1: none)
        int kind;              // type | row of its contact << 2 | D in shared memory << 4
        T bt, c, e, fk, lam;
    } ow[OWN];
    bool con = false;
#pragma unroll
    for (int k = 0; k < OWN; ++k) {
        const int t = xg + k * groups;
        Own &o = ow[k];
        o.nv = o.d = o.w = o.row = 0;
        o.other = -1;
        o.kind = 16;
        o.bt = o.c = o.e = o.fk = o.lam = (T)0;
        if (t >= nsr || ib[5 * nsr + t] == 0) continue;
        const int meta = map[t], dr = ib[2 * nsr + t], type = meta >> 16 & 3;
        o.nv = (ib[5 * nsr + t] + VN - 1) / VN;
        o.w = ib[4 * nsr + t];
        o.row = ib[t];
        o.other = (meta & 0xffff) - 1;
        const bool sh = dr < 0 || !S.hot_global;
        o.d = dr < 0 ? ~dr : dr;
        o.kind = type | (meta >> 18 & 3) << 2 | (sh ? 16 : 0);
        o.bt = tb[S.ot_b + t];
        o.c = htb[ib[3 * nsr + t]];
        o.e = E[o.row];
        o.fk = type == TYPE_SOFT ? tb[S.ot_kf + o.row] : tb[S.ot_invs + o.row];
        o.lam = LAM[o.row];
        con = con || type == TYPE_CONTACT;
    }
    con = __any_sync(0xffffffffu, con);
    IterResult res{l, 0, 0, 0, 0ull, 0.0, 0ll};
    for (; l < lend; ++l) {
        const int wc = par ? w1 : w0, wn = par ? w0 : w1;
        // ---- v-step
#pragma unroll
        for (int k = 0; k < OWN; ++k) {
            if (k * groups >= nsr) break;
            Own &o = ow[k];
            T acc = xgl == 0 ? o.c : (T)0, a1 = (T)0;
            const VT *wv = reinterpret_cast<const VT *>(tb + wc + o.w);
            auto dot = [&](const VT *dp) {
                int q = xgl;
                for (; q + 3 * SPLIT < o.nv; q += 4 * SPLIT) {
                    const VT d0 = dp[q], d1 = dp[q + SPLIT], d2 = dp[q + 2 * SPLIT], d3 = dp[q + 3 * SPLIT];
                    const VT v0 = wv[q], v1 = wv[q + SPLIT], v2 = wv[q + 2 * SPLIT], v3 = wv[q + 3 * SPLIT];
                    acc = vdot(d0, v0, acc);
                    if (sizeof(T) == 4) { a1 = vdot(d1, v1, a1); acc = vdot(d2, v2, acc); a1 = vdot(d3, v3, a1); }
                    else { acc = vdot(d1, v1, acc); acc = vdot(d2, v2, acc); acc = vdot(d3, v3, acc); }
                }
                for (; q < o.nv; q += SPLIT) acc = vdot(dp[q], wv[q], acc);
            };
            if (o.kind & 16) dot(reinterpret_cast<const VT *>(tb + o.d));
            else dot(reinterpret_cast<const VT *>(htb + o.d));
            if (sizeof(T) == 4) acc += a1;
#pragma unroll
            for (int h = SPLIT / 2; h; h >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, h);
            if (o.nv > 0 && xgl == 0) {
                X[xg + k * groups] = acc;
                if ((o.kind & 3) == TYPE_CONTACT) LAM[o.row] = o.lam;
            }
        }
        __syncthreads();
        // ---- z-step and u-step
        U mloc = 0;
        const bool keep = STOP || want_max || l + 2 >= max_iters;
#pragma unroll
        for (int k = 0; k < OWN; ++k) {
            if (k * groups >= nsr) break;
            Own &o = ow[k];
            const int t = xg + k * groups, type = o.kind & 3, fr = o.kind >> 2 & 3;
            if (o.nv == 0 || xgl != 0) continue;
            const T x = X[t], g = o.other >= 0 ? x + X[o.other] : x;
            T la;
            if (type == TYPE_SOFT) {
                const T al = tb[S.ot_al + o.row];
                la = o.fk * al / tb[S.ot_invs + o.row] * o.lam - (al * g + o.e) * o.fk;
            } else {
                la = o.lam - (g + o.e) * o.fk;
            }
            if (type == TYPE_HARD) la = above0(la) ? la : (T)0;
            if (con && type == TYPE_CONTACT) {
                if (fr == 0) {
                    la = above0(la) ? la : (T)0;
                } else {
                    // a tangent row needs the contact's normal row and the other tangent
                    auto trial = [&](int d) {
                        const T gr = o.other >= 0 ? X[t + d] + X[o.other + d] : X[t + d];
                        return LAM[o.row + d] - (gr + E[o.row + d]) * o.fk;
                    };
                    const T l0 = trial(-fr), l1 = trial(3 - 2 * fr);
                    if (!above0(l0)) {
                        la = (T)0;
                    } else {
                        const T t2 = la * la + l1 * l1, lim = tb[S.ot_mu + o.row] * l0;
                        if (above0(t2 - lim * lim)) la = la * (lim * rsq(t2));
                    }
                }
            }
            const T y = o.bt * x - o.lam;
            tb[wn + t] = (T)2 * la + y;
            if (keep) {
                T *const Y = tb + S.ot_y, *const YO = tb + S.ot_yo, *const Z = tb + S.ot_z, *const ZO = tb + S.ot_zo;
                const T dz = (la - o.lam) * tb[S.ot_invb + t], zn = x + dz, zo = Z[t];
                mloc = umax(mloc, umax(rbits(fabs(dz)), rbits(fabs(zn - zo))));
                ZO[t] = zo;
                Z[t] = zn;
                YO[t] = Y[t];
                Y[t] = y;
            }
            o.lam = la;
        }
        par ^= 1;
        if (want_max && l + 1 == lend) {
            mloc = warp_umax(mloc);
            if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mloc;
            __syncthreads();
            U mx = 0;
            for (int q = 0; q < NT / 32; ++q) mx = umax(mx, red[q]);
            res.mx = (unsigned long long)mx;
        } else if (STOP) {
            // (the stop test rides on the barrier, see step_kernel)
            if (__syncthreads_count(mloc > tolb && mloc < inf_bits(T(0))) == 0) {
                res.conv = 1;
                ++l;
                break;
            }
        } else {
            __syncthreads();
        }
    }
#pragma unroll
    for (int k = 0; k < OWN; ++k)
        if (ow[k].nv > 0 && xgl == 0) LAM[ow[k].row] = ow[k].lam;
    __syncthreads();
    res.l = l;
    res.par = par;
    res.last_par = par ^ 1;
    return res;
}

}  // namespace subadmm
