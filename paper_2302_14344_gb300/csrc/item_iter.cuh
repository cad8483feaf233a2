// The block kernel's general iteration: scenes whose items have more than two sides or whose
// side-rows are more than threads can own (own_iter.cuh), the theta stop rule, Projected Jacobi.
//
// v-step (lane groups, two side-rows per trip: independent load and FMA chains overlap), a barrier,
// z-step (a thread per projection item, the item's y, x and z through shared memory), a barrier.
// A call of its own, like own_iterate: inline, its tables and the code around it spilled each
// other's registers (280 bytes of spill stores in FP64; here none).  Explicit blocks of 3 sides,
// FP64: 8.9k -> 7.7k cycles an iteration.  Plain arguments, no struct by value: nvcc 13.0 handed a
// struct of ints, bools and two T on with other fields' values.
#pragma once
#include "layout.h"

namespace subadmm {

// what decides the projection and the end of the step
enum { ITEM_PJ = 1, ITEM_THETA = 2, ITEM_TOL = 4, ITEM_TRACE = 8 };

// Iterations l .. lend - 1 of the scene whose descriptor and shared arrays these are; par: which of
// the two w holds iteration l's; rule: ITEM_*; want_max: the residual of iteration lend - 1 is
// returned, not tested
template <typename T, int SPLIT, int NT>
__device__ __noinline__ IterResult item_iterate(const SceneDesc &S, const T *htb, int rule, T pj_omega, T theta_th,
                                                int l, int lend, int par, typename VecOf<T>::U tolb, bool want_max)
{
    using VT = typename VecOf<T>::V;
    using U = typename VecOf<T>::U;
    constexpr int VN = VecOf<T>::N, NW = NT / 32, groups = NT / SPLIT;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ U red[NW];
    __shared__ T tred[2][NW];
    T *const tb = reinterpret_cast<T *>(smraw + S.t_base);
    const int *const ib = reinterpret_cast<const int *>(smraw + S.i_base);
    const int nsr = S.nsr, nitem = S.nitem;
    const int *const row = ib, *const drow = ib + 2 * nsr, *const coff = ib + 3 * nsr;
    const int *const wbase = ib + 4 * nsr, *const mlen = ib + 5 * nsr;
    const Item *const item = reinterpret_cast<const Item *>(ib + 6 * nsr);
    const int *const list = ib + 6 * nsr + 4 * nitem;
    T *const X = tb + S.ot_x, *const Y = tb + S.ot_y, *const Z = tb + S.ot_z, *const LAM = tb + S.ot_lam;
    T *const YO = tb + S.ot_yo, *const ZO = tb + S.ot_zo;
    const T *const E = tb + S.ot_e, *const INVB = tb + S.ot_invb, *const BT = tb + S.ot_b;
    const T *const INVS = tb + S.ot_invs, *const KF = tb + S.ot_kf, *const AL = tb + S.ot_al, *const MU = tb + S.ot_mu;
    const int w0 = S.ot_w0, w1 = S.ot_w1;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int xg = tid / SPLIT, xgl = tid - xg * SPLIT, trips = (nsr + groups - 1) / groups;
    const bool stop_theta = rule & ITEM_THETA;
    IterResult res{l, 0, par, par, 0ull, 0.0, 0ll};
    for (; l < lend; ++l) {
        const T *const w = tb + (par ? w1 : w0);
        T *const wn = tb + (par ? w0 : w1);
        // ---- v-step through the affine map x = c + D w; y = beta x - lambda
        T tpart = (T)0;
        for (int k = 0; k < trips; k += 2) {
            int tt[2], mm[2];
            T acc[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                tt[h] = xg + (k + h) * groups;
                mm[h] = (k + h < trips && tt[h] < nsr) ? mlen[tt[h]] : 0;
                T a0 = (T)0, a1 = (T)0;
                if (mm[h] > 0) {
                    const int o = drow[tt[h]];          // (complemented: the copy in shared memory)
                    const VT *Dr = reinterpret_cast<const VT *>(o < 0 ? tb + ~o : htb + o);
                    const VT *wb = reinterpret_cast<const VT *>(w + wbase[tt[h]]);
                    const int nv = (mm[h] + VN - 1) / VN;
                    int c = xgl;
                    for (; c + SPLIT < nv; c += 2 * SPLIT) {
                        a0 = vdot(Dr[c], wb[c], a0);
                        a1 = vdot(Dr[c + SPLIT], wb[c + SPLIT], a1);
                    }
                    if (c < nv) a0 = vdot(Dr[c], wb[c], a0);
                }
                acc[h] = a0 + a1;
            }
#pragma unroll
            for (int o = SPLIT / 2; o; o >>= 1) {
                acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
                acc[1] += __shfl_xor_sync(0xffffffffu, acc[1], o);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int t = tt[h];
                if (mm[h] > 0 && xgl == 0) {
                    const T a = acc[h] + htb[coff[t]];
                    const T ynew = BT[t] * a - LAM[row[t]];
                    if (stop_theta) {
                        const T d = ynew - Y[t];
                        tpart += d * d;
                    }
                    YO[t] = Y[t];
                    Y[t] = ynew;
                    X[t] = a;
                }
            }
        }
        if (stop_theta) {
#pragma unroll
            for (int o = 16; o; o >>= 1) tpart += __shfl_xor_sync(0xffffffffu, tpart, o);
            if (lane == 0) tred[l & 1][warp] = tpart;
        }
        __syncthreads();
        if (stop_theta) {
            T ths = (T)0;
            for (int q = 0; q < NW; ++q) ths += tred[l & 1][q];
            if (l >= 1 && ths < theta_th) {
                // (before the z-step: w is that of this v-step)
                res.theta = (double)ths;
                res.conv = 1;
                res.l = l + 1;
                res.par = res.last_par = par;
                return res;
            }
        }
        const long long t0 = rule & ITEM_TRACE ? clock64() : 0ll;
        // ---- z-step (Sec. III-C); u = -lambda; max(|x - z|, |dz|) as bits
        U mloc = 0;
        for (int i = tid; i < nitem; i += NT) {
            const Item it = item[i];
            if (it.type < 0) continue;
            const int *ls = list + it.lo;
            if (rule & ITEM_PJ) {
                mloc = pj_item<T, U>(it, ls, X, E, INVS, KF, AL, MU, LAM, Z, ZO, wn, pj_omega, mloc);
                continue;
            }
            if (it.type == TYPE_CONTACT) {
                T q0 = (T)0, q1 = (T)0, q2 = (T)0;
                for (int s = 0; s < it.ns; ++s) {
                    const int t = ls[s];
                    const T ibt = INVB[t];
                    q0 += Y[t] * ibt; q1 += Y[t + 1] * ibt; q2 += Y[t + 2] * ibt;
                }
                const T is = INVS[it.row];
                const T ln = -(q0 + E[it.row]) * is;
                const T l1 = -(q1 + E[it.row + 1]) * is;
                const T l2 = -(q2 + E[it.row + 2]) * is;
                T lv[3];
                if (ln <= (T)0) {
                    lv[0] = lv[1] = lv[2] = (T)0;
                } else {
                    const T t2 = l1 * l1 + l2 * l2;
                    const T lim = MU[it.row] * ln;
                    lv[0] = ln;
                    if (t2 > lim * lim) { const T f = lim * rsq(t2); lv[1] = l1 * f; lv[2] = l2 * f; }
                    else { lv[1] = l1; lv[2] = l2; }
                }
                LAM[it.row] = lv[0]; LAM[it.row + 1] = lv[1]; LAM[it.row + 2] = lv[2];
                for (int s = 0; s < it.ns; ++s) {
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        const int t = ls[s] + r;
                        const T yv = Y[t], zo = Z[t];
                        const T zn = (yv + lv[r]) * INVB[t];
                        mloc = umax(mloc, umax(rbits(fabs(X[t] - zn)), rbits(fabs(zn - zo))));
                        ZO[t] = zo;
                        Z[t] = zn;
                        wn[t] = yv + (T)2 * lv[r];
                    }
                }
            } else {
                T q = (T)0;
                for (int s = 0; s < it.ns; ++s) q += Y[ls[s]] * INVB[ls[s]];
                const T e = E[it.row];
                T lv;
                if (it.type == TYPE_EQUALITY) lv = -(q + e) * INVS[it.row];
                else if (it.type == TYPE_HARD) { lv = -(q + e) * INVS[it.row]; lv = lv > (T)0 ? lv : (T)0; }
                else lv = -(e + AL[it.row] * q) * KF[it.row];
                LAM[it.row] = lv;
                for (int s = 0; s < it.ns; ++s) {
                    const int t = ls[s];
                    const T yv = Y[t], zo = Z[t];
                    const T zn = (yv + lv) * INVB[t];
                    mloc = umax(mloc, umax(rbits(fabs(X[t] - zn)), rbits(fabs(zn - zo))));
                    ZO[t] = zo;
                    Z[t] = zn;
                    wn[t] = yv + (T)2 * lv;
                }
            }
        }
        par ^= 1;
        if (want_max && l + 1 == lend) {
            mloc = warp_umax(mloc);
            if (lane == 0) red[warp] = mloc;
            __syncthreads();
            U mx = 0;
            for (int q = 0; q < NW; ++q) mx = umax(mx, red[q]);
            res.mx = (unsigned long long)mx;
        } else {
            // (the stop test rides on the barrier, see step_kernel)
            int over = 1;
            if (rule & ITEM_TOL) over = __syncthreads_count(mloc > tolb && mloc < inf_bits(T(0)));
            else __syncthreads();
            if (over == 0) res.conv = 1;
        }
        if (rule & ITEM_TRACE) res.z_cycles += clock64() - t0;
        if (res.conv) { ++l; break; }
    }
    res.l = l;
    res.par = par;
    res.last_par = par ^ 1;
    return res;
}

}  // namespace subadmm
