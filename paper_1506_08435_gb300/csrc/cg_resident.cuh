// The CG phase of mid-size solves with every vector but one on the SM.
//
// Pipelined CG (Ghysels & Vanroose, Parallel Comput. 40, 2014) on the face, as
// form 2 of gpcg.cuh: the same recurrences, start and stop test.  What differs
// is where things live and who waits.  A mid-size system gives an SM a few tens
// of slices of 32 rows, whose operator is in shared memory (SellF64Local,
// SellF32DiffLocal).  Here the block's rows of the nine CG vectors are there
// too for the whole phase; only m = D^-1 w, which other rows gather, goes
// through global memory, double-buffered.  (In registers, unrolled over a
// thread's rows, they spilled from three rows a thread on.)
//
// What bounds an iteration on GB300 is latency: an FP64 warp instruction holds
// its sub-core for 64 cycles whatever it adds up, so a block-wide sum over 16
// warps, the division behind a coefficient and a grid barrier each cost as
// much as the arithmetic of the pass.  Therefore
//   * few compute warps with several slices each: a thread's rows are added by
//     the dot products' own FMAs, and the tree over the block has 4-12 warps;
//   * the two things that every block waits for are apart and hidden.  m goes
//     out first and its barrier (the first serving warp; the grid's counter count2, or a
//     cluster's mbarriers) runs while the other five recurrences and the dot
//     products are computed; the sums and the scalar step (the other three) run
//     while the next product is computed, which needs m only.
// The product of the iteration after the last one is thus computed and not
// used (one per phase; it is counted).
//
// Measured against form 2 with 16 warps and the vectors in L2, us per product
// of the whole solve: 50 x 50 6.4 -> 4.6, 120 x 120 6.4 -> 4.4, 397 x 283 10.2
// -> 6.5, 30^3 7.6 -> 4.5, 44^3 11.8 -> 7.6, 50^3 12.6 -> 10.1; the 40^3
// transient run, where every fourth product is a gradient projection's, 9.6 ->
// 7.4 in FP64.  At 40^3 an iteration is 12,500 cycles: product 6,200, waiting
// for the coefficients 1,200, recurrences and dot products 3,700, tree 700.
//
// Named barriers: 1 m written, 2 m visible grid-wide, 3 warp totals written,
// 4 coefficients ready, 5 among the summing warps.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include "team.cuh"
#include "ops.cuh"
#include "batch_place.h"

namespace nnqp {

// Compute warps at most.  A block's last four warps serve: 12-15 of 512-thread
// blocks; 4-7 of the 256-thread blocks of systems with at most four slices a
// block, of which two share an SM.
constexpr int kResWarps = 12;

// Compute warps for at most `per` slices a block: 8 (two a sub-core) up to
// three slices a warp, then 12; 4 where a warp has one slice at most.
__host__ __device__ __forceinline__ int resident_warps(int64_t per) { return per <= 4 ? 4 : per <= 24 ? 8 : 12; }

__device__ __forceinline__ void named_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
template <typename P>
__device__ __forceinline__ P *in_shared(P *p) {
    return (P *)__cvta_shared_to_generic(__cvta_generic_to_shared((const void *)p));
}
__device__ __forceinline__ void named_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Whether the phase ends after update `it`, read by every warp behind barrier
// 4.  The words are double-buffered by the update's parity: a warp that is
// slow to read them must not meet those of the next update, or it would leave
// alone and the block's barriers would no longer match.  (They lie behind the
// words of the phase's first reduction, which a slow warp may still read.)
__device__ __forceinline__ bool resident_done(const RedSmem &sm, int it, int64_t left) {
    const double *sc = sm.sc + 16 + 8 * (it & 1);
    return flag_set(sc[0]) || flag_set(sc[4]) || !flag_set(sc[3]) || flag_set(sc[7]) || sm.flag2[it & 1] == 0 ||
           it >= left;
}

// Whether it ended on the trust region's boundary (and for no other reason).
__device__ __forceinline__ bool resident_hit(const double *sc, int it, int64_t left) {
    return flag_set(sc[7]) && !flag_set(sc[0]) && !flag_set(sc[4]) && flag_set(sc[3]) && it < left;
}

// The trust region of TRON's subspace steps (tron.cuh; TR below).  The step ends
// where ||s|| would reach Delta.  ||s + alpha p||, with p the next direction, is
// followed by recurrences of s's, s'p and p'p from three more sums (u'u, u'p,
// u's), so the test needs no pass of its own.
struct ResidentTrust {
    double dd;           // Delta^2
    double ksp2, face2;  // stop at ||r||^2 <= max(ksp2 ||r_0||^2, face2), ...
    double ktol2;        // ... set here on the phase's first step (< 0 on entry), kept for the others
    bool hit;            // out: the step ends on the boundary
};

// Products y = A x of the rows of a compute warp's slices (local slices warp,
// warp + na, ... < ns).  The warp issues in order and 8 multiply-adds hold the
// sub-core's FP64 unit for 512 cycles, so the gathers run two batches of 8
// entries ahead of them: the next rows' loads are in flight while this row's
// terms are added (measured at 40^3: 6,300 cycles per product with a row's
// gathers issued at once and the next row's behind its multiply-adds).
// done(l, a0, a1) takes the sums of local row l = 32 slice + lane.
template <class Op, typename V, class FX, class F>
__device__ __forceinline__ void resident_product(const Op &A, const int *sl, bool wide, int warp, int na, int ns,
                                                 int lane, const V *x, FX &&xi, F &&done) {
    V X0[8], X1[8];
    auto width = [&](int t) { return t < ns ? (sl[t + 1] - sl[t]) >> 5 : 0; };
    int t = warp, w = width(t);
    if (!wide) {   // rows of at most 8 entries (2D meshes): one batch a slice
        int w1 = width(t + na);
        A.gather8(t < ns ? sl[t] : 0, w, 0, lane, x, X0);
        A.gather8(w1 ? sl[t + na] : 0, w1, 0, lane, x, X1);
        while (t < ns) {
            V a0 = (V)0, a1 = (V)0;
            A.fma8(sl[t], w, 0, lane, X0, xi(32 * t + lane), a0, a1);
            const int t2 = t + 2 * na, w2 = width(t2);
            A.gather8(w2 ? sl[t2] : 0, w2, 0, lane, x, X0);
            done(32 * t + lane, a0, a1);
            t += na;
            if (t >= ns) break;
            a0 = (V)0;
            a1 = (V)0;
            A.fma8(sl[t], w1, 0, lane, X1, xi(32 * t + lane), a0, a1);
            const int t3 = t + 2 * na;
            w = w2;
            w1 = width(t3);
            A.gather8(w1 ? sl[t3] : 0, w1, 0, lane, x, X1);
            done(32 * t + lane, a0, a1);
            t += na;
        }
        return;
    }
    if (t >= ns) return;
    int off = sl[t];
    A.gather8(off, w, 0, lane, x, X0);
    A.gather8(off, w, 8, lane, x, X1);
    for (;;) {
        const int tn = t + na, wn = width(tn), offn = tn < ns ? sl[tn] : 0;
        const V xl = xi(32 * t + lane);
        V a0 = (V)0, a1 = (V)0;
        A.fma8(off, w, 0, lane, X0, xl, a0, a1);
        A.gather8(offn, wn, 0, lane, x, X0);
        A.fma8(off, w, 8, lane, X1, xl, a0, a1);
        for (int k = 16; k < w; k += 8) {
            A.gather8(off, w, k, lane, x, X1);
            A.fma8(off, w, k, lane, X1, xl, a0, a1);
        }
        A.gather8(offn, wn, 8, lane, x, X1);
        done(32 * t + lane, a0, a1);
        if (tn >= ns) break;
        t = tn;
        off = offn;
        w = wn;
    }
}

// One CG phase from v.x, v.g; leaves the step in v.s.  Every thread of every
// block calls it; na compute warps.  Returns 0, ST_TIMEOUT when a wait gave
// up, or 1 when the face has nothing to reduce.  A call of its own: the
// registers the caller keeps live are saved once per phase.  TR: tr is its trust
// region and the stall test is left out.
template <bool TR, class Team, class Op, typename V>
__device__ __noinline__ int cg_resident(Team &T_, const Rows &R_, const Op &A_, const Bounds<V> &B,
                                        const GpcgVecs<V> &v_, const GpcgCtl &C_, GpcgStats &st, double ftol2,
                                        int na, ResidentTrust *tr) {
    constexpr int K = TR ? 6 : 3;   // sums of an update: gamma, delta, r'r (, u'u, u'p, u's)
    Team T = T_;
    const Rows R = R_;
    Op A = A_;
    if constexpr (IsResidentOp<Op>::local) {
        A.col = in_shared(A.col);   // (the compiler would read them with generic loads)
        A.val = in_shared(A.val);
    }
    const GpcgVecs<V> v = v_;
    const double eta2 = C_.eta2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool compute = warp < na;
    constexpr int serve = IsResidentOp<Op>::threads / 32 - 4;   // the first serving warp
    RedSmem &sm = *in_shared(T.sm);
    const V zero = (V)0;
    const int ns = (int)(R.s1 - R.s0), nl = ns * 32, base = (int)(R.s0 * 32);
    const int n = (int)(R.n - base) < nl ? (int)(R.n - base) : nl;   // local rows in use
    V *const z = in_shared(v.res), *const q = z + nl, *const p = q + nl, *const s = p + nl, *const r = s + nl,
            *const w = r + nl, *const u = w + nl, *const di = u + nl, *const y = di + nl;
    int *const sl = in_shared(v.res_sl);   // [ns + 1] first entry of each local slice
    V *mc = v.gw + base, *mn = v.m2 + base;
    const int64_t e0 = __ldg(A.sptr + R.s0);   // entries are counted from the block's first
    if constexpr (!IsResidentOp<Op>::local) {
        A.col += e0;
        A.val += e0;
    }
    for (int t = threadIdx.x; t <= ns; t += blockDim.x) sl[t] = (int)(__ldg(A.sptr + R.s0 + t) - (IsResidentOp<Op>::local ? A.e0 : e0));
    // rows l = 32 t + lane of the slices t = warp, warp + na, ... belong to
    // this thread throughout; a row off the face (or past the end) has di = 0
    if (compute)
#pragma unroll 1
        for (int l = 32 * warp + lane; l < nl; l += 32 * na) {
            V ri = zero, ui = zero, dl = zero;
            if (l < n) {
                const int64_t i = base + l;
                const V xi = v.x[i];
                if (num_lt(B.l(i), xi) && num_lt(xi, B.h(i))) {
                    dl = v.dinv[i];
                    ri = -v.g[i];
                    ui = dl * ri;
                }
                mn[l] = ui;
            }
            z[l] = q[l] = p[l] = s[l] = zero;
            r[l] = ri;
            u[l] = ui;
            di[l] = dl;
        }
    st.vec += 4;
    st.fl += 1;
    if (!T.sync()) return ST_TIMEOUT;
    bool wide = false;
    for (int t = threadIdx.x; t < ns; t += blockDim.x) wide = wide || sl[t + 1] - sl[t] > 8 * 32;
    wide = __syncthreads_or(wide);
    Acc<V> a3[TR ? 4 : 2];
    if (compute)
        resident_product(
            A, sl, wide, warp, na, ns, lane, mn - base, [&](int l) { return u[l]; },
            [&](int l, V a0, V a1) {
                const V dl = di[l], wl = is_set(dl) ? A.row_end(a0, a1, u[l], A.own(base + l, l < n), r[l]) : zero;
                w[l] = wl;
                if (l < n) mc[l] = dl * wl;
                a3[0] += r[l] * u[l];
                a3[1] += wl * u[l];
                if constexpr (TR) {
                    a3[2] += r[l] * r[l];
                    a3[3] += u[l] * u[l];
                }
            });
    double d3[TR ? 4 : 2], oc[TR ? 10 : 7], o3[7];
    // TR: (.., outside Delta, step to it, ktol2) of the first direction u
    if (!team_sum_scalar(T, a3, d3, oc, [&](const double (&d)[TR ? 4 : 2], double (&o)[TR ? 10 : 7]) {
            const double d2[2] = {d[0], d[1]};
            double o2[7];
            cg_scalar_start(d2, o2);
#pragma unroll
            for (int k = 0; k < 7; ++k) o[k] = o2[k];
            if constexpr (TR) {
                const double kt = tr->ktol2 < 0.0 ? fmax(tr->ksp2 * d[2], tr->face2) : tr->ktol2;
                if (tr->ktol2 >= 0.0 && d[2] <= kt) o[0] = 1.0;   // the face gradient is small enough
                const bool out = o2[1] * o2[1] * d[3] >= tr->dd;
                o[7] = out ? 1.0 : 0.0;
                o[8] = out ? sqrt(tr->dd / d[3]) : 0.0;
                o[9] = kt;
            }
        }))
        return ST_TIMEOUT;
    ++st.spmv;
    st.fl += 6;
#pragma unroll
    for (int k = 0; k < 7; ++k) o3[k] = oc[k];
    if constexpr (TR) {
        if (tr->ktol2 < 0.0) tr->ktol2 = oc[9];
        ftol2 = oc[9];
    }
    if (flag_set(o3[0])) {
        __syncthreads();
        T_ = T;
        return 1;   // no step on this face
    }
    if constexpr (TR) {
        if (flag_set(oc[7])) {
            if (compute)
#pragma unroll 1
                for (int l = 32 * warp + lane; l < n; l += 32 * na) v.s[base + l] = oc[8] * u[l];
            tr->hit = true;
            __syncthreads();
            T_ = T;
            return 0;
        }
    }
    CgScalars cs;
    cg_take(cs, o3);
    // updates allowed: at least one, as in the other forms
    int64_t left = C_.max_spmv - st.spmv;
    if (left > C_.cg_max) left = C_.cg_max;
    if (left < 1) left = 1;
    const int n1 = na * 32 + 32, n4 = na * 32 + 128;
    int it = 0;   // updates done
    if (compute) {
        V va = (V)cs.alpha, vb = (V)cs.beta;
        for (;;) {
            resident_product(
                A, sl, wide, warp, na, ns, lane, mc - base, [&](int l) { return di[l] * w[l]; },
                [&](int l, V a0, V a1) {
                    const V dl = di[l];
                    y[l] = is_set(dl) ? A.row_end(a0, a1, dl * w[l], A.own(base + l, l < n), w[l]) : zero;
                });
            if (it > 0) {
                named_sync(4, n4);
                if (resident_done(sm, it, left)) break;
                va = (V)sm.sc[16 + 8 * (it & 1) + 1];
                vb = (V)sm.sc[16 + 8 * (it & 1) + 2];
            }
#pragma unroll 1
            for (int l = 32 * warp + lane; l < nl; l += 32 * na) {
                const V wl = w[l], zl = y[l] + vb * z[l], wn = wl - va * zl;
                z[l] = zl;
                w[l] = wn;
                y[l] = wl;   // w before the update, for q below
                if (l < n) mn[l] = di[l] * wn;
            }
            __syncwarp();
            named_arrive(1, n1);
            Acc<V> a4[K];
#pragma unroll 1
            for (int l = 32 * warp + lane; l < nl; l += 32 * na) {
                const V ql = y[l] + vb * q[l], pl = u[l] + vb * p[l];
                const V rl = r[l] - va * ql, ul = di[l] * rl;
                q[l] = ql;
                p[l] = pl;
                const V sn = s[l] + va * pl;
                s[l] = sn;
                r[l] = rl;
                u[l] = ul;
                a4[0] += rl * ul;
                a4[1] += w[l] * ul;
                a4[2] += rl * rl;
                if constexpr (TR) {
                    a4[3] += ul * ul;
                    a4[4] += ul * pl;
                    a4[5] += ul * sn;
                }
            }
            double d4[K];
#pragma unroll
            for (int k = 0; k < K; ++k) d4[k] = a4[k].value();
            warp_stage<K>(d4, sm);
            __syncwarp();
            named_arrive(3, n1);
            ++it;
            V *t = mc;
            mc = mn;
            mn = t;
            named_sync(2, n1);
        }
        const double *sc = sm.sc + 16 + 8 * (it & 1);
        const bool hit = TR && resident_hit(sc, it, left);
        const V tau = hit ? (V)sc[6] : zero, bh = hit ? (V)sc[2] : zero;
#pragma unroll 1
        for (int l = 32 * warp + lane; l < n; l += 32 * na)
            v.s[base + l] = hit ? s[l] + tau * (u[l] + bh * p[l]) : s[l];
    } else if (warp == serve) {
        // m of every block visible
        for (;;) {
            named_sync(1, n1);
            ++it;
            const int ok = T.res_vector_barrier(it);
            if (lane == 0) sm.flag2[it & 1] = ok;
            __syncwarp();
            named_arrive(2, n1);
            named_sync(4, n4);
            if (resident_done(sm, it, left)) break;
        }
    } else if (warp > serve) {
        // sums over the block, then over the grid (entries k, k + 3 by serving warp 1 + k); then
        // the scalar step of cg_scalar_step, its two divisions and the stop test
        // on a warp (and sub-core) each: k = 0 alpha, 1 beta and 1 / gamma, 2 the
        // test.  (One warp after the other it took 1,850 cycles.)
        const int k = warp - (serve + 1);
        double t = cs.igamma * cs.ialpha;                          // k = 0
        double ig = cs.igamma;                                     // k = 1
        double dec = 0.5 * cs.alpha * cs.gamma, maxdec = dec;      // k = 2
        // TR, k = 0: p'p and s'p of the update to come, s's before it
        double pp = TR ? d3[TR ? 3 : 0] : 0.0, sp = 0.0, ss = 0.0, al = cs.alpha;
        for (;;) {
            ++it;
            double *sc = sm.sc + 16 + 8 * (it & 1);
            if (k == 0) {
                named_sync(3, n1);
                warp0_sum_warps<K>(sm, na);
                __syncwarp();
                const int ok = T.template res_publish<K>(it);
                if (lane == 0) sm.flag = ok;
                __syncwarp();
            }
            named_sync(5, 96);
            const double sum = sm.flag ? T.res_sum(k, it) : 0.0;
            if (lane == 0) sm.bcast[8 + k] = sum;
            if constexpr (TR) {
                const double more = sm.flag ? T.res_sum(k + 3, it) : 0.0;
                if (lane == 0) sm.bcast[11 + k] = more;
            }
            named_sync(5, 96);
            const double gamma = sm.bcast[8];
            double den = 0.0;
            if (k == 0) {
                // delta - beta gamma / alpha (gamma t = beta / alpha first: gamma^2
                // leaves the range where gamma, a square of the data, does not)
                den = fma(-(gamma * t), gamma, sm.bcast[9]);
                const double an = gamma / den;
                double out = 0.0, tau = 0.0;
                if constexpr (TR) {
                    ss += al * (2.0 * sp + al * pp);               // after update `it`
                    const double bn = gamma * ig, sps = sp + al * pp;
                    pp = sm.bcast[11] + bn * (2.0 * sm.bcast[12] + bn * pp);
                    sp = sm.bcast[13] + bn * sps;
                    al = an;
                    if (ss + an * (2.0 * sp + an * pp) >= tr->dd) {
                        out = 1.0;
                        const double ip = 1.0 / pp, h = sp * ip;   // (not sp^2, for the same reason)
                        tau = sqrt(fmax(fma(h, h, (tr->dd - ss) * ip), 0.0)) - h;
                    }
                }
                if (lane == 0) {
                    sc[1] = an;
                    sc[4] = den > 0.0 ? 0.0 : 1.0;
                    sc[6] = tau;
                    sc[7] = out;
                }
            } else if (k == 1) {
                const double bn = gamma * ig;
                ig = 1.0 / gamma;
                if (lane == 0) {
                    sc[2] = bn;
                    sc[5] = ig;
                }
            } else {
                const bool stop = (!TR && dec <= eta2 * maxdec) || sum <= ftol2 || !(gamma > 0.0);
                if (lane == 0) {
                    sc[0] = stop ? 1.0 : 0.0;
                    sc[3] = sm.flag ? 1.0 : 0.0;
                }
            }
            __syncwarp();
            named_sync(4, n4);
            if (resident_done(sm, it, left)) break;
            if (k == 0) {
                ig = sc[5];
                t = (den * ig) * ig;
            } else if (k == 2) {
                dec = 0.5 * sc[1] * gamma;
                maxdec = dec > maxdec ? dec : maxdec;
            }
        }
        if (k == 0 && lane == 0) sm.its = flag_set(sm.sc[16 + 8 * (it & 1) + 3]) && sm.flag2[it & 1] ? it : -1;
    }
    __syncthreads();
    it = sm.its;
    if (!T.res_agree(it >= 0)) return ST_TIMEOUT;
    if constexpr (TR) tr->hit = resident_hit(sm.sc + 16 + 8 * (it & 1), it, left);
    T_ = T;
    T_.res_end(it);
    st.spmv += it + 1;
    st.cg += it;
    st.fl += (TR ? 26 : 20) * (int64_t)it;
    return 0;
}

}  // namespace nnqp
