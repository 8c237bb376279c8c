// Kernels of the batched solve: many independent QPs of uneven size in ONE
// persistent launch.  An instance is solved by one thread block (block
// barriers and reductions) or by one thread-block cluster (hardware cluster
// barrier, reductions through distributed shared memory); blocks / clusters
// take the next instance (largest first) from a device work counter, so no
// block ever waits on a block of another instance.  The solver is the same
// GPCG (and mixed-precision refinement) code as the single-system path.
// Instantiated per precision in batch_fp64.cu / batch_mixed.cu.
#pragma once
#include <stdint.h>
#include "internal.h"
#include "gpcg.cuh"
#include "refine.cuh"

namespace nnqp {


struct BatchInst {
    int64_t n, N, nslices;
    const int64_t *sptr;
    const int32_t *col;
    const double *val;
    const double *diag;
    const double *dinv64;
    const float *val32;
    const float *rsum32;
    const float *dinv32;
    const double *b0;
    const int32_t *free_node;
    const uint8_t *dmask;
    const double *dval;
    double lo, hi, den;
    double *c;          // full node vector: warm start in, solution out
    double *w64;        // 11 n doubles
    float *w32;         // 13 n floats (mixed)
    uint8_t *fm;        // n bytes: face mask of the CG phases
};

constexpr int kBatchResThreads = 512;

constexpr int kBatchCounters = 9;

// Solves instance `id` with team T; this CTA owns the rows R of it.
// RES: with the resident CG phase; its operator (LOCAL: in shared memory at op,
// entries from e0 on) and its shared memory at res.
template <int MIXED, int CGV, bool RES = false, bool LOCAL = false, class Team>
__device__ void solve_instance(Team &T, const Rows &R, const BatchInst &I, int id, unsigned rank, unsigned size,
                               const GpcgCtl &ctl, double rtol, double inner_rtol, int max_ref, int64_t *counters,
                               double *scalars, unsigned char *op = nullptr, unsigned char *res = nullptr,
                               int64_t e0 = 0) {
    const int64_t n = I.n;
    double *x = I.w64;
    R.each([&](int64_t i) { x[i] = I.c[I.free_node[i]]; });
    if (!T.sync()) return;
    const SellF64 A{n, I.nslices, I.sptr, I.col, I.val, I.diag};
    int64_t cnt[kBatchCounters] = {0};
    double gp2 = 0.0;
    int status;
    if (MIXED) {
        float *w = I.w32;
        GpcgVecs<float> v{w, w + n, w + 2 * n, w + 3 * n, w + 4 * n, w + 5 * n, w + 6 * n, w + 7 * n, w + 8 * n,
                          w + 9 * n, I.dinv32, I.fm, w + 12 * n};
        const SellF32Diff A32{n, I.nslices, I.sptr, I.col, I.val32, I.rsum32};
        double *w6 = I.w64;
        GpcgVecs<double> v64{x, w6 + n, w6 + 2 * n, w6 + 3 * n, w6 + 4 * n, w6 + 5 * n, w6 + 6 * n,
                             w6 + 7 * n, w6 + 8 * n, I.b0, I.dinv64, I.fm, w6 + 10 * n};
        MixedStats ms;
        if constexpr (RES) {
            const int64_t per = (I.nslices + size - 1) / size, ne = I.sptr[R.s1] - I.sptr[R.s0];
            v.res_sl = reinterpret_cast<int *>(res);
            v.res = reinterpret_cast<float *>(res + batch_res_table(per));
            SellF32DiffResX<LOCAL> Ar;
            if constexpr (LOCAL)
                static_cast<SellF32DiffLocal &>(Ar) =
                    SellF32DiffLocal{n, I.nslices, I.sptr, reinterpret_cast<const int32_t *>(op),
                                     reinterpret_cast<const float *>(op + ne * 4), I.rsum32, false, e0};
            else
                static_cast<SellF32Diff &>(Ar) = A32;
            status = mixed_solve<CGV, CGV, true>(T, R, A, Ar, I.lo, I.hi, I.b0, x, v, w + 9 * n, w + 10 * n, w + 11 * n,
                                                 v64, rtol * I.den, inner_rtol, max_ref, ctl.max_spmv,
                                                 batch_inner_product_cap(n), ctl, ctl, ms);
        } else {
            status = mixed_solve<CGV, CGV, true>(T, R, A, A32, I.lo, I.hi, I.b0, x, v, w + 9 * n, w + 10 * n, w + 11 * n, v64,
                                rtol * I.den, inner_rtol, max_ref, ctl.max_spmv, batch_inner_product_cap(n), ctl, ctl, ms);
        }
        cnt[1] = ms.spmv64;
        cnt[2] = ms.spmv32;
        cnt[3] = ms.cg;
        cnt[4] = ms.phases;
        cnt[5] = ms.refinements;
        cnt[6] = ms.vec64;
        cnt[7] = ms.vec32;
        cnt[8] = ms.fallback;
        gp2 = ms.gp2;
    } else {
        double *w = I.w64;
        GpcgVecs<double> v{w, w + n, w + 2 * n, w + 3 * n, w + 4 * n, w + 5 * n, w + 6 * n, w + 7 * n,
                           w + 8 * n, I.b0, I.dinv64, I.fm, w + 10 * n};
        GpcgCtl c = ctl;
        c.tol = rtol * I.den;
        c.face_tol = 0.5 * c.tol;
        GpcgStats gs;
        const Bounds<double> B{I.lo, I.hi, nullptr, nullptr};
        if constexpr (RES) {
            const int64_t per = (I.nslices + size - 1) / size, ne = I.sptr[R.s1] - I.sptr[R.s0];
            v.res_sl = reinterpret_cast<int *>(res);
            v.res = reinterpret_cast<double *>(res + batch_res_table(per));
            SellF64ResX<LOCAL> Ar;
            if constexpr (LOCAL)
                static_cast<SellF64Local &>(Ar) =
                    SellF64Local{n, I.nslices, I.sptr, reinterpret_cast<const int32_t *>(op),
                                 reinterpret_cast<const double *>(op + ne * 4), I.diag, false, e0};
            else
                static_cast<SellF64 &>(Ar) = A;
            status = gpcg_solve<Team, SellF64ResX<LOCAL>, double, CGV>(T, R, Ar, B, v, c, gs);
        } else {
            status = gpcg_solve<Team, SellF64, double, CGV>(T, R, A, B, v, c, gs);
        }
        x = v.x;
        cnt[1] = gs.spmv;
        cnt[3] = gs.cg;
        cnt[4] = gs.phases;
        cnt[6] = gs.vec;
        gp2 = gs.gp2;
    }
    R.each([&](int64_t i) { I.c[I.free_node[i]] = x[i]; });
    for (int64_t v = (int64_t)rank * blockDim.x + threadIdx.x; v < I.N; v += (int64_t)size * blockDim.x)
        if (I.dmask[v]) I.c[v] = I.dval[v];
    if (rank == 0 && threadIdx.x == 0) {
        cnt[0] = status;
        for (int k = 0; k < kBatchCounters; ++k) counters[(int64_t)id * kBatchCounters + k] = cnt[k];
        scalars[2 * id] = gp2;
        scalars[2 * id + 1] = I.den;
    }
}

// One thread block per instance.
template <int TPB, int MIXED, int CGV>
__global__ void __launch_bounds__(TPB) k_batch(const BatchInst *__restrict__ insts, const int *__restrict__ order,
                                               int count, unsigned *next, GpcgCtl ctl, double rtol,
                                               double inner_rtol, int max_ref, int64_t *counters, double *scalars) {
    __shared__ RedSmem sm;
    __shared__ int s_q;
    BlockTeam T{&sm};
    for (;;) {
        if (threadIdx.x == 0) s_q = (int)atomicAdd(next, 1u);
        __syncthreads();
        const int q = s_q;
        __syncthreads();
        if (q >= count) return;
        const int id = order[q];
        const BatchInst I = insts[id];
        solve_instance<MIXED, CGV>(T, Rows{0, I.nslices, I.n}, I, id, 0, 1, ctl, rtol, inner_rtol, max_ref, counters,
                              scalars);
        __syncthreads();
    }
}

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

// One thread-block cluster per instance: the instance's slices are split
// over the cluster's CTAs (one per SM), barriers are the hardware cluster
// barrier, reductions go through distributed shared memory.
template <int TPB, int MIXED, int CGV>
// CTAs per SM: 3 for FP64 (more clusters in flight hide more latency;
// measured 2.08 -> 1.94 s on the 512-instance batch), 2 for mixed precision,
// whose inner solves would spill at the 3-CTA register budget
__global__ void __launch_bounds__(TPB, MIXED ? 2 : 3) k_batch_cluster(const BatchInst *__restrict__ insts,
                                                       const int *__restrict__ order, int count, unsigned *next,
                                                       GpcgCtl ctl, double rtol, double inner_rtol, int max_ref,
                                                       int64_t *counters, double *scalars) {
    __shared__ RedSmem sm;
    __shared__ double xch[2 * kMaxCluster * kMaxRed];
    __shared__ int s_q;
    const unsigned rank = cluster_rank(), size = cluster_size();
    ClusterTeam T{&sm, xch, rank, size, 0, TPB / 32, nullptr, 0};
    for (;;) {
        if (rank == 0 && threadIdx.x == 0) s_q = (int)atomicAdd(next, 1u);
        T.sync();
        // every CTA reads the instance index taken by CTA 0
        __shared__ int s_q0;
        if (threadIdx.x == 0) {
            const uint32_t local = (uint32_t)__cvta_generic_to_shared(&s_q);
            uint32_t remote;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(0u));
            int q;
            asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(q) : "r"(remote) : "memory");
            s_q0 = q;
        }
        T.sync();
        const int q = s_q0;
        if (q >= count) break;
        const int id = order[q];
        const BatchInst I = insts[id];
        solve_instance<MIXED, CGV>(T, rows_of_block(I.n, I.nslices, (int)rank, (int)size), I, id, rank, size, ctl, rtol,
                              inner_rtol, max_ref, counters, scalars);
        T.sync();
    }
    T.sync();   // no CTA leaves while another may still read its shared memory
}

// The same with the CG phase's vectors in shared memory (cg_resident.cuh), and
// with LOCAL the CTA's slices of the operator too: 512 threads, one CTA per SM,
// clusters of 1 to 16 CTAs (an instance of 20 x 20 on one, of 120 x 120 on 16).
// Bound like the grid's mid-size solves (cg_resident.cuh), with a cluster's
// mbarriers and pushed sums (about 600 cycles) in place of the grid barrier
// (2,500).  Measured: see the rule of the launch shapes in batch.cu.
template <int MIXED, bool LOCAL>
__global__ void __launch_bounds__(kBatchResThreads, 1) k_batch_res(const BatchInst *__restrict__ insts,
                                                                  const int *__restrict__ order, int count,
                                                                  unsigned *next, GpcgCtl ctl, double rtol,
                                                                  double inner_rtol, int max_ref, int64_t *counters,
                                                                  double *scalars, unsigned long long wait_ns,
                                                                  int wait_extra) {
    __shared__ RedSmem sm;
    __shared__ double xch[2 * kMaxCluster * kMaxRed];
    __shared__ ClusterWaits cw;
    __shared__ int s_q, s_q0;
    extern __shared__ __align__(16) unsigned char dyn[];
    const unsigned rank = cluster_rank(), size = cluster_size();
    ClusterTeam T{&sm, xch, rank, size, 0, 1, &cw, 0};
    if (threadIdx.x == 0) T.res_init(wait_ns, wait_extra);
    for (;;) {
        if (rank == 0 && threadIdx.x == 0) s_q = (int)atomicAdd(next, 1u);
        T.sync();
        // every CTA reads the instance index taken by CTA 0
        if (threadIdx.x == 0) {
            int q;
            asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(q) : "r"(ClusterTeam::remote(&s_q, 0)) : "memory");
            s_q0 = q;
        }
        T.sync();
        if (s_q0 >= count) break;
        const int id = order[s_q0];
        const BatchInst I = insts[id];
        const Rows R = rows_of_block(I.n, I.nslices, (int)rank, (int)size);
        T.active = R.active_warps(kBatchResThreads / 32);
        const int64_t per = (I.nslices + size - 1) / size, e0 = I.sptr[R.s0], ne = I.sptr[R.s1] - e0;
        const int vbytes = MIXED ? 4 : 8;
        unsigned char *at = dyn;
        if constexpr (LOCAL) {
            const int4 *gc = reinterpret_cast<const int4 *>(I.col + e0);
            const int4 *gv = MIXED ? reinterpret_cast<const int4 *>(I.val32 + e0) : reinterpret_cast<const int4 *>(I.val + e0);
            for (int64_t q = threadIdx.x; q < ne / 4; q += blockDim.x) reinterpret_cast<int4 *>(dyn)[q] = __ldg(gc + q);
            for (int64_t q = threadIdx.x; q < ne * vbytes / 16; q += blockDim.x)
                reinterpret_cast<int4 *>(dyn + ne * 4)[q] = __ldg(gv + q);
            at += ne * (4 + vbytes);
        }
        GpcgCtl c = ctl;
        c.res_warps = resident_warps(per);
        solve_instance<MIXED, 2, true, LOCAL>(T, R, I, id, rank, size, c, rtol, inner_rtol, max_ref, counters, scalars,
                                              dyn, at, e0);
        T.sync();
        if (cw.gave_up) break;   // (the same on every CTA; the instances left go to other clusters or stay unsolved)
    }
    T.sync();   // no CTA leaves while another may still read its shared memory
}

using BatchKernel = void (*)(const BatchInst *, const int *, int, unsigned *, GpcgCtl, double, double, int,
                             int64_t *, double *);
using BatchResKernel = void (*)(const BatchInst *, const int *, int, unsigned *, GpcgCtl, double, double, int,
                                int64_t *, double *, unsigned long long, int);

// Kernel for threads per block tpb (128, 256, 512; clusters use 256), CTAs per
// instance cluster (1 = one block) and CG variant cgv (0, 1, 2); nullptr if
// that combination is not built.
BatchKernel batch_kernel_fp64(int tpb, int cluster, int cgv);
BatchKernel batch_kernel_mixed(int tpb, int cluster, int cgv);
// k_batch_res, any cluster size.
BatchResKernel batch_res_kernel_fp64(bool local);
BatchResKernel batch_res_kernel_mixed(bool local);

}  // namespace nnqp
