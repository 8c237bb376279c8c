// Batched solves, host side: per-instance scratch, the launch shape (threads
// per block x CTAs per instance), the autotuner and the per-instance records.
// The kernels are in batch.cuh.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <numeric>
#include <vector>
#include "internal.h"
#include "batch.cuh"

namespace nnqp {

namespace {

BatchKernel pick_kernel(bool mixed, int tpb, int cluster, int cgv) {
    return mixed ? batch_kernel_mixed(tpb, cluster, cgv) : batch_kernel_fp64(tpb, cluster, cgv);
}

// Launch shape of the batch kernel: threads per block and CTAs per instance
// (1 = one block per instance, > 1 = a cluster per instance).  512 threads with
// more than one CTA is the resident kernel with at most that many CTAs per
// instance: each instance gets a cluster of its own size (batch_place.h).
//
// The default is 512 x 16.  A batch of 40 instances of 20 x 20 to 120 x 120
// cells in FP64: one 256-thread block per instance (the former default) 590 ms,
// bounded by the largest instance on one SM; clusters of 16 x 256 threads with
// form 0 / 2 of CG 105 / 104 ms; this 52 ms (with the same phase-end ratios; 38
// with the early ones).
struct BatchShape {
    int tpb = 512;
    int cluster = 16;
};
bool resident_shape(const BatchShape &s) { return s.tpb == 512 && s.cluster > 1; }

BatchShape g_tuned;          // process-wide choice of the autotuner
bool g_have_tuned = false;

double bytes_spmv(int64_t nnz, int64_t n, int sv, int sx) {
    return (double)nnz * (sv + 4) + 4.0 * (n + 1) + 2.0 * sx * n;
}

struct Scratch {
    DevArena a;
    cudaStream_t st;
    ~Scratch() { a.release(st); }
};

double den_of(const nn_system *s) {
    if (s->b0norm > 0.0) return s->b0norm;
    double m = 1.0;
    if (std::isfinite(s->lo)) m = std::max(m, std::fabs(s->lo));
    if (std::isfinite(s->hi)) m = std::max(m, std::fabs(s->hi));
    double d = s->anorm_inf * m;
    return d > 0 ? d : 1.0;
}

}  // namespace

nn_status check_opts(const nn_solve_opts *o);

// Runs the batch kernel; returns elapsed device milliseconds in *ms.
static nn_status run_batch(int count, nn_system *const *systems, double *const *c, const nn_solve_opts *o,
                           cudaStream_t st, BatchShape shape, nn_solve_info *infos, float *ms_out) {
    const bool mixed = o->precision == NN_PREC_MIXED;
    if (o->solver != NN_SOLVER_GPCG || o->format != NN_FMT_SELL) {
        set_error("nn_batch_solve runs GPCG on the SELL format");
        return NN_ERR_INVALID_ARG;
    }
    // (the resident kernel has the pipelined CG form without the crossing count)
    if (resident_shape(shape) && (getenv("NNQP_BATCH_CG_VARIANT") || getenv("NNQP_CG_BOUND_STOP"))) shape = {256, 1};
    std::vector<BatchInst> h(count);
    size_t w64 = 0, w32 = 0;
    for (int i = 0; i < count; ++i) {
        const nn_system *s = systems[i];
        if (!s || !c[i]) {
            set_error("nn_batch_solve: NULL system or vector at %d", i);
            return NN_ERR_INVALID_ARG;
        }
        if (s->dt > 0.0) {
            set_error("nn_batch_solve: system %d is transient", i);
            return NN_ERR_INVALID_ARG;
        }
        if (mixed && !s->has_mixed) {
            set_error("nn_batch_solve: system %d has no FP32 copy", i);
            return NN_ERR_INVALID_ARG;
        }
        w64 += (size_t)11 * s->NF;
        if (mixed) w32 += (size_t)13 * s->NF;
    }
    Scratch S;
    S.st = st;
    double *d64;
    float *d32 = nullptr;
    uint8_t *dfm;
    NN_TRY(S.a.alloc(&d64, w64, st));
    if (mixed) NN_TRY(S.a.alloc(&d32, w32, st));
    NN_TRY(S.a.alloc(&dfm, w64 / 11, st));
    size_t o64 = 0, o32 = 0, ofm = 0;
    for (int i = 0; i < count; ++i) {
        const nn_system *s = systems[i];
        BatchInst &b = h[i];
        b.n = s->NF;
        b.N = s->N;
        b.nslices = s->A64.nslices;
        b.sptr = s->A64.sptr;
        b.col = s->A64.col;
        b.val = s->A64.val;
        b.diag = s->diag64;
        b.dinv64 = s->dinv64;
        b.val32 = s->A32.val;
        b.rsum32 = s->rsum32;
        b.dinv32 = s->dinv32;
        b.b0 = s->b0;
        b.free_node = s->free_node;
        b.dmask = s->dmask;
        b.dval = s->dval;
        b.lo = s->lo;
        b.hi = s->hi;
        b.den = den_of(s);
        b.c = c[i];
        b.w64 = d64 + o64;
        o64 += (size_t)11 * s->NF;
        b.fm = dfm + ofm;
        ofm += (size_t)s->NF;
        if (mixed) {
            b.w32 = d32 + o32;
            o32 += (size_t)13 * s->NF;
        } else {
            b.w32 = nullptr;
        }
    }
    // largest first, by class of launch
    std::vector<int> order(count);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(),
                     [&](int a, int b) { return systems[a]->nnzF > systems[b]->nnzF; });
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    struct Launch {
        BatchShape shape;
        bool local = false;
        int first = 0, count = 0;
        size_t smem = 0;
        int clusters = 0;   // that the device runs at once
    };
    // CG form of the kernels other than the resident one
    const char *cgv_env = getenv("NNQP_BATCH_CG_VARIANT");
    const int cgv = cgv_env ? atoi(cgv_env) : 0;
    // Clusters of C CTAs of kernel k that the device runs at once, 0 = none.
    // NNQP_TEST_MAX_CLUSTER stands for a device that schedules none of more CTAs.
    const char *mc_env = getenv("NNQP_TEST_MAX_CLUSTER");
    const int max_cluster = mc_env ? atoi(mc_env) : kMaxCluster;
    auto schedulable = [&](const void *k, int tpb, int C, size_t smem) {
        if (!k || C > max_cluster) return 0;
        int n = 0;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = C;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.blockDim = dim3(tpb);
        cfg.gridDim = dim3(C * std::max(1, sms / C));
        cfg.dynamicSmemBytes = smem;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if ((smem && cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) ||
            (C > 8 && cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ||
            cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess)
            n = 0;
        cudaGetLastError();   // a refusal means the next choice
        return n;
    };
    auto res_kernel = [&](bool local) { return mixed ? batch_res_kernel_mixed(local) : batch_res_kernel_fp64(local); };
    std::vector<Launch> launches;
    if (!resident_shape(shape)) {
        launches.push_back({shape, false, 0, count, 0, 0});
    } else {
        // slices per CTA: what spreads the whole batch over the SMs, from 4 (a
        // warp each) to 24 (three a warp).  Measured with 4 / 8 / 16 / 24 / 36: 40
        // instances of 20 to 120 cells a side 46.3 / 44.4 / 42.0 / 42.8 / 39.0 ms
        // and with other data 43.4 / 41.4 / 39.0 / 37.8 / 38.9; 20 mixed ones of 30
        // to 90 15.7 / 14.1 / 14.0 / 11.0 / 12.9; 64 of 20 to 200 226 / 226 / 224 /
        // 226 / 219; 8 small ones of 20 to 50, which do not fill the device, 3.1 /
        // 3.4 / 4.3 / 5.5 / 6.8.
        int64_t total = 0;
        for (int i = 0; i < count; ++i) total += systems[i]->A64.nslices;
        const int64_t target = std::min<int64_t>(24, std::max<int64_t>(4, total / sms));
        const int vbytes = mixed ? 4 : 8;
        // (one CTA of the resident kernel fills an SM's registers, so the count does
        // not depend on how much of the shared memory a class takes)
        int at_once[2][kMaxCluster + 1];
        std::fill(&at_once[0][0], &at_once[0][0] + 2 * (kMaxCluster + 1), -1);
        auto clusters = [&](int c, bool local) {
            int &n = at_once[local][c];
            if (n < 0) n = schedulable((const void *)res_kernel(local), kBatchResThreads, c, kBatchSmemBytes);
            return n;
        };
        std::vector<ResPlace> place(count);
        for (int i = 0; i < count; ++i)
            place[i] = place_instance(systems[i]->A64.nslices, systems[i]->max_slice_slots, vbytes, target, shape.cluster,
                                      [&](int c, bool local) { return clusters(c, local) > 0; });
        auto key = [&](int i) { return place[i].cluster == 0 ? 64 : 2 * place[i].cluster + (place[i].local ? 0 : 1); };
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return key(a) > key(b); });
        for (int q = 0; q < count; ++q) {
            const int i = order[q];
            const ResPlace &pl = place[i];
            if (q == 0 || key(i) != key(order[q - 1])) {
                Launch l;
                l.shape = BatchShape{512, pl.cluster};
                if (!pl.cluster)
                    l.shape = {256, plain_cluster(kMaxCluster, [&](int c) {
                                   return schedulable((const void *)pick_kernel(mixed, 256, c, cgv), 256, c, 0) > 0;
                               })};
                l.local = pl.local;
                l.clusters = pl.cluster ? clusters(pl.cluster, pl.local) : 0;
                l.first = q;
                launches.push_back(l);
            }
            Launch &l = launches.back();
            ++l.count;
            if (pl.cluster) {
                const int64_t per = (systems[i]->A64.nslices + pl.cluster - 1) / pl.cluster;
                l.smem = std::max(l.smem, batch_res_bytes(per, pl.local ? systems[i]->max_slice_slots : 0, vbytes));
            }
        }
    }
    const int nl = (int)launches.size();
    BatchInst *dinst;
    int *dorder;
    unsigned *dnext;
    int64_t *dcnt;
    double *dsc;
    NN_TRY(S.a.alloc(&dinst, count, st));
    NN_TRY(S.a.alloc(&dorder, count, st));
    NN_TRY(S.a.alloc(&dnext, nl, st));
    NN_TRY(S.a.alloc(&dcnt, (size_t)count * kBatchCounters, st));
    NN_TRY(S.a.alloc(&dsc, (size_t)2 * count, st));
    NN_CUDA_TRY(cudaMemcpyAsync(dinst, h.data(), sizeof(BatchInst) * count, cudaMemcpyHostToDevice, st));
    NN_CUDA_TRY(cudaMemcpyAsync(dorder, order.data(), sizeof(int) * count, cudaMemcpyHostToDevice, st));
    NN_CUDA_TRY(cudaMemsetAsync(dnext, 0, sizeof(unsigned) * nl, st));
    // (-1: an instance that no cluster took, as every one of its class gave up)
    NN_CUDA_TRY(cudaMemsetAsync(dcnt, 0xff, sizeof(int64_t) * count * kBatchCounters, st));
    NN_CUDA_TRY(cudaMemsetAsync(dsc, 0xff, sizeof(double) * 2 * count, st));
    GpcgCtl ctl;
    ctl.tol = 0;
    ctl.face_tol = 0;
    ctl.max_spmv = o->max_iter;
    ctl.gp_max = 50;
    ctl.cg_max = 1 << 30;
    ctl.eta1 = kEta1;
    ctl.eta2 = kEta2;
    ctl.early_ratios = 0;   // (the batch has a cap of its own)
    ctl.mu = 1e-4;
    ctl.cg_variant = cgv;
    ctl.cg_bound_stop = 0;
    ctl.keep_p = 0;
    ctl.res_warps = 0;
    if (const char *e = getenv("NNQP_CG_BOUND_STOP")) ctl.cg_bound_stop = atoi(e);
    if (const char *e = getenv("NNQP_GP_MAX")) ctl.gp_max = atoi(e);
    if (const char *e = getenv("NNQP_ETA1")) ctl.eta1 = atof(e);
    if (const char *e = getenv("NNQP_ETA2")) ctl.eta2 = atof(e);
    // what may refuse a class comes before the first launch: a refused call has
    // touched no c[i]
    for (Launch &l : launches) {
        if (resident_shape(shape) && l.shape.tpb == 512) continue;   // (as placed)
        const int C = l.shape.cluster, tpb = C > 1 ? 256 : l.shape.tpb;
        BatchKernel k = pick_kernel(mixed, tpb, C, cgv);
        if (!k) {
            set_error("nn_batch_solve: no kernel for %d threads x %d CTAs, CG variant %d", tpb, C, cgv);
            return NN_ERR_INVALID_ARG;
        }
        if (C <= 1) continue;
        l.clusters = schedulable((const void *)k, tpb, C, 0);
        if (l.clusters < 1) {
            set_error("nn_batch_solve: clusters of %d CTAs cannot be scheduled on this device", C);
            return NN_ERR_INVALID_ARG;
        }
    }
    // The classes run side by side: the first on the caller's stream, each other
    // one on a stream of its own between two events of the caller's.
    struct Side {
        cudaStream_t st = nullptr;
        cudaEvent_t done = nullptr;
        ~Side() {
            if (done) cudaEventDestroy(done);
            if (st) cudaStreamDestroy(st);   // (its work is joined or, after an error, finishes by itself)
        }
    };
    std::vector<Side> sides(std::max(nl - 1, 0));
    struct Events {
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        ~Events() {
            if (e0) cudaEventDestroy(e0);
            if (e1) cudaEventDestroy(e1);
        }
    } ev;
    NN_CUDA_TRY(cudaEventCreate(&ev.e0));
    NN_CUDA_TRY(cudaEventCreate(&ev.e1));
    for (Side &x : sides) {
        NN_CUDA_TRY(cudaStreamCreateWithFlags(&x.st, cudaStreamNonBlocking));
        NN_CUDA_TRY(cudaEventCreateWithFlags(&x.done, cudaEventDisableTiming));
    }
    // bound on the waits of the resident kernel; NNQP_TEST_STALL_BARRIER=1 makes
    // them run out, as in a single solve
    const unsigned long long wait_ns = (unsigned long long)(o->wait_timeout_s * 1e9);
    const char *stall = getenv("NNQP_TEST_STALL_BARRIER");
    const int wait_extra = stall && stall[0] == '1' ? 1 : 0;
    // one launch of class l on stream q
    auto launch = [&](const Launch &l, unsigned *next, cudaStream_t q) -> nn_status {
        const bool res = resident_shape(shape) && l.shape.tpb == 512;
        const int C = l.shape.cluster, tpb = res ? kBatchResThreads : C > 1 ? 256 : l.shape.tpb;
        const BatchKernel kp = res ? nullptr : pick_kernel(mixed, tpb, C, cgv);
        if (!res && C <= 1) {
            int per = 0;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kp, tpb, 0);
            const int grid = std::max(1, std::min(l.count, std::max(per, 1) * sms));
            (kp<<<grid, tpb, 0, q>>>(dinst, dorder + l.first, l.count, next, ctl, o->rtol, o->inner_rtol, 200, dcnt, dsc),
             count_launch());
            return NN_OK;
        }
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = C;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.blockDim = dim3(tpb);
        cfg.gridDim = dim3(C * std::min(l.count, l.clusters));
        cfg.dynamicSmemBytes = l.smem;
        cfg.stream = q;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const BatchInst *di = dinst;
        const int *ord = dorder + l.first;
        NN_CUDA_TRY(res ? cudaLaunchKernelEx(&cfg, res_kernel(l.local), di, ord, l.count, next, ctl, o->rtol, o->inner_rtol, 200, dcnt, dsc,
                                             wait_ns, wait_extra)
                        : cudaLaunchKernelEx(&cfg, kp, di, ord, l.count, next, ctl, o->rtol, o->inner_rtol, 200, dcnt, dsc));
        count_launch();
        return NN_OK;
    };
    cudaEventRecord(ev.e0, st);
    nn_status lr = NN_OK;
    for (int q = 0; q < nl && lr == NN_OK; ++q) {
        cudaStream_t on = st;
        if (q > 0) {
            on = sides[q - 1].st;
            // (no early return past the join below)
            if (cudaStreamWaitEvent(on, ev.e0, 0) != cudaSuccess) {
                set_error("nn_batch_solve: a side stream cannot wait for the caller's");
                lr = NN_ERR_CUDA;
                break;
            }
        }
        lr = launch(launches[q], dnext + q, on);
    }
    // joined also after a failed launch: the others use this call's memory
    for (Side &x : sides) {
        cudaEventRecord(x.done, x.st);
        cudaStreamWaitEvent(st, x.done, 0);
    }
    cudaEventRecord(ev.e1, st);
    if (lr != NN_OK) {
        cudaStreamSynchronize(st);
        return lr;
    }
    std::vector<int64_t> hc((size_t)count * kBatchCounters);
    std::vector<double> hs((size_t)2 * count);
    NN_CUDA_TRY(cudaMemcpyAsync(hc.data(), dcnt, sizeof(int64_t) * hc.size(), cudaMemcpyDeviceToHost, st));
    NN_CUDA_TRY(cudaMemcpyAsync(hs.data(), dsc, sizeof(double) * hs.size(), cudaMemcpyDeviceToHost, st));
    NN_CUDA_TRY(cudaStreamSynchronize(st));
    NN_CUDA_TRY(cudaGetLastError());
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, ev.e0, ev.e1);
    if (ms_out) *ms_out = ms;
    nn_status worst = NN_OK;
    for (int i = 0; i < count; ++i) {
        int64_t *q = &hc[(size_t)i * kBatchCounters];
        nn_solve_info inf;
        std::memset(&inf, 0, sizeof(inf));
        if (q[0] < 0) {
            std::fill(q, q + kBatchCounters, 0);
            q[0] = NN_ERR_TIMEOUT;
        }
        inf.status = (int)q[0];
        inf.spmv64 = q[1];
        inf.spmv = q[1] + q[2];
        inf.cg_iters = q[3];
        inf.iterations = q[4];
        inf.refinements = q[5];
        inf.fp64_fallback = q[8];
        inf.kkt_rel = std::sqrt(hs[2 * i]) / hs[2 * i + 1];
        inf.kkt_inf = NAN;
        inf.objective = NAN;
        inf.time_ms = i == 0 ? ms : 0.0;
        const nn_system *s = systems[i];
        inf.bytes_algo = q[1] * bytes_spmv(s->nnzF, s->NF, 8, 8) + q[2] * bytes_spmv(s->nnzF, s->NF, 4, 4) +
                         (double)q[6] * 8.0 * s->NF + (double)q[7] * 4.0 * s->NF;
        if (infos) infos[i] = inf;
        if (inf.status != NN_OK && (worst == NN_OK || inf.status == NN_ERR_TIMEOUT)) worst = (nn_status)inf.status;
    }
    if (worst == NN_ERR_NOT_CONVERGED) set_error("some batch instances reached the iteration cap");
    else if (worst == NN_ERR_TIMEOUT) set_error("a device-side wait of the batch gave up after %.3g s", o->wait_timeout_s);
    return worst;
}

}  // namespace nnqp

using namespace nnqp;

extern "C" {

nn_status nn_batch_solve(int count, nn_system *const *systems, double *const *c, const nn_solve_opts *o,
                         void *stream, nn_solve_info *infos) {
    clear_error();
    nn_solve_opts d;
    nn_solve_opts_default(&d);
    if (!o) o = &d;
    NN_TRY(check_opts(o));
    if (o->precond != NN_PC_JACOBI) {
        set_error("batched solves use the Jacobi preconditioner");
        return NN_ERR_INVALID_ARG;
    }
    if (count < 1 || !systems || !c) {
        set_error("nn_batch_solve: count >= 1 and arrays are required");
        return NN_ERR_INVALID_ARG;
    }
    BatchShape shape;
    if (g_have_tuned) shape = g_tuned;
    // NNQP_BATCH_SHAPE="<threads>x<ctas>" overrides the shape (tests, sweeps)
    if (const char *e = getenv("NNQP_BATCH_SHAPE")) {
        int t = 0, c = 0;
        if (sscanf(e, "%dx%d", &t, &c) == 2 && (t == 128 || t == 256 || t == 512) && c >= 1 && c <= kMaxCluster &&
            (c & (c - 1)) == 0) {
            shape.tpb = c > 1 && t != 512 ? 256 : t;
            shape.cluster = c;
        }
    }
    return run_batch(count, systems, c, o, (cudaStream_t)stream, shape, infos, nullptr);
}

nn_status nn_batch_autotune(int count, nn_system *const *systems, const nn_solve_opts *o, void *stream,
                            int *best_shape) {
    clear_error();
    nn_solve_opts d;
    nn_solve_opts_default(&d);
    if (!o) o = &d;
    NN_TRY(check_opts(o));
    if (o->precond != NN_PC_JACOBI) {
        set_error("batched solves use the Jacobi preconditioner");
        return NN_ERR_INVALID_ARG;
    }
    if (count < 1 || !systems) {
        set_error("nn_batch_autotune: count >= 1 and systems are required");
        return NN_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    // Every candidate shape solves the whole batch to the requested tolerance
    // and the shape with the shortest elapsed time wins: the makespan depends
    // on how many instances run side by side as much as on how fast each one
    // runs, so a sample of the batch misjudges it (measured: a quarter of the
    // batch picked 16 CTAs per instance, 19% slower on the whole batch than 8).
    // One block per instance is a candidate only for batches of small
    // instances; clusters win as soon as an instance has thousands of rows.
    std::vector<nn_system *> sample(systems, systems + count);
    int64_t largest = 0;
    for (int i = 0; i < count; ++i) largest = std::max<int64_t>(largest, systems[i]->NF);
    const int ns = (int)sample.size();
    Scratch S;
    S.st = st;
    std::vector<double *> cs(ns);
    for (int i = 0; i < ns; ++i) NN_TRY(S.a.alloc(&cs[i], sample[i]->N, st));
    nn_solve_opts t = *o;
    std::vector<BatchShape> cands;
    if (largest <= 8192) {
        cands = {{512, 16}, {256, 1}, {512, 1}, {256, 4}, {256, 8}};
    } else {
        cands = {{512, 16}, {512, 8}, {256, 8}, {256, 16}};
    }
    float best = 1e30f;
    BatchShape pick_shape;
    std::vector<nn_solve_info> inf(ns);
    for (const BatchShape &sh : cands) {
        for (int i = 0; i < ns; ++i) NN_CUDA_TRY(cudaMemsetAsync(cs[i], 0, sizeof(double) * sample[i]->N, st));
        float ms = 0.0f;
        nn_status r = run_batch(ns, sample.data(), cs.data(), &t, st, sh, inf.data(), &ms);
        if (r == NN_ERR_INVALID_ARG) continue;   // shape not schedulable here
        if (r != NN_OK && r != NN_ERR_NOT_CONVERGED) return r;
        if (ms < best) {
            best = ms;
            pick_shape = sh;
        }
    }
    g_tuned = pick_shape;
    g_have_tuned = true;
    if (best_shape) *best_shape = pick_shape.tpb * 100 + pick_shape.cluster;
    clear_error();
    return NN_OK;
}

}  // extern "C"
