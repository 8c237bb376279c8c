// Products allowed to the FP32 inner solves of a mixed solve (host and device
// code).
#pragma once
#include <math.h>
#include <stdint.h>

#if defined(__CUDACC__)
#define NN_CAPS_FN __host__ __device__ __forceinline__
#else
#define NN_CAPS_FN inline
#endif

namespace nnqp {

// The first inner solve.  It starts from zero and
// has to do most of the solve's work: CG needs O(sqrt(cond)) steps and cond
// grows like n^(2/d), and GPCG adds the phases that find the active set
// (steady solves of 5e4 - 1e6 unknowns from zero take 6k - 40k products).  A
// cap only guards against an FP32 solve that cannot converge, so it is set
// well above that: 64 sqrt(n), at least 4000.
NN_CAPS_FN int64_t inner_product_cap(int64_t n) {
    const int64_t c = (int64_t)(64.0 * sqrt((double)n));
    return c > 4000 ? c : 4000;
}

// The same for the small instances of a batched solve (at most ~4e4
// unknowns): 8 sqrt(n), at least 4000.  A capped inner solve there still
// contracts the residual four-fold, and the refinement continues; with the
// larger cap some FP32 inner solves ran long before converging (measured on
// the 512-instance batch: 1.73M FP32 products and 275 solves/s against 1.63M
// and 310 solves/s).
NN_CAPS_FN int64_t batch_inner_product_cap(int64_t n) {
    const int64_t c = (int64_t)(8.0 * sqrt((double)n));
    return c > 4000 ? c : 4000;
}

// Every later inner solve, a correction of a residual already reduced, by the
// products of the first: at most twice as many, so that a stagnating FP32 solve
// is cut off early and the contraction test hands the solve to FP64.
//
// With the early phase-end ratios (a steady solve from afar) a quarter more, and
// at least 1,000: a later solve starts near its face and takes about half of
// the first (4,400 to 5,100, then 2,100 twice at 112 x 104 x 120).  One in
// ten there stalls in FP32 just above its tolerance, contracted by 7e3, and runs
// to the cap: 15,058 products and 756 ms with twice the first, 11,914 and 598 so
// (late ratios, whose first solve is twice as long: 619 ms).  On 2D meshes of
// 22k to 384k unknowns, 40^3, 60^3, 80^3 and a cube with a hole (69 solves at
// 1e-10, 34 at 1e-12) no later solve took as many as the first.
NN_CAPS_FN int64_t later_product_cap(int64_t first, bool early_ratios) {
    const int64_t base = first > 1000 ? first : 1000;
    if (!early_ratios) return 2 * base;
    return base + (base / 4 > 1000 ? base / 4 : 1000);
}

}  // namespace nnqp
