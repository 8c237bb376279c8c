// Where the instances of a batched solve run (host logic, plain C++).
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace nnqp {

constexpr int kResVectors = 9;        // vectors of a block's rows in the resident CG phase's shared memory

// Dynamic shared memory a CTA of the resident kernel may take (its static 22 KB
// come on top).
constexpr size_t kBatchSmemBytes = 204 * 1024;

// Shared memory of a CTA with `per` slices at most, of at most `slots` entries
// each, `vbytes` bytes a value (0 slots: the operator stays in global memory).
#if defined(__CUDACC__)
__host__ __device__ __forceinline__
#else
inline
#endif
size_t batch_res_table(int64_t per) { return ((size_t)(per + 1) * 4 + 15) / 16 * 16; }
inline size_t batch_res_bytes(int64_t per, int64_t slots, int vbytes) {
    return (size_t)per * slots * (4 + vbytes) + batch_res_table(per) + (size_t)kResVectors * per * 32 * vbytes;
}

// Where an instance of the resident kernel runs: CTAs of its cluster (0 = the
// plain kernels take it) and whether its operator is in shared memory.
struct ResPlace {
    int cluster = 0;
    bool local = false;
};

// Place of an instance of `slices` slices, the widest of `widest` entries, in
// clusters of at most `most` CTAs (a power of two).  As few CTAs as give each
// at most `target` slices -- an iteration's barrier and sums cost the same for
// 1 and 28 slices a CTA -- and as many as there are where the operator needs
// them to fit.  can(ctas, local) says whether the device schedules such
// clusters: one that does not (a partition, a part with fewer SMs side by
// side) gets the next size it does.
template <class Can>
ResPlace place_instance(int64_t slices, int64_t widest, int vbytes, int64_t target, int most, Can &&can) {
    auto fits = [&](int c, int64_t slots) {
        return batch_res_bytes((slices + c - 1) / c, slots, vbytes) <= kBatchSmemBytes;
    };
    for (int c = 1; c <= most; c *= 2)
        if ((slices + c - 1) / c <= target && fits(c, widest) && can(c, true)) return {c, true};
    for (int c = most; c >= 1; c /= 2)
        if (fits(c, widest) && can(c, true)) return {c, true};
    for (int c = most; c >= 1; c /= 2)
        if (fits(c, 0) && can(c, false)) return {c, false};
    return {};
}

// CTAs of the plain kernel for the instances that fit no resident place: the
// largest cluster that can(ctas), else 1 (a block per instance, which every
// device schedules).
template <class Can>
int plain_cluster(int most, Can &&can) {
    for (int c = most; c > 1; c /= 2)
        if (can(c)) return c;
    return 1;
}

}  // namespace nnqp
