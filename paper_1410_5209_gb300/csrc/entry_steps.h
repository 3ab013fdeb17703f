// Walks over an item's entries in steps of consecutive entries, shared by the mode passes.
// Positions are ints (nnz < 2^31), but a position past an item's end need not fit one, so every
// test compares distances from the end and a walk advances only to a step that exists.
// Host code too: the walks of the last items of the largest tensors are checked there.
#pragma once

#include <stdint.h>

#include "../../include/tf_sals.h"

#ifdef __CUDACC__
#define TFS_HD __host__ __device__ __forceinline__
#else
#define TFS_HD inline
#endif

namespace tfs {

// Entry j0 + k (k >= 0) lies before jend.  j0 <= jend.
TFS_HD bool has_entry(int j0, int k, int jend) { return k < jend - j0; }
// A step of n entries at j0 reaches jend.
TFS_HD bool last_step(int j0, int n, int jend) { return jend - j0 <= n; }

struct Step {
    int32_t j0, jend;
    int32_t it;
    int32_t flags;  // 1 valid, 2 first step of its item, 4 last step of its item
};

// Steps of one warp, an entry per lane.
constexpr int kStepEntries = 32;

TFS_HD Step first_step(const tf_item &x, int64_t it) {
    Step s;
    s.it = (int32_t)it;
    s.j0 = (int32_t)x.begin;
    s.jend = (int32_t)(x.begin + x.len);
    s.flags = 1 | 2 | (last_step(s.j0, kStepEntries, s.jend) ? 4 : 0);
    return s;
}
TFS_HD Step no_step(int64_t it) {
    Step s;
    s.it = (int32_t)it;
    s.j0 = s.jend = 0;
    s.flags = 0;
    return s;
}
// The step after s in its item (s is not its last).
TFS_HD Step step_on(const Step &s) {
    Step n = s;
    n.j0 += kStepEntries;
    n.flags = 1 | (last_step(n.j0, kStepEntries, n.jend) ? 4 : 0);
    return n;
}

}  // namespace tfs
