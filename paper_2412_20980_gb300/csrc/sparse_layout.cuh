// Shared memory, launch shapes and scratch blocks of the sparse fitness
// kernel.  Plain C++ when compiled without nvcc: the rules are checked on the
// host.
#pragma once

#include <algorithm>
#include <cstddef>

#include "local_layout.cuh"

namespace gapa_dev {

GAPA_LAYOUT_FN size_t sp_bitmap_bytes(int n) { return ((((size_t)n + 31) >> 5) * 4 + 15) & ~(size_t)15; }
GAPA_LAYOUT_FN size_t sp_smem_bytes(int n, int k, int threads) {
    return sp_bitmap_bytes(n) + (((size_t)2 * k + 1) * 4 + 15) / 16 * 16 + (size_t)3 * threads * 4;
}

// Teams per SM and their threads: 1 x 1024, 2 x 512, 4 or 6 x 256 (the small teams' kernel is held to 42
// registers), the most that leave every SM two rounds of members to balance, that shared memory holds and
// that keep the scratch within 2.4 GB.  A member's phases wait at barriers and on scattered reads, so several
// smaller teams cover each other; with a single round the largest member, now on fewer threads, is what the
// call waits for (310 members of 2000 genes, n = 70000, BA(3): 139 us at 1 per SM, 167 at 2).  At 1 / 2 / 4
// per SM: 620 members 227 / 183 / 283 us, 1300 members 416 / 300 / 294.  One (mu+lambda) generation with 2048
// children (2000 genes, n = 100000, BA(3)), at 1 / 2 / 4 / 6: 706 / 529 / 510 / 472 us.  Members of uneven cost
// (up to all genes among the hubs, n = 100000) go the other way, 2048 of them 3551 / 3620 / 4396 / 3872, 762 of
// them 1421 / 1734 at 1 / 2: the order kernel keeps such calls at one member per SM.
constexpr int kSpShapes = 4;
constexpr int kSpTeams[kSpShapes] = {1, 2, 4, 6}, kSpThreads[kSpShapes] = {1024, 512, 256, 256};
constexpr long long kSpMaxEntries = 100000000;  // slices times nodes: 2.4 GB of scratch

// One CTA's scratch: six int32 per node, an int32 and two int64 per component of two nodes or more.
inline size_t sp_slice_bytes(size_t stride, size_t comps) { return stride * 24 + comps * 20; }

struct SpLimits {
    int num_sms;
    size_t smem_per_sm, reserved;
};

inline int sp_shape(int n, int s, int k, const SpLimits& d) {
    int i = kSpShapes - 1;
    for (; i > 0; --i) {
        const long long teams = (long long)kSpTeams[i] * d.num_sms;
        if (s >= 2 * teams && teams * n <= kSpMaxEntries &&
            kSpTeams[i] * (sp_smem_bytes(n, k, kSpThreads[i]) + d.reserved + 1024) <= d.smem_per_sm)
            break;
    }
    return i;
}

// The largest shape whose block is held after a call that wants `shape` (held: before it, -1 for none; alloc(i)
// makes the block of shape i and says whether it could).  A shape whose block could not be had is not asked
// for again (*refused; the next graph starts over), and the next smaller one serves.  may_grow false (a stream
// is being captured): what is held serves.
template <class Alloc>
inline int sp_grow(int held, int shape, bool may_grow, int* refused, Alloc alloc) {
    if (held >= 0 && !may_grow) return held;
    for (int i = std::min(shape, *refused - 1); i > held; --i) {
        if (alloc(i)) return i;
        if (i > 0) *refused = i;
    }
    return held;
}

}  // namespace gapa_dev
