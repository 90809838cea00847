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

// Teams per SM and their threads: 1 x 1024, 2 x 512 or 6 x 256 (the small teams' kernel is held to 42
// registers).  A member's phases wait at barriers and on scattered reads, so several smaller teams cover each
// other; but a member then has fewer threads, and where one of them is what the call waits for, or where most
// of them list long subtrees, the call gets slower.  So small teams need (times against one team per SM, random
// sets of 200 to 2000 genes)
//  * a mean degree of 3.5: on sparser graphs a deleted node cuts off whole subtrees (recursive trees 1.06 to
//    2.8, G(n, M) of mean degree 3 0.51 to 1.24, of degree 4 to 8 0.43 to 1.12);
//  * eight members per SM for two teams (620 members, four per SM: 0.72 to 1.62; 920: 0.66 to 1.28; 1300 of up to
//    262144 nodes: 0.64 to 0.96), twelve for six (2048 members of up to 109649 nodes: 0.33 to 0.97);
//  * slices whose scattered reads the L2 holds: slices times nodes at most kSpEntries (two teams at n = 300000
//    and 400000: to 1.28 at 920 members and more; six at n = 160000: to 1.55);
//  * members that are light and alike, which the order kernel decides.
// Four teams of 256 are no better where they are safe (n up to 104000, 2048 members: 0.33 to 0.95) and up to 1.5
// times slower than one on lattices and on trees hung on a core (n = 160000).  A (mu+lambda) generation with 2048
// children (2000 genes, n = 100000, BA(3)) takes 706 / 529 / 472 us at 1 / 2 / 6 teams.
constexpr int kSpShapes = 3;
constexpr int kSpTeams[kSpShapes] = {1, 2, 6}, kSpThreads[kSpShapes] = {1024, 512, 256};
constexpr int kSpMembers[kSpShapes] = {0, 8, 12};  // members per SM from which a shape is taken
constexpr long long kSpEntries[kSpShapes] = {0, 80000000, 100000000};
constexpr int kSpMinDegree16 = 56;  // 16 times the mean degree

// One CTA's scratch: six int32 per node, an int32 and two int64 per component of two nodes or more.
inline size_t sp_slice_bytes(size_t stride, size_t comps) { return stride * 24 + comps * 20; }

struct SpLimits {
    int num_sms;
    size_t smem_per_sm, reserved;
};

inline int sp_shape(int n, int mean_deg_x16, int s, int k, const SpLimits& d) {
    if (mean_deg_x16 < kSpMinDegree16) return 0;
    int i = kSpShapes - 1;
    for (; i > 0; --i)
        if (s >= kSpMembers[i] * d.num_sms && (long long)kSpTeams[i] * d.num_sms * n <= kSpEntries[i] &&
            kSpTeams[i] * (sp_smem_bytes(n, k, kSpThreads[i]) + d.reserved + 1024) <= d.smem_per_sm)
            break;
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
