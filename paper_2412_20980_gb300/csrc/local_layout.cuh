// Shared-memory sizes of the TREE fitness kernels and the launch shape of the
// cut-local one.  Plain C++ when compiled without nvcc: the arithmetic is
// checked on the host for every graph size.
#pragma once

#include <algorithm>
#include <cstddef>

#ifdef __CUDACC__
#define GAPA_LAYOUT_FN __host__ __device__ __forceinline__
#else
#define GAPA_LAYOUT_FN inline
#endif

namespace gapa_dev {

GAPA_LAYOUT_FN size_t tree16_lab_bytes(int n) { return ((size_t)n * 2 + 15) & ~(size_t)15; }

// Shared-memory bytes of one member of the full pipeline on 32-bit labels: labels + deleted-node bitmap
// (reused as a node list once the labels are set) + four team-wide scalars.
GAPA_LAYOUT_FN size_t tree32_smem_bytes(int n) { return (size_t)n * 4 + (size_t)((n + 31) >> 5) * 4 + 16; }

// Layout of one member of the cut-local kernel: labels (16-byte units for the bulk copy), the list
// region (16-bit node ids, then the bitmap of listed nodes), twelve team scalars and the mbarrier.
GAPA_LAYOUT_FN size_t tree16l_bitmap_bytes(int n) { return ((((size_t)n + 31) >> 5) * 4 + 15) & ~(size_t)15; }
// The tops beyond which a member runs the full pipeline on 32-bit labels, by 16 times the mean degree.  Measured
// on BA, HK and G(n, M) graphs of mean degree 4 (2500 to 52000 nodes, 40 to 1000 members), n / 16, n / 8, n / 5 and
// n / 3: random sets 0.68, 0.56, 0.53 and 0.53 of the former kernel's time, hub-heavy ones 0.86, 0.77, 0.74 and 0.76 (at
// most 1.28, 1.17, 1.16 and 1.74).
GAPA_LAYOUT_FN bool tree16l_sparse(int mean_deg_x16) { return mean_deg_x16 < 80; }
GAPA_LAYOUT_FN int tree16l_tops_max(int n, int mean_deg_x16) { return tree16l_sparse(mean_deg_x16) ? n / 5 : n; }
// The least list region: the full pipeline's bitmap and scalars, and 512 entries (sparse graphs: all of
// the full pipeline on 32-bit labels).
GAPA_LAYOUT_FN size_t tree16l_min_list_bytes(int n, int mean_deg_x16) {
    const size_t least = tree16l_bitmap_bytes(n) + 1024 + 16;
    const size_t full = tree16l_sparse(mean_deg_x16) ? ((tree32_smem_bytes(n) + 15) & ~(size_t)15) - tree16_lab_bytes(n) : 0;
    return least > full ? least : full;
}
GAPA_LAYOUT_FN size_t tree16l_smem_bytes(int n, size_t list_bytes) { return tree16_lab_bytes(n) + list_bytes + 48 + 16; }

// Members per SM of the cut-local kernel, its threads per member and its list region: as many members as
// shared memory holds with lists of n / 2 entries, sharing the SM's 2048 threads, but no more than the
// population spreads over the SMs, and no more than 256 (512) threads up to 1024 (2048) nodes.  Measured at
// n = 20000 (1023 members of 1000 genes, random generation / hub-heavy fitness, whole call): three of 672
// threads 68 / 85 us, three of 512 66 / 93; four of 512 hold lists of n / 3 entries only, and hub-heavy members
// outgrow them.  80 members at n = 5009: 25 us with 1024 threads, 33 with 512.
struct LocalShape {
    int per_sm, threads, list_bytes;
};

// What the device offers: SMs, shared memory per SM, what the runtime reserves of it per block, and the most
// dynamic shared memory that one block of the fitness kernels may ask for.
struct LocalLimits {
    int num_sms;
    size_t smem_per_sm, reserved, block_max;
};

// Whether the kernel takes a graph: its least layout within one block's limit.
inline bool local_admits(int n, int mean_deg_x16, size_t block_max) {
    return tree16l_smem_bytes(n, tree16l_min_list_bytes(n, mean_deg_x16)) <= block_max;
}

inline LocalShape local_shape(int n, int mean_deg_x16, int s, const LocalLimits& d) {
    const size_t bm = tree16l_bitmap_bytes(n), fixed = tree16l_smem_bytes(n, 0);
    const size_t least = std::max(tree16l_min_list_bytes(n, mean_deg_x16), bm + (((size_t)n + 15) & ~(size_t)15));
    const size_t most = bm + (((size_t)n * 2 + 1024 + 15) & ~(size_t)15);
    int m = std::max(1, std::min(8, (s + d.num_sms - 1) / d.num_sms));
    for (;; --m) {
        // several members per SM share its memory, each with the runtime's reserve and 1 KB for the kernel's static
        // share; a member alone has the block's limit, which also decides what graphs the upload admits
        const size_t block = d.smem_per_sm / (size_t)m, other = d.reserved + 1024;
        const size_t room = m == 1 ? d.block_max : std::min(block > other ? block - other : 0, d.block_max);
        if (m == 1 || room >= fixed + least) {
            const size_t list = std::min(std::max(least, most), (room - fixed) & ~(size_t)15);
            return LocalShape{m, std::min(n <= 1024 ? 256 : n <= 2048 ? 512 : 1024, (2048 / m) & ~31), (int)list};
        }
    }
}

}  // namespace gapa_dev
