// SixDST reachability (Section III-C, Eqs. 14-17) by bit rows: the same
// M = Normalizer((A + I)^N) as sixdst.cu, formed hop by hop along the arcs of
// the sparse graph instead of by dense products.
//
// The columns of M are independent: column c after h hops holds the nodes
// within h hops of c, and X_{h+1}[v] = X_h[v] | OR over live neighbours u of
// X_h[u].  A CTA takes one member and a strip of 32 W columns, keeps the
// strip's bits of every row in shared memory (two buffers of n + 1 rows of W
// words; a deleted node's row stays zero, so neighbours need no test) and
// runs the N hops with one barrier each, stopping early once a hop changes
// nothing.  Row sums are popcounts: PC_N sums them over the strips; MCN_N
// needs each row's sum over all strips, which the strips add into global
// counts.  The last strip of a member to finish writes its fitness.
//
// Adjacency layout (built at upload): nodes ranked by decreasing degree, ids
// 16-bit ranks.  Nodes of degree kBitsBig and more come first, one padded
// list each, walked by a whole warp; the others in slices of 32 ranks whose
// j-th neighbours are stored side by side, so that a warp reads 32
// neighbours with one 64-byte load and, degrees being sorted, hardly any lane
// waits for a longer list (padding points at row n, which stays zero).
//
// What bounds it: shared-memory gathers of 16 bytes per arc, strip and hop
// ((2E + n) n / 32 words per hop and member).  Measured at n = 2018, E = 2705,
// 80 members, 6 hops: 90 us against 1,700 us for the dense products (by node
// ids with a thread per row: 258 us with rows strided over the warps, 129 us
// with consecutive rows; ranked slices: 101 us; X_1 from the columns' own
// lists: 90 us).
#include <algorithm>
#include <vector>

#include "gapa_internal.cuh"

namespace {

constexpr int kBitsBig = 64;  // degree from which a whole warp walks a node's list

template <int W>
struct BitRow {
    unsigned w[W];
};

template <int W>
__device__ __forceinline__ BitRow<W> bits_load(const unsigned* p) {
    BitRow<W> r;
    if constexpr (W == 4) {
        const uint4 x = *reinterpret_cast<const uint4*>(p);
        r.w[0] = x.x, r.w[1] = x.y, r.w[2] = x.z, r.w[3] = x.w;
    } else {
        const uint2 x = *reinterpret_cast<const uint2*>(p);
        r.w[0] = x.x, r.w[1] = x.y;
    }
    return r;
}

template <int W>
__device__ __forceinline__ void bits_store(unsigned* p, const BitRow<W>& r) {
    if constexpr (W == 4) *reinterpret_cast<uint4*>(p) = make_uint4(r.w[0], r.w[1], r.w[2], r.w[3]);
    else *reinterpret_cast<uint2*>(p) = make_uint2(r.w[0], r.w[1]);
}

template <int W>
__device__ __forceinline__ void bits_or(BitRow<W>& a, const BitRow<W>& b) {
#pragma unroll
    for (int i = 0; i < W; ++i) a.w[i] |= b.w[i];
}

// The ranked adjacency (see above): rank[original id]; hub x's list = lines
// line[x] .. line[x+1]-1 of 32 entries for x < hubs, then slice x's likewise.
struct BitsGraph {
    int n, hubs, slices;
    const int* rank;
    const int* line;
    const unsigned short* col;
};

// sums[m]: the member's row sums over the strips done so far; done[m]: strips
// done; rows[m][n] (MCN only): row sums.  All zero at launch.
template <int W>
__global__ void __launch_bounds__(1024) sdst_bits_kernel(BitsGraph g, int strips, const int* __restrict__ pop, int k,
                                                         int hops, int mcn, unsigned long long* __restrict__ sums,
                                                         int* __restrict__ done, int* __restrict__ rows,
                                                         long long* __restrict__ fit, int* status) {
    extern __shared__ __align__(16) unsigned bits_smem[];
    __shared__ unsigned long long red[32];
    __shared__ int s_last;
    const int n = g.n, m = (int)(blockIdx.x / (unsigned)strips), strip = (int)(blockIdx.x % (unsigned)strips);
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = T >> 5;
    const int words = (n + 31) >> 5;
    unsigned* cur = bits_smem;
    unsigned* nxt = bits_smem + (size_t)(n + 1) * W;
    unsigned* dead = nxt + (size_t)(n + 1) * W;
    for (int w = tid; w < words; w += T) dead[w] = 0u;
    __syncthreads();
    for (int j = tid; j < k; j += T) {
        const int d = __ldg(&pop[(size_t)m * k + j]);
        if ((unsigned)d < (unsigned)n) {
            const int r = __ldg(&g.rank[d]);
            atomicOr(&dead[r >> 5], 1u << (r & 31));
        } else if (strip == 0) {
            atomicOr(status, GAPA_DEV_BAD_GENE);
        }
    }
    __syncthreads();
    // X_0 = I on the live nodes; deleted rows and the padding row are zero in both buffers
    for (int v = tid; v <= n; v += T) {
        BitRow<W> r{};
        bits_store<W>(nxt + (size_t)v * W, r);
        const bool live = v < n && !((dead[v >> 5] >> (v & 31)) & 1u);
#pragma unroll
        for (int i = 0; i < W; ++i) r.w[i] = live && (v >> 5) == strip * W + i ? 1u << (v & 31) : 0u;
        bits_store<W>(cur + (size_t)v * W, r);
    }
    __syncthreads();
    // X_1 from the lists of the strip's own columns (four lanes per column, a warp per hub) instead of a
    // pass over all rows
    for (int i = tid >> 2; i < 32 * W; i += T >> 2) {
        const int c = strip * 32 * W + i;
        if (c < g.hubs || c >= n || ((dead[c >> 5] >> (c & 31)) & 1u)) continue;
        const int x = g.hubs + ((c - g.hubs) >> 5), l1 = __ldg(&g.line[x + 1]);
        for (int l = __ldg(&g.line[x]) + (lane & 3); l < l1; l += 4) {
            const int u = __ldg(&g.col[(size_t)l * 32 + ((c - g.hubs) & 31)]);
            if (u < n && !((dead[u >> 5] >> (u & 31)) & 1u)) atomicOr(&cur[(size_t)u * W + (i >> 5)], 1u << (i & 31));
        }
    }
    for (int c = strip * 32 * W + warp; c < min(g.hubs, (strip + 1) * 32 * W); c += nw) {
        if ((dead[c >> 5] >> (c & 31)) & 1u) continue;
        for (int e = __ldg(&g.line[c]) * 32 + lane, e1 = __ldg(&g.line[c + 1]) * 32; e < e1; e += 32) {
            const int u = __ldg(&g.col[e]), i = c - strip * 32 * W;
            if (u < n && !((dead[u >> 5] >> (u & 31)) & 1u)) atomicOr(&cur[(size_t)u * W + (i >> 5)], 1u << (i & 31));
        }
    }
    __syncthreads();
    for (int h = 1; h < hops; ++h) {
        bool changed = false;
        for (int x = warp; x < g.hubs + g.slices; x += nw) {
            const int l0 = __ldg(&g.line[x]), l1 = __ldg(&g.line[x + 1]);
            const unsigned short* c = g.col + (size_t)l0 * 32 + lane;
            const bool hub = x < g.hubs;
            const int v = hub ? x : g.hubs + (x - g.hubs) * 32 + lane;
            BitRow<W> acc{};
#pragma unroll 4
            for (int l = l0; l < l1; ++l, c += 32) bits_or<W>(acc, bits_load<W>(cur + (size_t)__ldg(c) * W));
            if (hub) {
#pragma unroll
                for (int i = 0; i < W; ++i) acc.w[i] = __reduce_or_sync(0xffffffffu, acc.w[i]);
            }
            if (v < n && !((dead[v >> 5] >> (v & 31)) & 1u) && (!hub || lane == 0)) {
                const BitRow<W> old = bits_load<W>(cur + (size_t)v * W);
                bits_or<W>(acc, old);
#pragma unroll
                for (int i = 0; i < W; ++i) changed |= acc.w[i] != old.w[i];
                bits_store<W>(nxt + (size_t)v * W, acc);
            }
        }
        unsigned* t = cur;
        cur = nxt;
        nxt = t;
        if (!__syncthreads_or(changed)) break;  // every component is saturated: further hops add nothing
    }
    // row sums of this strip
    unsigned long long acc = 0;
    for (int v = tid; v < n; v += T) {
        const BitRow<W> r = bits_load<W>(cur + (size_t)v * W);
        int c = 0;
#pragma unroll
        for (int i = 0; i < W; ++i) c += __popc(r.w[i]);
        acc += (unsigned long long)c;
        if (mcn && c) atomicAdd(&rows[(size_t)m * n + v], c);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) red[warp] = acc;
    __threadfence();  // the row sums are visible before this strip counts as done
    __syncthreads();
    if (tid == 0) {
        unsigned long long tot = 0;
        for (int w = 0; w < nw; ++w) tot += red[w];
        if (!mcn) atomicAdd(&sums[m], tot);
        __threadfence();
        s_last = atomicAdd(&done[m], 1) == strips - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // the last strip: every other strip's sums are visible.  Deleted rows count nothing.
    int best = 0, gone = 0;
    if (mcn)
        for (int v = tid; v < n; v += T) best = max(best, __ldcg(&rows[(size_t)m * n + v]));
    else
        for (int w = tid; w < words; w += T) gone += __popc(dead[w]);
    best = __reduce_max_sync(0xffffffffu, best);
    gone = __reduce_add_sync(0xffffffffu, gone);
    if (lane == 0) red[warp] = mcn ? (unsigned long long)best : (unsigned long long)gone;
    __syncthreads();
    if (tid == 0) {
        unsigned long long x = 0;
        for (int w = 0; w < nw; ++w) x = mcn ? (red[w] > x ? red[w] : x) : x + red[w];
        if (mcn) fit[m] = (long long)x;
        else fit[m] = ((long long)__ldcg(&sums[m]) - (n - (long long)x)) / 2;
    }
}

size_t bits_smem_bytes(int n, int W) { return ((size_t)n + 1) * W * 8 + (((size_t)n + 31) >> 5) * 4; }

// Words per strip: four where two buffers of n rows fit in shared memory, else two.
int bits_words(const gapa_ctx* c, int n) { return bits_smem_bytes(n, 4) <= c->sdst_bits_smem_max ? 4 : 2; }

// Threads per CTA by how many CTAs shared memory lets an SM hold, and at least 512 where the strips are
// too few to share SMs.  Measured with 256 / 512 / 1024 threads (us, 80 members up to n = 3000 and 16
// above, 6 hops, mean degree 2.7): n = 300: 16 / 13 / 19; 1000: 30 / 40 / 50; 2018: 88 / 90 / 121; 3000:
// 206 / 171 / 217; 4000: 141 / 96 / 86; 7500: 677 / 418 / 333.
int bits_threads(const gapa_ctx* c, int W, long long ctas) {
    const size_t per_sm = c->smem_per_sm / (bits_smem_bytes(c->g.n, W) + 1024 + c->smem_reserved);
    const int T = per_sm >= 5 ? 256 : per_sm >= 2 ? 512 : 1024;
    return ctas <= 2ll * c->num_sms ? std::max(T, 512) : T;
}

// Members per launch: the scratch (a sum and a counter per member, and n row sums for MCN) stays within 64 MiB.
int bits_batch(const gapa_ctx* c, int s) {
    const size_t per = 16 + (c->objective == GAPA_OBJECTIVE_SIXDST_MCN ? (size_t)c->g.n * 4 : 0);
    return (int)std::max<size_t>(1, std::min<size_t>((size_t)std::max(s, 1), ((size_t)64 << 20) / per));
}

size_t bits_scratch_bytes(const gapa_ctx* c, int batch) {
    return (size_t)batch * (16 + (c->objective == GAPA_OBJECTIVE_SIXDST_MCN ? (size_t)c->g.n * 4 : 0));
}

}  // namespace

int gapa_sixdst_bits_init(gapa_ctx* c) {
    int rc = gapa_set_smem_limit((const void*)sdst_bits_kernel<4>, c->smem_optin, &c->sdst_bits_smem_max);
    if (rc == GAPA_OK) rc = gapa_set_smem_limit((const void*)sdst_bits_kernel<2>, c->smem_optin, &c->sdst_bits_smem_max);
    return rc;
}

bool gapa_sixdst_bits_fits(const gapa_ctx* c) {
    return c->g.sb_rank && bits_smem_bytes(c->g.n, 2) <= c->sdst_bits_smem_max;
}

int gapa_sixdst_bits_upload(DeviceGraph& g, const std::vector<int32_t>& rp, const std::vector<int32_t>& col) {
    const int n = g.n;
    std::vector<int32_t> by_deg((size_t)n), rank((size_t)n), line{0};
    for (int32_t v = 0; v < n; ++v) by_deg[v] = v;
    std::stable_sort(by_deg.begin(), by_deg.end(),
                     [&](int32_t a, int32_t b) { return rp[a + 1] - rp[a] > rp[b + 1] - rp[b]; });
    for (int32_t r = 0; r < n; ++r) rank[by_deg[r]] = r;
    auto degree = [&](int r) { return rp[by_deg[r] + 1] - rp[by_deg[r]]; };
    int hubs = 0;
    while (hubs < n && degree(hubs) >= kBitsBig) ++hubs;
    std::vector<uint16_t> out;
    for (int r = 0; r < hubs; ++r) {
        for (int32_t e = rp[by_deg[r]]; e < rp[by_deg[r] + 1]; ++e) out.push_back((uint16_t)rank[col[e]]);
        out.resize((out.size() + 31) / 32 * 32, (uint16_t)n);
        line.push_back((int32_t)(out.size() / 32));
    }
    const int slices = (n - hubs + 31) / 32;
    for (int s = 0; s < slices; ++s) {
        const int r0 = hubs + 32 * s, len = degree(r0);  // the slice's largest degree
        const size_t at = out.size();
        out.resize(at + (size_t)len * 32, (uint16_t)n);
        for (int r = r0; r < std::min(n, r0 + 32); ++r)
            for (int j = 0; j < degree(r); ++j) out[at + (size_t)j * 32 + (r - r0)] = (uint16_t)rank[col[rp[by_deg[r]] + j]];
        line.push_back((int32_t)(out.size() / 32));
    }
    if (cudaMalloc(&g.sb_rank, sizeof(int) * (size_t)n) != cudaSuccess ||
        cudaMalloc(&g.sb_line, sizeof(int) * line.size()) != cudaSuccess ||
        cudaMalloc(&g.sb_col, std::max<size_t>(out.size() * 2, 16)) != cudaSuccess) {
        cudaGetLastError();
        return gapa_fail(GAPA_ERR_OOM, "ranked adjacency of %d nodes", n);
    }
    GAPA_CUDA(cudaMemcpy(g.sb_rank, rank.data(), sizeof(int) * (size_t)n, cudaMemcpyHostToDevice));
    GAPA_CUDA(cudaMemcpy(g.sb_line, line.data(), sizeof(int) * line.size(), cudaMemcpyHostToDevice));
    if (!out.empty()) GAPA_CUDA(cudaMemcpy(g.sb_col, out.data(), out.size() * 2, cudaMemcpyHostToDevice));
    g.sb_hubs = hubs;
    g.sb_slices = slices;
    return GAPA_OK;
}

int gapa_sixdst_bits_prepare(gapa_ctx* c, int s) {
    return gapa_reserve(&c->sdst_buf, &c->sdst_cap, bits_scratch_bytes(c, bits_batch(c, s)), 1);
}

int gapa_launch_sixdst_bits(gapa_ctx* c, const int32_t* pop, int s, int k, int64_t* fit, cudaStream_t st,
                            int* kernels) {
    const int n = c->g.n, W = bits_words(c, n), strips = (n + 32 * W - 1) / (32 * W), batch = bits_batch(c, s);
    int rc = gapa_sixdst_bits_prepare(c, s);
    if (rc != GAPA_OK) return rc;
    const int mcn = c->objective == GAPA_OBJECTIVE_SIXDST_MCN;
    const int T = bits_threads(c, W, (long long)strips * batch);
    const BitsGraph bg{n, c->g.sb_hubs, c->g.sb_slices, c->g.sb_rank, c->g.sb_line, c->g.sb_col};
    unsigned long long* sums = reinterpret_cast<unsigned long long*>(c->sdst_buf);
    int* done = reinterpret_cast<int*>(sums + batch);
    int* rows = done + 2 * (size_t)batch;
    int launched = 0;
    for (int m0 = 0; m0 < s; m0 += batch) {
        const int cnt = std::min(batch, s - m0);
        GAPA_CUDA(cudaMemsetAsync(c->sdst_buf, 0, bits_scratch_bytes(c, batch), st));
        const auto kern = W == 4 ? sdst_bits_kernel<4> : sdst_bits_kernel<2>;
        kern<<<(unsigned)strips * (unsigned)cnt, T, bits_smem_bytes(n, W), st>>>(
            bg, strips, pop + (size_t)m0 * k, k, c->sixdst_hops, mcn, sums, done, rows,
            reinterpret_cast<long long*>(fit) + m0, c->status);
        GAPA_CUDA(cudaGetLastError());
        ++launched;
    }
    if (kernels) *kernels = launched;
    return GAPA_OK;
}
