// Shared-memory TREE fitness pipelines with 16-bit ids (graphs of up to 56,281
// nodes: the 32-bit labels and bitmap of the full pipeline within one block),
// written for a "team": a group of warps of one CTA that evaluates one
// population member with its own slice of shared memory and its own named
// barrier.  A whole CTA is one team (barrier 0); the batched persistent kernel
// splits a CTA into 2, 4 or 8 teams so that small graphs run several members
// per CTA.
//
// Fitness (Section III-C, Eq. 13; PC(G) of Table "Whole"): pairwise
// connectivity of G with the member's genes deleted.  Nodes are in BFS
// numbering (every tree parent precedes its child); see fitness.cu for the
// phases.
#pragma once

#include "gapa_internal.cuh"
#include "local_layout.cuh"

namespace gapa_dev {

struct Team {
    int tid;  // thread index within the team
    int T;    // team size (a multiple of 32)
    int bar;  // named barrier id (0 = the whole CTA)
    __device__ __forceinline__ void sync() const {
        asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(T) : "memory");
    }
};

// Path halving.  Invariant: a non-root's parent has a smaller id, so the
// walk terminates; roots change only by CAS in uf_unite.
__device__ __forceinline__ int uf_find(volatile int* lab, int x) {
    while (true) {
        const int p = lab[x];
        if (p == x) return x;
        const int gp = lab[p];
        if (gp == p) return p;
        lab[x] = gp;
        x = gp;
    }
}

// Root of x by a read-only walk.  Used once no hooking is left: every write
// then is an owner storing its node's final root, so no walk can leave a
// stale (non-root) ancestor behind, which path halving could.
__device__ __forceinline__ int uf_root(volatile int* lab, int x) {
    int p = lab[x];
    while (p != x) {
        x = p;
        p = lab[x];
    }
    return x;
}

// Union of the trees of live nodes a and b: hook the larger root under the
// smaller with a CAS on the root's slot; retry from the new parent on a race.
__device__ __forceinline__ void uf_unite(volatile int* lab, int a, int b) {
    a = uf_find(lab, a);
    b = uf_find(lab, b);
    while (a != b) {
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = atomicCAS((int*)&lab[a], a, b);
        if (old == a) return;
        a = uf_find(lab, old);
        b = uf_find(lab, b);
    }
}

// ---- 16-bit labels ---------------------------------------------------------
typedef unsigned short lab_t;
constexpr int kDead16 = 0xFFFF;  // the label of a deleted node (ids stay below it)

__device__ __forceinline__ unsigned* lab_word(volatile lab_t* lab, int i) {
    return reinterpret_cast<unsigned*>(const_cast<lab_t*>(lab)) + (i >> 1);
}

// Compare-and-swap of one label through its 32-bit word; returns the label
// found.  A retry means that the word's other label changed meanwhile.
__device__ __forceinline__ int lab_cas(volatile lab_t* lab, int i, int expect, int val) {
    unsigned* w = lab_word(lab, i);
    const int sh = (i & 1) * 16;
    unsigned old = *(volatile unsigned*)w;
    while (true) {
        const int cur = (int)((old >> sh) & 0xFFFFu);
        if (cur != expect) return cur;
        const unsigned seen = atomicCAS(w, old, (old & ~(0xFFFFu << sh)) | ((unsigned)val << sh));
        if (seen == old) return cur;
        old = seen;
    }
}
// A label used as a counter: += v (no carry: counts stay below 2^16), and exchange with 0.
__device__ __forceinline__ void lab_add(volatile lab_t* lab, int i, unsigned v) {
    atomicAdd(lab_word(lab, i), v << ((i & 1) * 16));
}
__device__ __forceinline__ int lab_take(volatile lab_t* lab, int i) {
    const int sh = (i & 1) * 16;
    return (int)((atomicAnd(lab_word(lab, i), ~(0xFFFFu << sh)) >> sh) & 0xFFFFu);
}

// The union-find above on 16-bit labels.
__device__ __forceinline__ int uf_find(volatile lab_t* lab, int x) {
    while (true) {
        const int p = lab[x];
        if (p == x) return x;
        const int gp = lab[p];
        if (gp == p) return p;
        lab[x] = (lab_t)gp;
        x = gp;
    }
}

__device__ __forceinline__ int uf_root(volatile lab_t* lab, int x) {
    int p = lab[x];
    while (p != x) {
        x = p;
        p = lab[x];
    }
    return x;
}

// (R is the smallest of all: any root may be given that place, since a root
// has no link upwards that could then descend.)
__device__ __forceinline__ void uf_unite(volatile lab_t* lab, int a, int b, int R = -1) {
    a = uf_find(lab, a);
    b = uf_find(lab, b);
    while (a != b) {
        if (b != R && (a == R || a < b)) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = lab_cas(lab, a, a, b);
        if (old == a) return;
        a = uf_find(lab, old);
        b = uf_find(lab, b);
    }
}

__device__ __forceinline__ bool bm_test(const unsigned* bm, int v) { return (bm[v >> 5] >> (v & 31)) & 1u; }

// Sum (or, with mx, maximum) of non-negative values over the team; valid in
// team thread 0.  red: 32 slots of this team.
__device__ __forceinline__ long long team_sum_ll(const Team& tm, long long v, long long* red, bool mx = false) {
    for (int o = 16; o > 0; o >>= 1) {
        const long long x = __shfl_down_sync(0xffffffffu, v, o);
        v = mx ? (x > v ? x : v) : v + x;
    }
    const int warp = tm.tid >> 5, lane = tm.tid & 31;
    if (lane == 0) red[warp] = v;
    tm.sync();
    long long tot = 0;
    if (warp == 0) {
        tot = lane < (tm.T >> 5) ? red[lane] : 0;
        for (int o = 16; o > 0; o >>= 1) {
            const long long x = __shfl_down_sync(0xffffffffu, tot, o);
            tot = mx ? (x > tot ? x : tot) : tot + x;
        }
    }
    return tot;
}

// A component of c nodes in the objective: C(c, 2) summed for PC, c maxed for MCN.
__device__ __forceinline__ long long objective_add(long long acc, long long c, int objective) {
    return objective ? (c > acc ? c : acc) : acc + c * (c - 1) / 2;
}

struct Tree16Graph {
    int n;
    const int* perm;     // original id -> BFS number
    const int2* palt;    // (tree parent, second lower-numbered neighbour or -1)
    const int* lo_ptr;   // lower-numbered neighbours (CSR)
    const int* lo_col;
    const unsigned* nontree;  // non-tree edges a<<16|b
    int num_nontree;
    const int* fptr;          // full adjacency in BFS numbering (CSR, 16-bit ids)
    const unsigned short* fcol;
    int join_mode;            // 0: per member, 1: non-tree edges, 2: scan outside the giant piece
    int mean_deg_x16;         // 16 * 2E / n, rounded up
    int objective;            // 0: PC, 1: MCN
    CutTables cut;            // cut-local variant only
    int list_bytes;           // bytes of the member's list region
    int tops_max;             // more tops than this: the full pipeline on 32-bit labels
};

// The label pick of live node v: its tree parent if live, else its first
// live lower-numbered neighbour, else v; -1 for a deleted v.
__device__ __forceinline__ int tree16_pick(const unsigned* dead, const Tree16Graph& g, int v, int2 pa) {
    if (bm_test(dead, v)) return -1;
    if (pa.x == v || !bm_test(dead, pa.x)) return pa.x;
    if (pa.y < 0) return v;
    if (!bm_test(dead, pa.y)) return pa.y;
    const int beg = __ldg(&g.lo_ptr[v]) + 2, end = __ldg(&g.lo_ptr[v + 1]);
    for (int e = beg; e < end; ++e) {
        const int w = __ldg(&g.lo_col[e]);
        if (!bm_test(dead, w)) return w;
    }
    return v;
}

// Unite every live node of a warp's `cnt` nodes (node of lane j: nodes[j],
// -1 for none) with its live neighbours.  The arcs of the warp's nodes are
// laid end to end and dealt out one per lane; a lane finds its node by binary
// search over the warp's degree prefix sums.
template <class L>  // 16-bit labels, or 32-bit ones with -1 for deleted nodes
__device__ __forceinline__ void tree16_scan_warp(volatile L* lab, const Tree16Graph& g, int v, int lane) {
    int b = 0, d = 0;
    if (v >= 0) {
        b = __ldg(&g.fptr[v]);
        d = __ldg(&g.fptr[v + 1]) - b;
    }
    int incl = d;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    for (int s0 = 0; s0 < total; s0 += 32) {
        const int idx = s0 + lane;
        int lo = 0, hi = 31;
#pragma unroll
        for (int step = 0; step < 5; ++step) {
            const int mid = (lo + hi) >> 1;
            if (__shfl_sync(0xffffffffu, incl, mid) > idx) hi = mid; else lo = mid + 1;
        }
        const int ov = __shfl_sync(0xffffffffu, v, lo), ob = __shfl_sync(0xffffffffu, b, lo),
                  oi = __shfl_sync(0xffffffffu, incl, lo), od = __shfl_sync(0xffffffffu, d, lo);
        if (idx < total) {
            const int w = __ldg(&g.fcol[ob + idx - (oi - od)]);
            const int lw = lab[w];
            if (lw != (sizeof(L) == 2 ? kDead16 : -1) && lw != lab[ov]) uf_unite(lab, ov, w);
        }
    }
}

// Unites along the non-tree edges whose ends carry different labels, four
// edges per 16-byte load.
__device__ __forceinline__ void tree16_join_nontree(const Team& tm, volatile lab_t* lab, const Tree16Graph& g) {
    const int tid = tm.tid, T = tm.T;
    const uint4* e4 = reinterpret_cast<const uint4*>(g.nontree);
    const int quads = g.num_nontree >> 2;
    int q = tid;
    uint4 w = q < quads ? __ldg(&e4[q]) : make_uint4(0, 0, 0, 0);
    while (q < quads) {
        const int qn = q + T;
        const uint4 wn = qn < quads ? __ldg(&e4[qn]) : make_uint4(0, 0, 0, 0);
        const int a0 = (int)(w.x >> 16), b0 = (int)(w.x & 0xFFFFu), a1 = (int)(w.y >> 16), b1 = (int)(w.y & 0xFFFFu);
        const int a2 = (int)(w.z >> 16), b2 = (int)(w.z & 0xFFFFu), a3 = (int)(w.w >> 16), b3 = (int)(w.w & 0xFFFFu);
        const int la0 = lab[a0], lb0 = lab[b0], la1 = lab[a1], lb1 = lab[b1];
        const int la2 = lab[a2], lb2 = lab[b2], la3 = lab[a3], lb3 = lab[b3];
        if (la0 != lb0 && la0 != kDead16 && lb0 != kDead16) uf_unite(lab, la0, lb0);
        if (la1 != lb1 && la1 != kDead16 && lb1 != kDead16) uf_unite(lab, la1, lb1);
        if (la2 != lb2 && la2 != kDead16 && lb2 != kDead16) uf_unite(lab, la2, lb2);
        if (la3 != lb3 && la3 != kDead16 && lb3 != kDead16) uf_unite(lab, la3, lb3);
        q = qn;
        w = wn;
    }
    for (int e = quads * 4 + tid; e < g.num_nontree; e += T) {
        const unsigned x = __ldg(&g.nontree[e]);
        const int a = (int)(x >> 16), b = (int)(x & 0xFFFFu);
        const int la = lab[a], lb = lab[b];
        if (la != lb && la != kDead16 && lb != kDead16) uf_unite(lab, la, lb);
    }
}

// Component sizes of `listed` nodes (list: their ids, overwritten) of which
// some lie in R's component: returns through *joined (team scalar, zero
// before) the nodes in R's, and this thread's share of the objective over the
// other components.  No union is left; labels of the other components' roots
// become counters.  Starts after a barrier; contains three.
__device__ __forceinline__ long long tree16_list_sizes(const Team& tm, volatile lab_t* lab, lab_t* list, int listed,
                                                       int R, volatile int* joined, int objective) {
    const int tid = tm.tid, T = tm.T, lane = tid & 31;
    int in_r = 0;
    for (int i = tid; i < listed; i += T) {
        const int r = uf_root(lab, list[i]);
        list[i] = (lab_t)r;
        in_r += r == R;
    }
    in_r = __reduce_add_sync(0xffffffffu, in_r);
    if (lane == 0 && in_r) atomicAdd((int*)joined, in_r);
    tm.sync();
    for (int i = tid; i < listed; i += T) {
        const int r = list[i];
        if (r != R) lab[r] = 0;
    }
    tm.sync();
    for (int i0 = tid & ~31; i0 < listed; i0 += T) {
        const int i = i0 + lane, r = i < listed ? list[i] : R;
        const unsigned peers = __match_any_sync(0xffffffffu, r);
        if (r != R && lane == __ffs(peers) - 1) lab_add(lab, r, (unsigned)__popc(peers));
    }
    tm.sync();
    long long acc = 0;
    for (int i = tid; i < listed; i += T) {
        const int r = list[i];
        if (r == R) continue;
        const int c = lab_take(lab, r);  // the first to ask gets the count
        if (c) acc = objective_add(acc, c, objective);
    }
    return acc;
}

// Root of live node v (labels may carry count bits above bit 16).
__device__ __forceinline__ int tree32_root16(volatile int* lab, int v) {
    int x = lab[v] & 0xFFFF;
    while (true) {
        const int q = lab[x] & 0xFFFF;
        if (q == x) return x;
        x = q;
    }
}

// The full pipeline on 32-bit labels (the TREE settings, and members of sparse
// graphs that leave much apart): lab = n labels, dead = (n+31)/32 bitmap words
// followed by four scalars (all in this team's shared memory).  Deleted nodes
// end as -1.
//
// Phases: deletion bitmap; labels (tree parent, or on a deleted parent the
// first live lower-numbered neighbour, or the node itself); flatten every
// piece onto its top node.  The piece of the first live node R is the giant
// candidate: R has no live lower-numbered neighbour, so it is its piece's
// root and the smallest live id, and no union ever hooks it under another
// root.  The live nodes outside R's piece are listed (in the bitmap's words,
// which nothing reads any more) and counted; then the pieces are joined,
// either by letting only the listed nodes scan their adjacency (an edge
// inside R's piece joins nothing) or along every non-tree edge, whichever is
// cheaper (an arc scan costs about half a non-tree edge).  Sizes: only listed nodes can end outside R's
// component, so only they walk to their roots and add themselves into the root slot
// (count << 16 | id); R's component has the other
// live nodes plus the listed ones that reached R.  Without room for the list
// every live node walks and counts.
__device__ __forceinline__ void tree32_member(const Team& tm, volatile int* lab, unsigned* dead, const Tree16Graph& g,
                                              const int* __restrict__ genes, int k, long long* out, long long* red,
                                              int* status) {
    const int tid = tm.tid, T = tm.T, n = g.n, lane = tid & 31;
    const int words = (n + 31) >> 5;
    volatile int* scalar = reinterpret_cast<volatile int*>(dead + words);  // R, mode, list length, live
    for (int w = tid; w < words; w += T) dead[w] = 0u;
    tm.sync();
    // perturbation P^(A, p) of Eq. 13 in BFS numbering
    for (int j = tid; j < k; j += T) {
        const int d = __ldg(&genes[j]);
        if ((unsigned)d < (unsigned)n) {
            const int b = __ldg(&g.perm[d]);
            atomicOr(&dead[b >> 5], 1u << (b & 31));
        } else {
            atomicOr(status, GAPA_DEV_BAD_GENE);
        }
    }
    tm.sync();
    if (tid == 0) {
        int f = -1;
        for (int w = 0; w < words; ++w) {
            const unsigned live = ~dead[w];
            if (live) {
                f = (w << 5) + __ffs(live) - 1;
                break;
            }
        }
        scalar[0] = f < n ? f : -1;
        scalar[2] = 0;
    }
    // labels, four nodes per thread per step
    constexpr int kU = 4;
    for (int base = tid; base < n; base += kU * T) {
        int2 pa[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int v = base + u * T;
            pa[u] = v < n ? __ldg(&g.palt[v]) : make_int2(0, -1);
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int v = base + u * T;
            if (v < n) lab[v] = tree16_pick(dead, g, v, pa[u]);
        }
    }
    tm.sync();
    const int R = scalar[0];
    // flatten (owner writes only) and list the live nodes outside R's piece
    int* list = reinterpret_cast<int*>(dead);
    long long live_out = 0;  // live << 32 | outside
    for (int base = 0; base < n; base += T) {
        const int v = base + tid;
        int r = -1;
        if (v < n) {
            const int p = lab[v];
            if (p != -1) {
                r = p == v ? v : uf_root(lab, p);
                if (p != v) lab[v] = r;
            }
        }
        const bool outside = r >= 0 && r != R;
        live_out += (r >= 0 ? (1ll << 32) : 0) + (outside ? 1 : 0);
        const unsigned m = __ballot_sync(0xffffffffu, outside);
        if (m) {
            int first = 0;
            if (lane == 0) first = atomicAdd((int*)&scalar[2], __popc(m));
            first = __shfl_sync(0xffffffffu, first, 0);
            const int slot = first + __popc(m & ((1u << lane) - 1));
            if (outside && slot < words) list[slot] = v;
        }
    }
    live_out = team_sum_ll(tm, live_out, red);
    if (tid == 0) {
        const long long outside = live_out & 0xFFFFFFFFll;
        // scanning costs about half as much per arc as uniting along a non-tree edge
        const bool scan = g.join_mode == 2 || (g.join_mode == 0 && outside * g.mean_deg_x16 <= 32ll * g.num_nontree);
        scalar[1] = (scan ? 1 : 0) | (outside <= words ? 2 : 0);
        scalar[3] = (int)(live_out >> 32);
    }
    tm.sync();
    const int mode = scalar[1], listed = scalar[2];
    const bool have_list = (mode & 2) != 0;
    const int nw = T >> 5;
    if ((mode & 1) && have_list) {
        // the listed nodes scan their adjacency, 32 per warp step
        for (int i0 = (tid >> 5) * 32; i0 < listed; i0 += nw * 32)
            tree16_scan_warp(lab, g, i0 + lane < listed ? list[i0 + lane] : -1, lane);
    } else if (mode & 1) {
        // the same over every node, skipping the groups of 32 with nobody outside R's piece
        for (int base = (tid >> 5) * 32; base < n; base += nw * 32) {
            const int v = base + lane;
            const int l = v < n ? lab[v] : -1;
            const bool outside = l != -1 && l != R;
            if (!__ballot_sync(0xffffffffu, outside)) continue;
            tree16_scan_warp(lab, g, outside ? v : -1, lane);
        }
    } else {
        // join the pieces along the non-tree edges, four per 16-byte load
        const uint4* e4 = reinterpret_cast<const uint4*>(g.nontree);
        const int quads = g.num_nontree >> 2;
        int q = tid;
        uint4 w = q < quads ? __ldg(&e4[q]) : make_uint4(0, 0, 0, 0);
        while (q < quads) {
            const int qn = q + T;
            const uint4 wn = qn < quads ? __ldg(&e4[qn]) : make_uint4(0, 0, 0, 0);
            const int a0 = (int)(w.x >> 16), b0 = (int)(w.x & 0xFFFFu), a1 = (int)(w.y >> 16), b1 = (int)(w.y & 0xFFFFu);
            const int a2 = (int)(w.z >> 16), b2 = (int)(w.z & 0xFFFFu), a3 = (int)(w.w >> 16), b3 = (int)(w.w & 0xFFFFu);
            const int la0 = lab[a0], lb0 = lab[b0], la1 = lab[a1], lb1 = lab[b1];
            const int la2 = lab[a2], lb2 = lab[b2], la3 = lab[a3], lb3 = lab[b3];
            if (la0 != lb0 && la0 != -1 && lb0 != -1) uf_unite(lab, la0, lb0);
            if (la1 != lb1 && la1 != -1 && lb1 != -1) uf_unite(lab, la1, lb1);
            if (la2 != lb2 && la2 != -1 && lb2 != -1) uf_unite(lab, la2, lb2);
            if (la3 != lb3 && la3 != -1 && lb3 != -1) uf_unite(lab, la3, lb3);
            q = qn;
            w = wn;
        }
        for (int e = quads * 4 + tid; e < g.num_nontree; e += T) {
            const unsigned x = __ldg(&g.nontree[e]);
            const int a = (int)(x >> 16), b = (int)(x & 0xFFFFu);
            const int la = lab[a], lb = lab[b];
            if (la != lb && la != -1 && lb != -1) uf_unite(lab, la, lb);
        }
    }
    tm.sync();
    // sizes: a root's slot becomes (members below it) << 16 | its id; a
    // root's own slot may already carry count bits, so it is classified by
    // the masked id; -1 (deleted) can equal no root slot because root ids are
    // below 65535.
    long long acc = 0;
    if (have_list) {
        long long joined = 0;  // listed nodes whose component is R's
        for (int i = tid; i < listed; i += T) {
            const int v = list[i];
            const int x = tree32_root16(lab, v);
            if (x == R) ++joined;
            else if (x != v) atomicAdd((unsigned*)&lab[x], 1u << 16);
        }
        joined = team_sum_ll(tm, joined, red);
        if (tid == 0) {
            const long long c = (long long)scalar[3] - listed + joined;  // R's component
            acc = objective_add(0, c, g.objective);
        }
        tm.sync();
        for (int i = tid; i < listed; i += T) {
            const int v = list[i];
            const unsigned l = (unsigned)lab[v];
            if ((int)(l & 0xFFFFu) == v) acc = objective_add(acc, (long long)(l >> 16) + 1, g.objective);
        }
    } else {
        // every live non-root walks to its root and adds itself: R's members by
        // one ballot, the other roots grouped with match_any
        for (int base = 0; base < n; base += T) {
            const int v = base + tid;
            int key = -1;
            if (v < n) {
                const int l = lab[v];
                if (l != -1 && (l & 0xFFFF) != v) key = tree32_root16(lab, v);
            }
            const unsigned giant = __ballot_sync(0xffffffffu, key >= 0 && key == R);
            if (giant && lane == 0) atomicAdd((unsigned*)&lab[R], (unsigned)__popc(giant) << 16);
            const bool other = key >= 0 && key != R;
            if (__any_sync(0xffffffffu, other)) {
                const unsigned peers = __match_any_sync(0xffffffffu, other ? key : -1);
                if (other && lane == __ffs(peers) - 1) atomicAdd((unsigned*)&lab[key], (unsigned)__popc(peers) << 16);
            }
        }
        tm.sync();
        for (int v = tid; v < n; v += T) {
            const unsigned l = (unsigned)lab[v];
            if (l != 0xFFFFFFFFu && (int)(l & 0xFFFFu) == v)
                acc = objective_add(acc, (long long)(l >> 16) + 1, g.objective);
        }
    }
    const long long tot = team_sum_ll(tm, acc, red, g.objective != 0);
    if (tid == 0) *out = tot;
}

// The same phases on 16-bit labels, for members that leave the cut-local
// kernel; deleted nodes end as kDead16.  Sizes without room for the list:
// every live node takes its root as label, the roots (marked in the bitmap's
// words) become counters and every other node adds itself.
__device__ __forceinline__ void tree16_member(const Team& tm, volatile lab_t* lab, unsigned* dead, const Tree16Graph& g,
                                              const int* __restrict__ genes, int k, long long* out, long long* red,
                                              int* status) {
    const int tid = tm.tid, T = tm.T, n = g.n, lane = tid & 31;
    const int words = (n + 31) >> 5;
    volatile int* scalar = reinterpret_cast<volatile int*>(dead + words);  // R, mode or joined, list length, live
    for (int w = tid; w < words; w += T) dead[w] = 0u;
    tm.sync();
    // perturbation P^(A, p) of Eq. 13 in BFS numbering
    for (int j = tid; j < k; j += T) {
        const int d = __ldg(&genes[j]);
        if ((unsigned)d < (unsigned)n) {
            const int b = __ldg(&g.perm[d]);
            atomicOr(&dead[b >> 5], 1u << (b & 31));
        } else {
            atomicOr(status, GAPA_DEV_BAD_GENE);
        }
    }
    tm.sync();
    if (tid == 0) {
        int f = -1;
        for (int w = 0; w < words; ++w) {
            const unsigned live = ~dead[w];
            if (live) {
                f = (w << 5) + __ffs(live) - 1;
                break;
            }
        }
        scalar[0] = f < n ? f : -1;
        scalar[2] = 0;
    }
    // labels, four nodes per thread per step
    constexpr int kU = 4;
    for (int base = tid; base < n; base += kU * T) {
        int2 pa[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int v = base + u * T;
            pa[u] = v < n ? __ldg(&g.palt[v]) : make_int2(0, -1);
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int v = base + u * T;
            if (v < n) lab[v] = (lab_t)tree16_pick(dead, g, v, pa[u]);  // -1 becomes kDead16
        }
    }
    tm.sync();
    const int R = scalar[0];
    // flatten (owner writes only) and list the live nodes outside R's piece
    lab_t* list = reinterpret_cast<lab_t*>(dead);
    const int cap = 2 * words;
    long long live_out = 0;  // live << 32 | outside
    for (int base = 0; base < n; base += T) {
        const int v = base + tid;
        int r = -1;
        if (v < n) {
            const int p = lab[v];
            if (p != kDead16) {
                r = p == v ? v : uf_root(lab, p);
                if (p != v) lab[v] = (lab_t)r;
            }
        }
        const bool outside = r >= 0 && r != R;
        live_out += (r >= 0 ? (1ll << 32) : 0) + (outside ? 1 : 0);
        const unsigned m = __ballot_sync(0xffffffffu, outside);
        if (m) {
            int first = 0;
            if (lane == 0) first = atomicAdd((int*)&scalar[2], __popc(m));
            first = __shfl_sync(0xffffffffu, first, 0);
            const int slot = first + __popc(m & ((1u << lane) - 1));
            if (outside && slot < cap) list[slot] = (lab_t)v;
        }
    }
    live_out = team_sum_ll(tm, live_out, red);
    if (tid == 0) {
        const long long outside = live_out & 0xFFFFFFFFll;
        // scanning costs about half as much per arc as uniting along a non-tree edge
        const bool scan = g.join_mode == 2 || (g.join_mode == 0 && outside * g.mean_deg_x16 <= 32ll * g.num_nontree);
        scalar[1] = (scan ? 1 : 0) | (outside <= cap ? 2 : 0);
        scalar[3] = (int)(live_out >> 32);
    }
    tm.sync();
    const int mode = scalar[1], listed = scalar[2], live = scalar[3];
    const bool have_list = (mode & 2) != 0;
    const int nw = T >> 5;
    if ((mode & 1) && have_list) {
        // the listed nodes scan their adjacency, 32 per warp step
        for (int i0 = (tid >> 5) * 32; i0 < listed; i0 += nw * 32)
            tree16_scan_warp(lab, g, i0 + lane < listed ? list[i0 + lane] : -1, lane);
    } else if (mode & 1) {
        // the same over every node, skipping the groups of 32 with nobody outside R's piece
        for (int base = (tid >> 5) * 32; base < n; base += nw * 32) {
            const int v = base + lane;
            const int l = v < n ? lab[v] : kDead16;
            const bool outside = l != kDead16 && l != R;
            if (!__ballot_sync(0xffffffffu, outside)) continue;
            tree16_scan_warp(lab, g, outside ? v : -1, lane);
        }
    } else {
        tree16_join_nontree(tm, lab, g);  // join the pieces along the non-tree edges
    }
    tm.sync();
    if (tid == 0) scalar[1] = 0;  // (every thread has read the mode)
    long long acc = 0;
    if (have_list) {
        tm.sync();
        acc = tree16_list_sizes(tm, lab, list, listed, R, &scalar[1], g.objective);
        if (tid == 0 && live) acc = objective_add(acc, (long long)live - listed + scalar[1], g.objective);
    } else {
        for (int v = tid; v < n; v += T) {
            const int l = lab[v];
            if (l == kDead16 || l == v) continue;
            const int r = uf_root(lab, l);
            if (r != l) lab[v] = (lab_t)r;
        }
        tm.sync();
        for (int base = 0; base < n; base += T) {
            const int v = base + tid;
            const bool root = v < n && lab[v] == v;
            const unsigned m = __ballot_sync(0xffffffffu, root);
            if (lane == 0 && v < n) dead[v >> 5] = m;
            if (root) lab[v] = 0;
        }
        tm.sync();
        // every live non-root adds itself: R's members by one ballot, the other roots grouped with match_any
        for (int base = 0; base < n; base += T) {
            const int v = base + tid;
            int key = -1;
            if (v < n && !bm_test(dead, v)) {
                const int l = lab[v];
                if (l != kDead16) key = l;
            }
            const unsigned giant = __ballot_sync(0xffffffffu, key >= 0 && key == R);
            if (giant && lane == 0) lab_add(lab, R, (unsigned)__popc(giant));
            const bool other = key >= 0 && key != R;
            if (__any_sync(0xffffffffu, other)) {
                const unsigned peers = __match_any_sync(0xffffffffu, other ? key : -1);
                if (other && lane == __ffs(peers) - 1) lab_add(lab, key, (unsigned)__popc(peers));
            }
        }
        tm.sync();
        for (int v = tid; v < n; v += T)
            if (bm_test(dead, v)) acc = objective_add(acc, (long long)lab[v] + 1, g.objective);
    }
    const long long tot = team_sum_ll(tm, acc, red, g.objective != 0);
    if (tid == 0) *out = tot;
}

// Helpers shared with the other fitness kernels.
// Exclusive prefix sum of v over the team in thread order; *total = the sum.
// ws: 32 ints of team scratch, free again after the caller's next barrier.
// Contains two team barriers.
__device__ __forceinline__ int tree16l_scan(const Team& tm, int v, int* ws, int* total) {
    const int lane = tm.tid & 31, warp = tm.tid >> 5, nw = tm.T >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) ws[warp] = incl;
    tm.sync();
    if (warp == 0) {
        int x = lane < nw ? ws[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane < nw) ws[lane] = x;
    }
    tm.sync();
    *total = ws[nw - 1];
    return (warp ? ws[warp - 1] : 0) + incl - v;
}

// The owner of item i among `owners` owners with exclusive offsets off[]:
// the last owner whose offset is at most i (owners without items share the
// next one's offset and come before it).
__device__ __forceinline__ int tree16l_owner(const int* off, int owners, int i) {
    int lo = 0, hi = owners - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ---------------------------------------------------------------------------
// Cut-local variant.  Same fitness as tree16_member, with work proportional
// to what the deletion disturbs instead of to n:
//  * the tree-parent array (16-bit) is copied into the labels by one bulk copy
//    (cp.async.bulk, completion on an mbarrier), so every live node whose
//    parent is live already holds a link of its piece;
//  * a gene costs one 8-byte read: its number and its children ("tops"),
//    consecutive numbers that go into a list while the copy is in flight;
//  * every live top takes its first live neighbour among four of its lower-
//    numbered ones as label (one 8-byte read); the tops without one
//    ("terminals") are united with up to two live higher-numbered neighbours
//    outside their own piece.  Any such links are exact - they only join what
//    an edge joins - and these leave little apart: with 1000 of 20000 nodes
//    deleted, 0 to 450 nodes on Barabasi-Albert and Holme-Kim graphs (4 links
//    per node) whatever share of the deleted ones are hubs, where the first
//    live neighbour alone leaves up to 16,000.  (Uniting every top with a
//    second neighbour leaves under 150, but its walks over the labels made the
//    kernel four times slower on hub-heavy members, bound by shared-memory
//    bandwidth.);
//  * R, the reference, is the root that most of a few live nodes reach; the
//    terminals and component roots that took no other's label and are not R are
//    the roots of the classes apart from R's.  From them a breadth-first search
//    over live arcs lists those classes: a neighbour in R's class joins the
//    node's class to R (which then needs no more), any other is united with it
//    and listed.  What is not listed lies in R's class; the sizes of the others
//    are counted on the list.
// Single-node components of G are kept out of all this: they add nothing to
// PC, and 1 to MCN.
// A member with repeated genes, or whose tops or list outgrow its region, or
// whose list outgrows a quarter of the graph or kLocalLevels rounds, runs
// the full pipeline, at up to twice that pipeline's time.  (The list of a graph
// without communities stays below: 0.11 n on Barabasi-Albert and Holme-Kim
// graphs with an eighth of the nodes deleted, up to all of them hubs, 0.16 n on
// G(n, M) of mean degree 3; small-world and community graphs lose 2 to 3
// members of 40 there.  Half of the graph as the limit made these 1.2 to 1.5
// times slower, a look at the share apart half-way through 1.3 to 1.9.)  On
// sparse graphs (mean degree below 5) a member with more than n / 5 tops, which
// leaves thousands of nodes apart, runs tree32_member from the start (2 links
// per node, n = 12000, 100 hub-heavy members of 600 genes: 107 us without;
// local_layout.cuh has other shares).
//
// What bounds it: instruction issue and shared-memory reads (55 % and 43 % of
// peak on hub-heavy members, 45 % and 31 % on random ones), and the chain of about ten short phases between
// team barriers, each one or two L2 reads deep; so members in flight per SM
// count most, which 16-bit labels serve.  Measured, 1023 members of 1000 genes
// at n = 20000 (kernel): random 86 us before (32-bit labels, listing down the
// tree, two forests), 35 us now; hub-heavy 209 us before, 75 us now.  Steps on
// the hub-heavy ones: every top united with two neighbours 190 us, links found
// in a dense list of terminals 118, breadth-first search instead of a walk from
// every top to its root 75; every node labelled with its root once there are
// many classes 80.

constexpr int kLocalLevels = 256;
constexpr long long kLocalSpinLimit = 1ll << 24;

__device__ __forceinline__ unsigned tree16l_smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool tree16l_wait(unsigned bar, unsigned parity) {
    for (long long i = 0; i < kLocalSpinLimit; ++i) {
        unsigned done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// Append of a node to the 16-bit list, marking it in the listed-node bitmap;
// entries past cap are dropped (the caller sees the count exceed cap).
__device__ __forceinline__ void tree16l_append(int val, volatile int* count, lab_t* list, int cap, unsigned* listed_bm) {
    const int slot = atomicAdd((int*)count, 1);
    if (slot < cap) {
        list[slot] = (lab_t)val;
        atomicOr(&listed_bm[val >> 5], 1u << (val & 31));
    }
}

// lab: the member's labels; region: its list region (g.list_bytes); scal_base:
// its twelve scalars followed by the mbarrier.  0: the result is in *out, as
// from tree16_member; 1: the member needs the full pipeline; 2: it needs it on
// 32-bit labels.
__device__ __forceinline__ int tree16_local_try(const Team& tm, volatile lab_t* lab, unsigned* region, int* scal_base,
                                                const Tree16Graph& g, const int* __restrict__ genes, int k,
                                                long long* out, long long* red, int* status) {
    const int tid = tm.tid, T = tm.T, n = g.n, lane = tid & 31;
    // 0 R, 1 list length, 2 tops, 3 distinct genes, 4 repeated genes, 5 deleted single-node components,
    // 6 the copy's wait ran out, 8 terminals, 9 listed nodes that joined R
    volatile int* scalar = scal_base;
    const unsigned bar_a = tree16l_smem_u32(scal_base + 12);
    const int bm_bytes = (int)tree16l_bitmap_bytes(n), words = (n + 31) >> 5;
    lab_t* list = reinterpret_cast<lab_t*>(region);
    unsigned* listed_bm = reinterpret_cast<unsigned*>(reinterpret_cast<char*>(region) + g.list_bytes - bm_bytes);
    const int cap = (g.list_bytes - bm_bytes) >> 1;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_a) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 12) scalar[tid] = 0;
    for (int w = tid; w < words; w += T) listed_bm[w] = 0u;
    tm.sync();
    if (tid == 0) {
        // labels <- tree parents, in chunks of 2 KB from a start that differs from team to team, so that the
        // teams starting together do not ask the same L2 slices for the same lines (the fence orders this
        // team's earlier generic-proxy use of the labels before the async-proxy writes)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        const unsigned bytes = (unsigned)tree16_lab_bytes(n), chunk = 2048u, chunks = (bytes + chunk - 1) / chunk;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_a), "r"(bytes) : "memory");
        const unsigned dst = tree16l_smem_u32((const void*)lab);
        unsigned o = (blockIdx.x * 7u + (unsigned)tm.bar * 3u) % chunks * chunk;
        for (unsigned i = 0; i < chunks; ++i) {
            const unsigned len = bytes - o < chunk ? bytes - o : chunk;
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                    dst + o),
                "l"(reinterpret_cast<const char*>(g.cut.par) + o), "r"(len), "r"(bar_a)
                : "memory");
            o = o + chunk < bytes ? o + chunk : 0u;
        }
    }
    // perturbation P^(A, p) of Eq. 13 in BFS numbering: the deleted nodes' labels, and their children listed
    bool waited = false, ok = true;
    int fresh = 0, repeated = 0, singles = 0;
    for (int j0 = tid & ~31; j0 < k; j0 += T) {
        const int j = j0 + lane;
        uint2 rec = make_uint2(kDead16, 0u);
        if (j < k) {
            const int d = __ldg(&genes[j]);
            if ((unsigned)d < (unsigned)n) rec = __ldg(&g.cut.gene[d]);
            else atomicOr(status, GAPA_DEV_BAD_GENE);
        }
        if (!waited) {  // the labels must have landed before anyone marks them
            ok = tree16l_wait(bar_a, 0u);
            waited = true;
        }
        const int b = (int)(rec.x & 0xFFFFu), first = (int)(rec.x >> 16), sh = (b & 1) * 16;
        int cnt = 0;
        if (b != kDead16) {
            const unsigned old = atomicOr(lab_word(lab, b), 0xFFFFu << sh);
            if (((old >> sh) & 0xFFFFu) == 0xFFFFu) {
                ++repeated;
            } else {
                ++fresh;
                singles += (int)(rec.y >> 16);
                cnt = (int)(rec.y & 0xFFFFu);
            }
        }
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        int at = 0;
        if (lane == 31 && incl) at = atomicAdd((int*)&scalar[2], incl);
        at = __shfl_sync(0xffffffffu, at, 31) + incl - cnt;
        const bool many = cnt >= 16;
        if (!many)
            for (int i = 0; i < cnt; ++i)
                if (at + i < cap) list[at + i] = (lab_t)(first + i);
        for (unsigned m = __ballot_sync(0xffffffffu, many); m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            const int c = __shfl_sync(0xffffffffu, cnt, src), f = __shfl_sync(0xffffffffu, first, src),
                      a = __shfl_sync(0xffffffffu, at, src);
            for (int i = lane; i < c; i += 32)
                if (a + i < cap) list[a + i] = (lab_t)(f + i);
        }
    }
    if (!waited) ok = tree16l_wait(bar_a, 0u);
    if (!ok) {
        atomicOr(status, GAPA_DEV_TIMEOUT);
        tree16l_wait(bar_a, 0u);  // bounded: the copy may still be in flight
        scalar[6] = 1;
    }
    fresh = __reduce_add_sync(0xffffffffu, fresh);
    repeated = __reduce_add_sync(0xffffffffu, repeated);
    singles = __reduce_add_sync(0xffffffffu, singles);
    if (lane == 0) {
        if (fresh) atomicAdd((int*)&scalar[3], fresh);
        if (repeated) atomicAdd((int*)&scalar[4], repeated);
        if (singles) atomicAdd((int*)&scalar[5], singles);
    }
    tm.sync();
    if (scalar[6]) {
        if (tid == 0) *out = -1;
        return 0;
    }
    // the copy has landed: the mbarrier's memory may be reused
    if (tid == 0) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar_a) : "memory");
    const int tops = scalar[2], live = n - scalar[3], live_singles = g.cut.singles - scalar[5];
    if (scalar[4]) return 1;  // repeated genes
    if (live == live_singles) {  // nothing, or single nodes only
        if (tid == 0) *out = g.objective && live ? 1 : 0;
        return 0;
    }
    if (tops > g.tops_max) return 2;
    if (tops > cap - cap / 8) return 1;  // (the rest is room for terminals)
    // every live top: its first live lower-numbered neighbour, else itself (a "terminal", listed downwards
    // from the list's end)
    lab_t* const term = list + cap - 1;
    const int term_cap = cap - tops;
    for (int i = tid; i < tops; i += T) {
        const int c = list[i];
        if (lab[c] == kDead16) continue;
        const uint2 l = __ldg(&g.cut.lower[c]);
        const unsigned x[4] = {l.x & 0xFFFFu, l.x >> 16, l.y & 0xFFFFu, l.y >> 16};
        int p = c;
#pragma unroll
        for (int e = 3; e >= 0; --e)
            if (x[e] != kDead16 && lab[x[e]] != kDead16) p = (int)x[e];
        lab[c] = (lab_t)p;
        if (p == c) {
            const int at = atomicAdd((int*)&scalar[8], 1);
            if (at < term_cap) term[-at] = (lab_t)c;
        }
    }
    if ((tid >> 5) == 0) {
        // R = the first live node, two labels per lane and step
        int f = -1;
        for (int w0 = 0; f < 0; w0 += 32) {
            unsigned x = 0xFFFFFFFFu;
            if (2 * (w0 + lane) < n) x = *(volatile unsigned*)lab_word(lab, 2 * (w0 + lane));
            const bool lo = (x & 0xFFFFu) != 0xFFFFu, hi = (x >> 16) != 0xFFFFu && 2 * (w0 + lane) + 1 < n;
            const unsigned m = __ballot_sync(0xffffffffu, lo || hi);
            if (m) f = 2 * (w0 + __ffs(m) - 1) + (__shfl_sync(0xffffffffu, (int)lo, __ffs(m) - 1) ? 0 : 1);
        }
        if (lane == 0) scalar[0] = f;
    }
    tm.sync();
    // the terminals unite with up to two live higher-numbered neighbours outside their own piece
    int R = scalar[0];
    const int terms = scalar[8];
    if (terms > term_cap) return 1;
    for (int i = tid; i < terms; i += T) {
        const int c = term[-i];
        const uint2 l = __ldg(&g.cut.higher[c]);
        const unsigned x[4] = {l.x & 0xFFFFu, l.x >> 16, l.y & 0xFFFFu, l.y >> 16};
        int links = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (x[e] != kDead16 && links < 2 && lab[x[e]] != kDead16) {
                uf_unite(lab, c, (int)x[e]);
                ++links;
            }
    }
    tm.sync();
    // with the top hub deleted, the first live node may lie in a small class: the reference becomes the
    // root that most of 32 spread-out live nodes reach
    if (R != 0) {
        if ((tid >> 5) == 0) {
            int v = (int)(((long long)n * (2 * lane + 1)) >> 6);
            for (int step = 0; step < 8 && lab[v] == kDead16; ++step) v = v + 1 < n ? v + 1 : 0;
            const int r = lab[v] == kDead16 ? R : uf_root(lab, v);
            const unsigned peers = __match_any_sync(0xffffffffu, r);
            const unsigned best = __reduce_max_sync(0xffffffffu, (unsigned)__popc(peers) << 16 | (unsigned)r);
            if (lane == 0) scalar[0] = (int)(best & 0xFFFFu);
        }
        tm.sync();
        R = scalar[0];
    }
    // the roots of the classes apart from R's - terminals and component roots that took no other's label -
    // seed the list (over the tops, which nothing reads any more, up to the terminals)
    const int seed_cap = cap - terms;
    for (int i = tid; i < terms; i += T) {
        const int c = term[-i];
        if (c != R && lab[c] == c) tree16l_append(c, &scalar[1], list, seed_cap, listed_bm);
    }
    for (int i = tid; i < g.cut.num_roots; i += T) {
        const int rho = __ldg(&g.cut.roots[i]);
        if (rho != R && lab[rho] == rho) tree16l_append(rho, &scalar[1], list, seed_cap, listed_bm);
    }
    tm.sync();
    const long long others = (long long)live - live_singles;
    int tail = scalar[1];
    if (tail == 0) {  // one class
        if (tid == 0) *out = objective_add(0, others, g.objective);
        return 0;
    }
    // breadth first from the seeds over live arcs, four lanes per node (eight from a mean degree of 6 on): a
    // neighbour in R's class joins the node's class to R, any other is united with it and listed.  Every
    // node of a class that stays apart is listed, and so are its arcs taken; a class that joins R needs no
    // more.
    const int sh = g.mean_deg_x16 < 96 ? 2 : 3, sub = tid & ((1 << sh) - 1);
    int head = 0, level = 0;
    const int lim = min(cap, max(n / 4, 1024));
    if (tail > seed_cap) tail = lim + 1;  // seeds were dropped
    while (head < tail && tail <= lim && level < kLocalLevels) {
        tm.sync();  // every thread has read the length before the round appends
        for (int i = head + (tid >> sh); i < tail; i += T >> sh) {
            const int v = list[i];
            int w = __ldg(&g.cut.near[8 * v + sub]);
            const int e0 = __ldg(&g.fptr[v]), e1 = __ldg(&g.fptr[v + 1]);
            if (uf_find(lab, v) == R) continue;
            for (int e = e0 + sub; e < e1;) {
                const int lw = lab[w];
                if (lw != kDead16) {
                    const unsigned bit = 1u << (w & 31);
                    const bool below = lw == v;  // hangs on v: v's class, without a walk
                    if (!bm_test(listed_bm, w)) {
                        if (!below && uf_find(lab, w) == R) {
                            uf_unite(lab, v, R, R);
                            break;
                        }
                        if (!(atomicOr(&listed_bm[w >> 5], bit) & bit)) {
                            if (below) lab[w] = lab[v];
                            const int at = atomicAdd((int*)&scalar[1], 1);
                            if (at < cap) list[at] = (lab_t)w;
                        }
                    }
                    if (!below && lab[w] != lab[v]) uf_unite(lab, v, w, R);
                }
                e += 1 << sh;
                if (e < e1) w = __ldg(&g.fcol[e]);
            }
        }
        tm.sync();
        head = tail;
        tail = scalar[1];
        ++level;
    }
    if (tail > lim || head < tail) return 1;  // the list too long or too deep
    const int listed = tail;
    const long long outer = others - listed;  // plus the listed nodes that joined R
    if (listed <= 32) {  // one warp counts by matching roots
        if ((tid >> 5) == 0) {
            const int r = lane < listed ? uf_root(lab, list[lane]) : -1;
            const unsigned peers = __match_any_sync(0xffffffffu, r);
            const int in_r = __popc(__ballot_sync(0xffffffffu, r == R));
            long long acc = 0;
            if (r >= 0 && r != R && lane == __ffs(peers) - 1) acc = objective_add(0, __popc(peers), g.objective);
            if (lane == 0) acc = objective_add(acc, outer + in_r, g.objective);
            for (int o = 16; o > 0; o >>= 1) {
                const long long x = __shfl_down_sync(0xffffffffu, acc, o);
                acc = g.objective ? (x > acc ? x : acc) : acc + x;
            }
            if (lane == 0) *out = acc;
        }
        return 0;
    }
    long long acc = tree16_list_sizes(tm, lab, list, listed, R, &scalar[9], g.objective);
    if (tid == 0) acc = objective_add(acc, outer + scalar[9], g.objective);
    const long long tot = team_sum_ll(tm, acc, red, g.objective != 0);
    if (tid == 0) *out = tot;
    return 0;
}

// The full pipeline where it has to be: on 32-bit labels wherever the region holds them (15 to 30 % faster than
// on 16-bit ones).  One place for all that need it keeps the kernel within its 32 registers without a spill
// (inlined at five places: 12 bytes spilled, 84 reloaded; whole small runs 2 % slower).
__device__ __forceinline__ void tree16_member_local(const Team& tm, volatile lab_t* lab, unsigned* region,
                                                    int* scal_base, const Tree16Graph& g,
                                                    const int* __restrict__ genes, int k, long long* out,
                                                    long long* red, int* status) {
    const int full = tree16_local_try(tm, lab, region, scal_base, g, genes, k, out, red, status);
    if (full == 0) return;
    tm.sync();
    if (full == 2 || tree16_lab_bytes(g.n) + (size_t)g.list_bytes >= tree32_smem_bytes(g.n)) {
        int* lab32 = reinterpret_cast<int*>(const_cast<lab_t*>(lab));
        tree32_member(tm, lab32, reinterpret_cast<unsigned*>(lab32 + g.n), g, genes, k, out, red, status);
    } else {
        tree16_member(tm, lab, region, g, genes, k, out, red, status);
    }
}
}  // namespace gapa_dev
