// split.cu -- the split step of GSP-Louvain (Section 4.1): break every
// community into the connected components of its intra-community edges.
//
//   LP  (Algorithm 2): labels start at the vertex id; every sweep each vertex
//        takes the minimum label over its same-community neighbours, in place,
//        until a sweep changes nothing.  Labels only decrease, so the in-place
//        updates of concurrent threads converge to the same fixpoint.
//   LPP (Algorithm 2 with pruning) and SV (hooking and shortcutting on the
//        intra-community edges, not in the paper) both run as one hooking
//        pass: a disjoint-set forest over the vertices whose roots are the
//        smallest id of their set, which is the fixpoint that pruned label
//        propagation reaches round by round.
//   BFS (Algorithm 3): rounds of multi-source, level-synchronous,
//        frontier-compacted BFS.  In each round the seed of a community is its
//        smallest unvisited vertex, found with atomicMin; vertices are claimed
//        with atomicCAS on their label.  The busy flags of the paper's
//        per-thread BFS become unnecessary: every community is searched from
//        one seed per round by the whole GPU.
// The seed of a round is the smallest vertex of its component (the smaller
// vertices of the community are already visited, and components are
// disjoint), so every mode yields label = smallest vertex id of the component.
#include <algorithm>

#include "internal.cuh"

namespace gsp {

template <typename T> __device__ __forceinline__ T ldcg_(const T *p) { return __ldcg(p); }
__device__ __forceinline__ uint8_t ldcg_(const uint8_t *p) {
    return (uint8_t)__ldcg(reinterpret_cast<const unsigned char *>(p));
}

// min over the same-community neighbours' labels of the edges b + first,
// b + first + step, ... < e; four gathers of C and lab in flight per thread.
__device__ __forceinline__ uint32_t min_label(const uint32_t *__restrict__ tgt, const uint32_t *__restrict__ C,
                                              const uint32_t *lab, uint32_t ci, uint64_t b, uint64_t e,
                                              uint32_t first, uint32_t step, uint32_t mn) {
    uint64_t p = b + first;
    for (; p + 3 * (uint64_t)step < e; p += 4 * (uint64_t)step) {
        uint32_t j[4], cj[4];
#pragma unroll
        for (int u = 0; u < 4; u++) j[u] = tgt[p + (uint64_t)u * step];
#pragma unroll
        for (int u = 0; u < 4; u++) cj[u] = C[j[u]];
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (cj[u] == ci) mn = min(mn, ldcg_(lab + j[u]));
    }
    for (; p < e; p += step) {
        const uint32_t j = tgt[p];
        if (C[j] == ci) mn = min(mn, ldcg_(lab + j));
    }
    return mn;
}

// ------------------------------------------------------------------------ LP
template <int G>
__global__ void __launch_bounds__(256) k_lp_group(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tgt,
                                                  const uint32_t *__restrict__ C, uint32_t *lab,
                                                  const uint32_t *__restrict__ list, uint32_t count,
                                                  unsigned long long *changed) {
    const int lane = threadIdx.x % G;
    const unsigned gmask = (G == 32) ? 0xFFFFFFFFu : (((1u << G) - 1u) << ((threadIdx.x & 31) & ~(G - 1)));
    unsigned long long ch = 0;
    for (uint64_t q = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) / G; q < count;
         q += (uint64_t)gridDim.x * blockDim.x / G) {
        const uint32_t i = list[q];
        const uint32_t cur = ldcg_(lab + i);
        uint32_t mn = min_label(tgt, C, lab, C[i], off[i], off[i + 1], lane, G, cur);
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) mn = min(mn, __shfl_xor_sync(gmask, mn, o));
        if (mn < cur && lane == 0) {
            lab[i] = mn;
            ch++;
        }
        __syncwarp(gmask);
    }
    __shared__ unsigned long long red[32];
    ch = block_sum(ch, red);
    if (threadIdx.x == 0 && ch) atomicAdd(changed, ch);
}

__global__ void __launch_bounds__(256) k_lp_block(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tgt,
                                                  const uint32_t *__restrict__ C, uint32_t *lab,
                                                  const uint32_t *__restrict__ list, uint32_t count,
                                                  unsigned long long *changed) {
    __shared__ uint32_t red[32];
    unsigned long long ch = 0;
    for (uint32_t q = blockIdx.x; q < count; q += gridDim.x) {
        const uint32_t i = list[q];
        __syncthreads();  // previous vertex done with red
        const uint32_t cur = ldcg_(lab + i);
        uint32_t mn = min_label(tgt, C, lab, C[i], off[i], off[i + 1], threadIdx.x, blockDim.x, cur);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mn = min(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, o));
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mn;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int t = 1; t < (int)(blockDim.x >> 5); t++) mn = min(mn, red[t]);
            if (mn < cur) {
                lab[i] = mn;
                ch++;
            }
        }
    }
    if (threadIdx.x == 0 && ch) atomicAdd(changed, ch);
}

static void split_lp(const DevGraph &g, const Classes &cl, const uint32_t *C, uint32_t *lab, cudaStream_t s) {
    size_t mk = arena().mark();
    unsigned long long *changed = arena().get<unsigned long long>(1);
    iota_u32(lab, g.n, s);
    // every class with all its waves (class c spans [cls_begin(c), cls_begin(c+1)))
    auto cnt = [&](int c) { return cl.cls_count(c); };
    auto lst = [&](int c) { return cl.list + cl.cls_begin(c); };
    const unsigned maxg = sms(8);
    const uint32_t nbig = cl.cls_count(CLS_BLOCK) + cl.cls_count(CLS_BIG) + cl.cls_count(CLS_HUGE);
    for (int it = 0; it < (1 << 30); it++) {
        GSP_CUDA(cudaMemsetAsync(changed, 0, sizeof(unsigned long long), s));
#define LPG(G, CLS)                                                                                            \
    if (cnt(CLS)) {                                                                                            \
        k_lp_group<G><<<grid_for((uint64_t)cnt(CLS) * G, 256, maxg), 256, 0, s>>>(g.off, g.tgt, C, lab, lst(CLS), \
                                                                                  cnt(CLS), changed);          \
        GSP_CHECK_LAUNCH();                                                                                    \
    }
        LPG(4, CLS_G4) LPG(8, CLS_G8) LPG(16, CLS_G16) LPG(32, CLS_G32) LPG(32, CLS_W512)
#undef LPG
        if (nbig) {
            k_lp_block<<<grid_for(nbig, 1, sms(4)), 256, 0, s>>>(g.off, g.tgt, C, lab, lst(CLS_BLOCK), nbig, changed);
            GSP_CHECK_LAUNCH();
        }
        unsigned long long h;
        GSP_CUDA(cudaMemcpyAsync(&h, changed, sizeof(h), cudaMemcpyDeviceToHost, s));
        GSP_CUDA(cudaStreamSynchronize(s));
        if (h == 0) break;
    }
    arena().release(mk);
}

// ------------------------------------------------------------- hooking split
// Disjoint-set forest over the vertices, parents in lab: every set is a tree
// whose pointers lead to smaller ids, so its root is its smallest vertex and
// after the last link lab (pointing at the roots) holds the split's labels.
// Links hook the larger root under the smaller by compare-and-swap; finds
// halve the path as they go.  Both may run on stale values: only a root is
// ever hooked, a stored parent is always an earlier ancestor (a smaller id of
// the same set), and a failed hook returns the parent it lost to, so that a
// link's larger end falls with every attempt.
//
// Label propagation read every edge and both ends' C in each of its rounds
// (a round trip to the host between them); one pass of links over all edges
// would read them once.  Most edges need not be read at all (the sampling of
// Sutton, Ben-Nun and Barak's Afforest, per community): after linking each
// vertex with the first few of its row, nearly every community already is one
// tree.  The vertices of one tree per community (`tree`: whichever vertex
// wrote last, likely of the largest) need no further look: an edge inside the
// tree is redundant, and an edge that leaves it is linked from its other end.
// Everyone else links along the whole row.  A vertex that joins the tree while
// the links run may be skipped too: its edges then lead into the tree or to
// vertices that link them.
// On R-MAT 22 the sample leaves 3 % of the vertices and 5 % of the edges to
// the row pass (4 entries instead of 8: 12 and 16 %).
// Measured (all splits of a call, ms, rounds of pruned propagation -> this):
// R-MAT 22 4.7 -> 1.0, R-MAT 24 17.6 -> 3.5, 2048^2 grid 3.4 -> 1.2, 512 planted
// graphs 8.1 -> 2.2, 611 vertices 0.38 -> 0.18.  With rows up to 4096 entries
// left to a warp, R-MAT 22 took 4.4: its hubs have neighbouring ids and queued
// in the same warps.
constexpr uint32_t HOOK_SAMPLE = 8;   // entries of a row linked in the sampling pass
constexpr uint32_t HOOK_MID = 256;    // longer rows are linked by a block each ...
constexpr uint32_t HOOK_HUB = 16384;  // ... or by a column of HOOK_COL blocks
constexpr uint32_t HOOK_COL = 16;

struct HookLists {  // open rows longer than HOOK_MID: one array filled from both ends
    uint32_t *rows, *nmid, *nhub;
    uint32_t cap;
};

__device__ __forceinline__ uint32_t hook_find(uint32_t *lab, uint32_t x) {
    uint32_t p = __ldca(lab + x);
    while (p != x) {
        const uint32_t g = __ldca(lab + p);
        if (g == p) return p;
        lab[x] = g;
        x = g;
        p = __ldca(lab + x);
    }
    return x;
}

// Link the trees of two roots; returns the smaller one met last.
__device__ __forceinline__ uint32_t hook_link(uint32_t *lab, uint32_t u, uint32_t v) {
    while (u != v) {
        if (u < v) {
            const uint32_t t = u;
            u = v;
            v = t;
        }
        const uint32_t old = atomicCAS(lab + u, u, v);
        if (old == u) return v;
        u = hook_find(lab, old);
    }
    return u;
}

// Link vertex i with the same-community targets of entries p, p + step, ... < e,
// four gathers of C in flight.
__device__ __forceinline__ void hook_row(const uint32_t *__restrict__ tgt, const uint32_t *__restrict__ C,
                                         uint32_t *lab, uint32_t i, uint32_t ci, uint64_t p, uint64_t e,
                                         uint32_t step) {
    uint32_t r = EMPTY;
    for (; p < e; p += 4ull * step) {
        uint32_t j[4], cj[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const uint64_t q = p + (uint64_t)u * step;
            j[u] = q < e ? __ldg(tgt + q) : i;
        }
#pragma unroll
        for (int u = 0; u < 4; u++) cj[u] = __ldg(C + j[u]);
#pragma unroll
        for (int u = 0; u < 4; u++) {
            if (j[u] == i || cj[u] != ci) continue;
            if (r == EMPTY) r = hook_find(lab, i);
            r = hook_link(lab, r, hook_find(lab, j[u]));
        }
    }
}

__global__ void __launch_bounds__(256) k_hook_sample(const uint64_t *__restrict__ off,
                                                     const uint32_t *__restrict__ tgt,
                                                     const uint32_t *__restrict__ C, uint32_t n, uint32_t *lab) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint64_t b = off[i];
        const uint32_t k = (uint32_t)min(off[i + 1] - b, (uint64_t)HOOK_SAMPLE), ci = C[i];
        uint32_t j[HOOK_SAMPLE], cj[HOOK_SAMPLE];
#pragma unroll
        for (uint32_t u = 0; u < HOOK_SAMPLE; u++) j[u] = u < k ? __ldg(tgt + b + u) : i;
#pragma unroll
        for (uint32_t u = 0; u < HOOK_SAMPLE; u++) cj[u] = __ldg(C + j[u]);
        uint32_t r = EMPTY;
#pragma unroll
        for (uint32_t u = 0; u < HOOK_SAMPLE; u++) {
            if (j[u] == i || cj[u] != ci) continue;
            if (r == EMPTY) r = hook_find(lab, i);
            r = hook_link(lab, r, hook_find(lab, j[u]));
        }
    }
}

// Point every vertex at its root; tree (optional): a root of each community.
// Read-only finds: a halving store could land on a vertex already finished.
__global__ void __launch_bounds__(256) k_hook_compress(const uint32_t *__restrict__ C, uint32_t n, uint32_t *lab,
                                                       uint32_t *tree) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        uint32_t r = __ldca(lab + i);
        for (uint32_t p; (p = __ldca(lab + r)) != r;) r = p;
        lab[i] = r;
        if (tree) tree[C[i]] = r;
    }
}

// Link the rows of the vertices outside their community's tree (of all
// vertices when there is no room for the trees and lists: h.rows null): a
// warp reads 32 vertices' state at once and takes the open ones in turn.
// Long rows are listed, so that neighbouring hubs do not queue in one warp.
__global__ void __launch_bounds__(256) k_hook_rows(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tgt,
                                                   const uint32_t *__restrict__ C, uint32_t n, uint32_t *lab,
                                                   const uint32_t *__restrict__ tree, HookLists h) {
    const uint32_t FULL = 0xFFFFFFFFu, lane = threadIdx.x & 31;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    for (uint64_t v0 = (uint64_t)warp * 32; v0 < n; v0 += (uint64_t)nwarps * 32) {
        const uint32_t v = (uint32_t)v0 + lane;
        uint64_t b = 0, e = 0;
        uint32_t c = 0;
        bool open = false;
        if (v < n) {
            c = C[v];
            open = !h.rows || ldcg_(lab + v) != tree[c];
            if (open) {
                b = off[v] + HOOK_SAMPLE;  // the sampled entries are linked already
                e = off[v + 1];
                open = b < e;
                if (open && h.rows && e - b > HOOK_MID) {
                    if (e - b > HOOK_HUB) h.rows[h.cap - 1 - atomicAdd(h.nhub, 1u)] = v;
                    else h.rows[atomicAdd(h.nmid, 1u)] = v;
                    open = false;
                }
            }
        }
        for (unsigned todo = __ballot_sync(FULL, open); todo; todo &= todo - 1) {
            const int src = __ffs((int)todo) - 1;
            const uint32_t i = (uint32_t)v0 + src, ci = __shfl_sync(FULL, c, src);
            const uint64_t bi = __shfl_sync(FULL, b, src), ei = __shfl_sync(FULL, e, src);
            hook_row(tgt, C, lab, i, ci, bi + lane, ei, 32);
            __syncwarp();
        }
    }
}

// The listed rows: block columns (x) take the longest rows in turn, their
// HOOK_COL blocks interleaved slices of each; then every block takes one of
// the others at a time.
__global__ void __launch_bounds__(256) k_hook_long(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tgt,
                                                   const uint32_t *__restrict__ C, uint32_t *lab, HookLists h) {
    const uint32_t nhub = *h.nhub, nmid = *h.nmid;
    for (uint32_t t = blockIdx.x; t < nhub; t += gridDim.x) {
        const uint32_t i = h.rows[h.cap - 1 - t];
        hook_row(tgt, C, lab, i, C[i], off[i] + HOOK_SAMPLE + blockIdx.y * blockDim.x + threadIdx.x, off[i + 1],
                 HOOK_COL * blockDim.x);
    }
    for (uint32_t t = blockIdx.y * gridDim.x + blockIdx.x; t < nmid; t += gridDim.x * HOOK_COL) {
        const uint32_t i = h.rows[t];
        hook_row(tgt, C, lab, i, C[i], off[i] + HOOK_SAMPLE + threadIdx.x, off[i + 1], blockDim.x);
    }
}

static void split_hook(const DevGraph &g, const uint32_t *C, uint32_t *lab, cudaStream_t s) {
    size_t mk = arena().mark();
    // trees, lists of long rows and their counts; without room for them in a
    // caller's workspace every row is linked by its warp
    HookLists h{};
    h.cap = (uint32_t)std::min<uint64_t>(g.n, g.nnz / HOOK_MID) + 1;
    uint32_t *tree = static_cast<uint32_t *>(arena().try_alloc(sizeof(uint32_t) * ((size_t)g.n + h.cap + 2)));
    if (tree) {
        h.rows = tree + g.n;
        h.nmid = h.rows + h.cap;
        h.nhub = h.nmid + 1;
        GSP_CUDA(cudaMemsetAsync(h.nmid, 0, 2 * sizeof(uint32_t), s));
    }
    iota_u32(lab, g.n, s);
    const unsigned gr = grid_for(g.n, 256);
    k_hook_sample<<<gr, 256, 0, s>>>(g.off, g.tgt, C, g.n, lab);
    GSP_CHECK_LAUNCH();
    if (tree) {
        k_hook_compress<<<gr, 256, 0, s>>>(C, g.n, lab, tree);
        GSP_CHECK_LAUNCH();
    }
    k_hook_rows<<<gr, 256, 0, s>>>(g.off, g.tgt, C, g.n, lab, tree, h);
    GSP_CHECK_LAUNCH();
    if (tree && h.cap > 1) {
        k_hook_long<<<dim3(sm_count(), HOOK_COL), 256, 0, s>>>(g.off, g.tgt, C, lab, h);
        GSP_CHECK_LAUNCH();
    }
    k_hook_compress<<<gr, 256, 0, s>>>(C, g.n, lab, nullptr);
    GSP_CHECK_LAUNCH();
    arena().release(mk);
}

// --------------------------------------------------------------------- BFS
// Seeds of a round: the smallest unvisited vertex of every community that
// still has one.  `cand` lists the vertices unvisited after the previous
// round (all vertices in the first round).
__global__ void k_bfs_seed_min(const uint32_t *__restrict__ C, const uint32_t *__restrict__ lab,
                               const uint32_t *__restrict__ cand, const uint32_t *__restrict__ ncand, uint32_t n,
                               uint32_t *seed) {
    uint32_t cnt = cand ? *ncand : n;
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += gridDim.x * blockDim.x) {
        uint32_t v = cand ? cand[t] : t;
        if (lab[v] == EMPTY) atomicMin(seed + C[v], v);
    }
}

// Warp-aggregated append of the lanes with `want` set.
__device__ __forceinline__ void push_warp(bool want, uint32_t v, uint32_t *q, uint32_t *qn) {
    uint32_t ballot = __ballot_sync(0xFFFFFFFFu, want);
    if (!ballot) return;
    int lane = threadIdx.x & 31;
    int leader = __ffs(ballot) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(qn, (uint32_t)__popc(ballot));
    base = __shfl_sync(0xFFFFFFFFu, base, leader);
    if (want) q[base + __popc(ballot & ((1u << lane) - 1u))] = v;
}

// Label the seeds and start the frontier; the other unvisited vertices form
// the candidate list of the next round.
__global__ void k_bfs_seed_push(const uint32_t *__restrict__ C, uint32_t *lab, const uint32_t *__restrict__ cand,
                                const uint32_t *__restrict__ ncand, uint32_t n, const uint32_t *__restrict__ seed,
                                uint32_t *q, uint32_t *qn, uint32_t *rest, uint32_t *nrest) {
    uint32_t cnt = cand ? *ncand : n;
    for (uint32_t t0 = blockIdx.x * blockDim.x; t0 < cnt; t0 += gridDim.x * blockDim.x) {
        uint32_t t = t0 + threadIdx.x;
        bool is_seed = false, keep = false;
        uint32_t v = 0;
        if (t < cnt) {
            v = cand ? cand[t] : t;
            if (lab[v] == EMPTY) {
                if (seed[C[v]] == v) {
                    lab[v] = v;
                    is_seed = true;
                } else {
                    keep = true;
                }
            }
        }
        push_warp(is_seed, v, q, qn);
        push_warp(keep, v, rest, nrest);
    }
}

__global__ void k_bfs_seed_reset(const uint32_t *__restrict__ C, const uint32_t *__restrict__ q,
                                 const uint32_t *__restrict__ qn, uint32_t *seed) {
    uint32_t cnt = *qn;
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += gridDim.x * blockDim.x)
        seed[C[q[t]]] = EMPTY;
}

constexpr uint32_t BFS_BIG = 1024;

__device__ __forceinline__ void bfs_visit_edges(const uint32_t *__restrict__ tgt, const uint32_t *__restrict__ C,
                                                uint32_t *lab, uint64_t p0, uint64_t e, uint64_t step, uint32_t cu,
                                                uint32_t lu, uint32_t *nq, uint32_t *nqn) {
    // all 32 lanes of the warp run the same trip count (push_warp ballots)
    for (uint64_t pb = p0; pb < e + (threadIdx.x & 31) && pb - (threadIdx.x & 31) < e; pb += step) {
        uint64_t p = pb;
        bool want = false;
        uint32_t j = 0;
        if (p < e) {
            j = tgt[p];
            if (C[j] == cu && ldcg_(lab + j) == EMPTY) want = atomicCAS(lab + j, EMPTY, lu) == EMPTY;
        }
        push_warp(want, j, nq, nqn);
    }
}

// One level: a warp per frontier vertex claims unvisited same-community
// neighbours with atomicCAS and appends them to the next frontier; frontier
// vertices of degree > BFS_BIG go to a list for k_bfs_expand_big.
__global__ void k_bfs_expand(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tgt,
                             const uint32_t *__restrict__ C, uint32_t *lab, const uint32_t *__restrict__ q,
                             const uint32_t *__restrict__ qn, uint32_t *nq, uint32_t *nqn, uint32_t *big,
                             uint32_t *nbig) {
    uint32_t cnt = *qn;
    int lane = threadIdx.x & 31;
    uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t t = warp; t < cnt; t += nwarps) {
        uint32_t u = q[t];
        uint64_t b = off[u], e = off[u + 1];
        if (e - b > BFS_BIG) {
            if (lane == 0) big[atomicAdd(nbig, 1u)] = u;
            continue;
        }
        uint32_t cu = C[u], lu = ldcg_(lab + u);
        bfs_visit_edges(tgt, C, lab, b + lane, e, 32, cu, lu, nq, nqn);
    }
}

// The big frontier vertices: every warp of the grid strides over each one's
// edges in turn.
__global__ void k_bfs_expand_big(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tgt,
                                 const uint32_t *__restrict__ C, uint32_t *lab, const uint32_t *__restrict__ big,
                                 const uint32_t *__restrict__ nbig, uint32_t *nq, uint32_t *nqn) {
    uint32_t cnt = *nbig;
    uint64_t tid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    uint64_t T = (uint64_t)gridDim.x * blockDim.x;
    for (uint32_t t = 0; t < cnt; t++) {
        uint32_t u = big[t];
        uint32_t cu = C[u], lu = ldcg_(lab + u);
        bfs_visit_edges(tgt, C, lab, off[u] + tid, off[u + 1], T, cu, lu, nq, nqn);
    }
}

// Rounds of multi-source BFS.  Levels are launched in batches of
// BFS_LEVEL_BATCH between host checks of the frontier size (an empty
// frontier makes the remaining launches of a batch return at once).
constexpr int BFS_LEVEL_BATCH = 6;

static void split_bfs(const DevGraph &g, const uint32_t *C, uint32_t *lab, cudaStream_t s) {
    size_t mk = arena().mark();
    uint32_t n = g.n;
    uint32_t *seed = arena().get<uint32_t>(n);
    uint32_t *fr[BFS_LEVEL_BATCH + 1];
    for (int k = 0; k <= BFS_LEVEL_BATCH; k++) fr[k] = nullptr;
    uint32_t *qa = arena().get<uint32_t>(n);
    uint32_t *qb = arena().get<uint32_t>(n);
    uint32_t *candA = arena().get<uint32_t>(n);
    uint32_t *candB = arena().get<uint32_t>(n);
    uint32_t *big = arena().get<uint32_t>(n);
    // counters: [0] seeds, [1] rest, [2 .. 2+BATCH] frontier sizes, big counts after
    uint32_t *cnts = arena().get<uint32_t>(4 + 2 * (BFS_LEVEL_BATCH + 1));
    uint32_t *ncandA = cnts + 0;  // candidate counts live beside the seed/rest counters
    GSP_CUDA(cudaMemsetAsync(lab, 0xFF, sizeof(uint32_t) * n, s));
    GSP_CUDA(cudaMemsetAsync(seed, 0xFF, sizeof(uint32_t) * n, s));
    const uint32_t *cand = nullptr;  // first round: every vertex
    uint32_t *cand_cnt = nullptr;
    uint32_t h_cand = n;
    uint32_t *cbuf[2] = {candA, candB};
    uint32_t *ccnt[2] = {cnts + 2 + 2 * (BFS_LEVEL_BATCH + 1), cnts + 3 + 2 * (BFS_LEVEL_BATCH + 1)};
    (void)ncandA;
    int cb = 0;
    for (int round = 0; h_cand > 0; round++) {
        uint32_t *rest = cbuf[cb], *nrest = ccnt[cb];
        uint32_t *qn = cnts + 0;
        GSP_CUDA(cudaMemsetAsync(cnts, 0, sizeof(uint32_t) * (2 + 2 * (BFS_LEVEL_BATCH + 1)), s));
        GSP_CUDA(cudaMemsetAsync(nrest, 0, sizeof(uint32_t), s));
        unsigned gr = grid_for(h_cand, 256);
        k_bfs_seed_min<<<gr, 256, 0, s>>>(C, lab, cand, cand_cnt, n, seed);
        GSP_CHECK_LAUNCH();
        k_bfs_seed_push<<<gr, 256, 0, s>>>(C, lab, cand, cand_cnt, n, seed, qa, qn, rest, nrest);
        GSP_CHECK_LAUNCH();
        k_bfs_seed_reset<<<gr, 256, 0, s>>>(C, qa, qn, seed);
        GSP_CHECK_LAUNCH();
        // levels, in batches
        uint32_t *q = qa, *nq = qb;
        uint32_t *fcnt = cnts + 2;        // fcnt[k]: frontier size of level k in the batch
        uint32_t *bcnt = cnts + 2 + (BFS_LEVEL_BATCH + 1);
        GSP_CUDA(cudaMemcpyAsync(fcnt, qn, sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
        for (;;) {
            for (int k = 0; k < BFS_LEVEL_BATCH; k++) {
                k_bfs_expand<<<sms(8), 256, 0, s>>>(g.off, g.tgt, C, lab, q, fcnt + k, nq, fcnt + k + 1, big,
                                                    bcnt + k);
                GSP_CHECK_LAUNCH();
                k_bfs_expand_big<<<sms(4), 256, 0, s>>>(g.off, g.tgt, C, lab, big, bcnt + k, nq,
                                                                 fcnt + k + 1);
                GSP_CHECK_LAUNCH();
                uint32_t *t = q; q = nq; nq = t;
            }
            uint32_t last;
            GSP_CUDA(cudaMemcpyAsync(&last, fcnt + BFS_LEVEL_BATCH, sizeof(last), cudaMemcpyDeviceToHost, s));
            GSP_CUDA(cudaStreamSynchronize(s));
            if (last == 0) break;
            GSP_CUDA(cudaMemcpyAsync(fcnt, fcnt + BFS_LEVEL_BATCH, sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
            GSP_CUDA(cudaMemsetAsync(fcnt + 1, 0, sizeof(uint32_t) * BFS_LEVEL_BATCH, s));
            GSP_CUDA(cudaMemsetAsync(bcnt, 0, sizeof(uint32_t) * (BFS_LEVEL_BATCH + 1), s));
        }
        // vertices still unvisited become the next round's candidates
        GSP_CUDA(cudaMemcpyAsync(&h_cand, nrest, sizeof(h_cand), cudaMemcpyDeviceToHost, s));
        GSP_CUDA(cudaStreamSynchronize(s));
        cand = rest;
        cand_cnt = nrest;
        cb ^= 1;
    }
    arena().release(mk);
}

void split_labels(const DevGraph &g, const Classes &cl, const uint32_t *C, int mode, uint32_t *labels,
                  cudaStream_t s) {
    if (mode == GSP_SPLIT_BFS) split_bfs(g, C, labels, s);
    else if (mode == GSP_SPLIT_LP) split_lp(g, cl, C, labels, s);
    else split_hook(g, C, labels, s);
}

}  // namespace gsp
