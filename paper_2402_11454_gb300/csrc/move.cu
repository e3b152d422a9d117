// move.cu -- local-moving phase of GSP-Louvain (Algorithm 4, louvainMove and
// scanCommunities) on sm_103a.
//
// Each active vertex i gathers K_{i->c} for every neighbouring community c
// (self-loop excluded) into an open-addressing hashtable, scores every
// candidate with Equation 2 and takes the argmax (ties to the lowest id);
// it moves only on a strictly positive gain.  The work is binned by degree:
//   groups of G = 4/8/16/32 lanes per vertex, table in shared memory (one
//     fused launch for the four group classes);
//   one warp per vertex, 1024-slot shared table (degree <= 512);
//   one block per vertex, table in shared memory (degree <= 2048, <= 8192);
//   the whole grid per vertex for larger degrees ("hubs"): edge-chunk tasks
//     combined in shared memory, published to a global-memory table.
// Duplicate community keys meet in the table through atomicCAS on the key and
// atomicAdd on the value.
//
// Parallel semantics.  Frozen-state mode (deterministic): the vertices of a
// sweep are split into W interleaved waves (vertex i in wave i mod W); a wave
// reads C, Sigma and the community sizes left by the earlier waves, appends
// its moves to a list, and apply_moves() applies them (Sigma/size atomics,
// neighbour re-marking) before the next wave.  In-place mode: the paper's
// parallel loop as written, every move applied at once, with L2-coherent
// loads (ld.global.cg) for values other threads update.
//
// Precision: FP64 evaluates Equation 2 term by term with round-to-nearest
// intrinsics (no fused multiply-add), in the order written.  MIXED accumulates
// K_{i->c} in float32 and compares the scaled score s_c = K_{i->c} - K_i *
// Sigma_c / 2m in float32 (m * dQ_{i:d->c} = s_c - s_d with Sigma_d taken
// without K_i); m and Sigma stay float64.
#include <algorithm>
#include <type_traits>

#include "internal.cuh"

namespace gsp {

struct MoveArgs {
    const uint64_t *off;
    const uint32_t *tgt;
    const void *w;
    uint32_t *C;
    const double *K;
    double *Sig;
    uint32_t *size;
    uint8_t *act;
    uint8_t *mark;  // re-marking target: a separate array merged after a frozen-state wave, act in place
    const double *m;  // m and 1/m
    // batches of independent graphs: graph of each vertex, m of each graph,
    // per-graph summed gains (null for a single graph)
    const uint32_t *gid;
    const double *m_g;
    const double *minv_g;  // 1/m of each graph
    double *dq_g;
    int lsb;  // K in exact integer units of 2^lsb (INT_MIN: float64 deltas)
    MoveCounters *ctr;
    int rule;
    // no-return rule: from iteration no_return_from on (0: never) a vertex
    // does not move back to the community it left in the previous iteration
    uint32_t *left;   // community each vertex last left
    int *left_it;     // iteration of that move (-2: none in this pass)
    const int *iteration;  // device scalar: the sweep's iteration (set before each launch or graph replay)
    int no_return_from;
    uint32_t *mv_vtx, *mv_cmt, *mv_cnt;  // frozen-state move list
    uint32_t *choice;                    // optional per-vertex decision
    // last-visit features for the learned predictor (optional)
    float *feat_kept, *feat_gain, *last_gain;
    uint8_t *moved_last;
    uint8_t *deferred;  // learned pruning: vertices the predictor put off (cleared when visited)
    // trace rows (optional): features before the visit, label = moved
    float *trace_x;
    uint8_t *trace_y;
    uint32_t *trace_cnt;
    uint64_t *trace_keys;  // optional: trace_tag | iteration << 48 | vertex per row
    uint64_t trace_tag;    // pass << 56 | repeat << 40
    uint32_t trace_cap, trace_every;
    float max_logk;
    int max_iterations;  // the iteration's position in the pass (a feature) is *iteration / max_iterations
    uint32_t salt;       // trace sampling: per pass; the iteration is mixed in on the device
};

template <typename T> __device__ __forceinline__ T ldcg(const T *p) { return __ldcg(p); }
__device__ __forceinline__ uint8_t ldcg(const uint8_t *p) {
    return (uint8_t)__ldcg(reinterpret_cast<const unsigned char *>(p));
}
// SYNC: 0 = in-place updates (the paper's loop), 1 = frozen-state wave in its
// own launch, 2 = frozen-state wave inside the persistent sweep kernel.  A
// frozen-state wave reads data that no thread writes during the wave; in its
// own launch that data is read-only for the whole launch (read-only cache
// path), inside the persistent kernel earlier phases of the same launch wrote
// it, so the loads go to L2 (the per-SM L1 is not coherent).
template <int SYNC, typename T> __device__ __forceinline__ T ld_state(const T *p) {
    if constexpr (SYNC == 1) return __ldg(p);
    else return ldcg(p);
}

// Open-addressing table of a vertex's K_{i->c} in shared memory, linear probing,
// 2^logcap slots, at least twice the vertex's degree.  It is empty between
// vertices: add() tells the thread that claimed a slot which one, that thread
// alone scores it once every edge is in, and empties it.  So nobody reads or
// clears the two to four slots per edge that stay free, and there is no shared
// list of occupied slots.  Float32 values share a 64-bit word with their key: a
// community seen for the first time (in a pass's first sweep nearly every one)
// is claimed and given its weight by one compare-and-swap, and key and value
// are read and cleared in one access.  Float64 values lie beside the keys.
template <typename V> struct Table;
template <> struct Table<float> {
    unsigned long long *t;
    static constexpr size_t slot_bytes = 8;
    static constexpr unsigned long long FREE = ~0ull;
    // slots [first, ...) of a region of `total` slots at base
    __device__ Table(unsigned char *base, uint32_t, uint32_t first)
        : t(reinterpret_cast<unsigned long long *>(base) + first) {}
    __device__ explicit Table(unsigned long long *global) : t(global) {}
    // Add N distinct communities (EMPTY: none) to a table of mask + 1 slots in
    // global memory, all first probes in flight together.
    template <int N> __device__ void publish(uint32_t mask, const uint32_t (&c)[N], const float (&v)[N]) {
        unsigned long long old[N];
#pragma unroll
        for (int u = 0; u < N; u++)
            if (c[u] != EMPTY)
                old[u] = atomicCAS(t + hub_home(hash32(c[u]), mask), FREE,
                                   ((unsigned long long)c[u] << 32) | __float_as_uint(v[u]));
#pragma unroll
        for (int u = 0; u < N; u++) {
            if (c[u] == EMPTY || old[u] == FREE) continue;
            uint32_t h = hub_home(hash32(c[u]), mask);
            for (uint64_t probe = 0; probe <= mask; probe++) {
                if ((uint32_t)(old[u] >> 32) == c[u]) {
                    atomicAdd(reinterpret_cast<float *>(t + h), v[u]);
                    break;
                }
                h = (h + 1) & mask;
                old[u] = atomicCAS(t + h, FREE, ((unsigned long long)c[u] << 32) | __float_as_uint(v[u]));
                if (old[u] == FREE) break;
            }
        }
    }
    __device__ void clear(uint32_t s) { t[s] = FREE; }
    __device__ uint32_t get(uint32_t s, float &v) const {
        const unsigned long long e = t[s];
        v = __uint_as_float((uint32_t)e);
        return (uint32_t)(e >> 32);
    }
    __device__ uint32_t add(int logcap, uint32_t c, float w) {  // the slot claimed, or EMPTY
        const uint32_t mask = (1u << logcap) - 1u;
        uint32_t h = logcap ? (hash32(c) >> (32 - logcap)) : 0u;
        const unsigned long long e = ((unsigned long long)c << 32) | __float_as_uint(w);
        for (uint32_t probe = 0; probe <= mask; probe++) {
            unsigned long long old = *(volatile unsigned long long *)(t + h);
            if (old == FREE) old = atomicCAS(t + h, FREE, e);
            if (old == FREE) return h;
            if ((uint32_t)(old >> 32) == c) {
                atomicAdd(reinterpret_cast<float *>(t + h), w);
                return EMPTY;
            }
            h = (h + 1) & mask;
        }
        return EMPTY;
    }
};
template <> struct Table<double> {
    uint32_t *keys;
    double *vals;
    static constexpr size_t slot_bytes = 12;
    __device__ Table(unsigned char *base, uint32_t total, uint32_t first)
        : keys(reinterpret_cast<uint32_t *>(base) + first),
          vals(reinterpret_cast<double *>(base + (size_t)total * sizeof(uint32_t)) + first) {}
    __device__ Table(uint32_t *gkeys, double *gvals) : keys(gkeys), vals(gvals) {}
    template <int N> __device__ void publish(uint32_t mask, const uint32_t (&c)[N], const double (&v)[N]) {
#pragma unroll
        for (int u = 0; u < N; u++) {
            if (c[u] == EMPTY) continue;
            uint32_t h = hub_home(hash32(c[u]), mask);
            for (uint64_t probe = 0; probe <= mask; probe++) {
                const uint32_t old = atomicCAS(keys + h, EMPTY, c[u]);
                if (old == EMPTY || old == c[u]) {
                    atomicAdd(vals + h, v[u]);
                    break;
                }
                h = (h + 1) & mask;
            }
        }
    }
    __device__ void clear(uint32_t s) {
        keys[s] = EMPTY;
        vals[s] = 0.0;
    }
    __device__ uint32_t get(uint32_t s, double &v) const {
        v = vals[s];
        return keys[s];
    }
    __device__ uint32_t add(int logcap, uint32_t c, double w) {
        uint32_t slot;
        return ht_add_slot<double>(keys, vals, logcap, c, w, &slot) == 1 ? slot : EMPTY;
    }
};

template <typename S> __device__ __forceinline__ bool better(S s1, uint32_t c1, S s2, uint32_t c2) {
    return s1 > s2 || (s1 == s2 && c1 < c2);
}

// Score the slots listed in slot[] (EMPTY: none) and empty them, four gathers
// of Sigma_c in flight.
template <int N, int SYNC, typename SC, typename S, typename V>
__device__ __forceinline__ void score_slots(Table<V> &tab, const uint32_t *slot, const double *Sig, const SC &sc,
                                            S &best, uint32_t &bestc, uint32_t &ncand) {
    constexpr int U = N < 4 ? N : 4;
#pragma unroll
    for (int s0 = 0; s0 < N; s0 += U) {
        uint32_t c[U];
        V v[U];
        double sg[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            c[u] = EMPTY;
            if (slot[s0 + u] != EMPTY) {
                c[u] = tab.get(slot[s0 + u], v[u]);
                tab.clear(slot[s0 + u]);
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++) sg[u] = c[u] != EMPTY ? ld_state<SYNC>(Sig + c[u]) : 0.0;
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (c[u] == EMPTY) continue;
            ncand++;
            S val = sc.score(v[u], sg[u]);
            if (better(val, c[u], best, bestc)) { best = val; bestc = c[u]; }
        }
    }
}

// Float64 scores of a warp's candidates, packed: what bounds them is the issue
// of two float64 divisions per candidate and warp, whether one lane scores or
// all do, and after the first sweeps a row of many edges has few communities, a
// lane's slots mostly none.  So the lanes hand their candidates to a queue of one
// per lane, and a full queue is scored at once.  R-MAT of 60 K vertices, a wave
// run, scored where they were claimed -> packed: degrees 2049-8192 154 -> 85 us,
// 513-2048 40 -> 35, hubs 36 -> 22; the phase 11.1 -> 7.1 ms.
template <typename V> struct ScoreQueue {
    uint32_t c = EMPTY;
    V v = V(0);
    int n = 0;  // lanes 0..n-1 hold a candidate

    template <int SYNC, typename SC, typename S>
    __device__ void score(bool on, uint32_t x, V k, const double *Sig, const SC &sc, S &best, uint32_t &bestc) {
        if (!on) return;
        const S val = sc.score(k, ld_state<SYNC>(Sig + x));
        if (better(val, x, best, bestc)) { best = val; bestc = x; }
    }
    // Take the candidates x[] with values k[] (EMPTY: none) of all 32 lanes.
    template <int SYNC, int U, typename SC, typename S>
    __device__ void put(const uint32_t (&x)[U], const V (&k)[U], const double *Sig, const SC &sc, S &best,
                        uint32_t &bestc) {
        constexpr unsigned FULL = 0xFFFFFFFFu;
        const int lane = threadIdx.x & 31;
        unsigned bal[U];
        int total = 0;
#pragma unroll
        for (int u = 0; u < U; u++) {
            bal[u] = __ballot_sync(FULL, x[u] != EMPTY);
            total += __popc(bal[u]);
        }
        if (total > 32 * (U - 1)) {  // packing would save no round: their gathers in flight together
            double sg[U];
#pragma unroll
            for (int u = 0; u < U; u++) sg[u] = x[u] != EMPTY ? ld_state<SYNC>(Sig + x[u]) : 0.0;
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (x[u] == EMPTY) continue;
                const S val = sc.score(k[u], sg[u]);
                if (better(val, x[u], best, bestc)) { best = val; bestc = x[u]; }
            }
            return;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (!bal[u]) continue;
            // the q-th candidate goes to lane n + q, round the end to the next queue
            const int m = __popc(bal[u]), q = (lane - n) & 31;
            const int src = q < m ? select_bit(bal[u], q) : 0;
            const uint32_t xs = __shfl_sync(FULL, x[u], src);
            const V ks = __shfl_sync(FULL, k[u], src);
            const bool next = lane < n;
            if (q < m && !next) { c = xs; v = ks; }
            if (n + m >= 32) {
                score<SYNC>(true, c, v, Sig, sc, best, bestc);
                if (q < m && next) { c = xs; v = ks; }
                n -= 32;
            }
            n += m;
        }
    }
    template <int SYNC, typename SC, typename S>
    __device__ void finish(const double *Sig, const SC &sc, S &best, uint32_t &bestc) {
        score<SYNC>((int)(threadIdx.x & 31) < n, c, v, Sig, sc, best, bestc);
        n = 0;
    }
};

// As score_slots, by all lanes of a warp together.
template <int N, int SYNC, typename SC, typename S, typename V>
__device__ __forceinline__ void score_slots_warp(Table<V> &tab, const uint32_t *slot, const double *Sig, const SC &sc,
                                                 S &best, uint32_t &bestc, uint32_t &ncand) {
    if constexpr (std::is_same<V, float>::value) {
        score_slots<N, SYNC>(tab, slot, Sig, sc, best, bestc, ncand);
    } else {
        ScoreQueue<V> queue;
        constexpr int U = N < 4 ? N : 4;
#pragma unroll
        for (int s0 = 0; s0 < N; s0 += U) {
            uint32_t c[U];
            V v[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                c[u] = EMPTY;
                v[u] = V(0);
                if (slot[s0 + u] == EMPTY) continue;
                c[u] = tab.get(slot[s0 + u], v[u]);
                tab.clear(slot[s0 + u]);
                ncand++;
            }
            queue.template put<SYNC>(c, v, Sig, sc, best, bestc);
        }
        queue.template finish<SYNC>(Sig, sc, best, bestc);
    }
}

// The same over a whole table of cap slots, this thread's lane, lane + step, ...
// (step: a multiple of the warp).
template <int SYNC, typename SC, typename S, typename V>
__device__ __forceinline__ void score_table(Table<V> &tab, uint32_t cap, uint32_t lane, uint32_t step,
                                            const double *Sig, const SC &sc, S &best, uint32_t &bestc,
                                            uint32_t &ncand) {
    ScoreQueue<V> queue;
    for (uint32_t s0 = 0; s0 < cap; s0 += 4 * step) {
        uint32_t slot[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const uint32_t s = s0 + u * step + lane;
            V v;
            slot[u] = s < cap && tab.get(s, v) != EMPTY ? s : EMPTY;
        }
        if constexpr (std::is_same<V, float>::value) {
            score_slots<4, SYNC>(tab, slot, Sig, sc, best, bestc, ncand);
        } else {
            uint32_t c[4];
            V v[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                c[u] = EMPTY;
                v[u] = V(0);
                if (slot[u] == EMPTY) continue;
                c[u] = tab.get(slot[u], v[u]);
                tab.clear(slot[u]);
                ncand++;
            }
            queue.template put<SYNC>(c, v, Sig, sc, best, bestc);
        }
    }
    if constexpr (!std::is_same<V, float>::value) queue.template finish<SYNC>(Sig, sc, best, bestc);
}

// Equation 2, evaluated in the order written, with no contraction.
__device__ __forceinline__ double eq2(double Kic, double Kid, double Ki, double Sc, double Sd, double m) {
    double t1 = __ddiv_rn(__dsub_rn(Kic, Kid), m);
    double t2 = __dmul_rn(Ki, __dsub_rn(__dadd_rn(Ki, Sc), Sd));
    double den = __dmul_rn(__dmul_rn(2.0, m), m);
    return __dsub_rn(t1, __ddiv_rn(t2, den));
}

// (float)x, rounded to nearest even, in integer operations.  Float64
// instructions, conversions included, issue at a fraction of the integer rate
// on this GPU, and the conversion of Sigma_c is the one a score needs.
// Values outside float32's normal range take the instruction.
__device__ __forceinline__ float f32_of(double x) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const uint32_t hi = (uint32_t)(u >> 32), mag = hi & 0x7FFFFFFFu;
    if (mag - 0x38100000u >= 0x0FE00000u) return (mag | (uint32_t)u) ? (float)x : __uint_as_float(hi);
    // 29 bits of the mantissa go; add half an ulp, less one bit when the kept part is even
    const unsigned long long r = (u & 0x7FFFFFFFFFFFFFFFull) + 0x0FFFFFFFull + ((u >> 29) & 1ull);
    return __uint_as_float(((uint32_t)(r >> 29) - (896u << 23)) | (hi & 0x80000000u));
}

// Per-vertex scoring context.
template <bool F64> struct Score;
template <> struct Score<true> {
    using S = double;
    double Ki, Kid, Sd, m;
    __device__ S score(double kic, double Sc) const { return eq2(kic, Kid, Ki, Sc, Sd, m); }
    __device__ bool gains(S best) const { return best > 0.0; }
    __device__ double gain(S best) const { return best; }  // in units of Q
};
// Float64 is a narrow pipe on this GPU: the mixed-precision scores take 1/m
// precomputed (0.5/m is 0.5 * RN(1/m) exactly, so K_i/2m is unchanged) and
// the gain of the chosen community is a product, not a division.
template <> struct Score<false> {
    using S = float;
    float kif, sd;
    double inv_m;
    __device__ S score(float kic, double Sc) const { return __fmaf_rn(-kif, f32_of(Sc), kic); }
    __device__ bool gains(S best) const { return best - sd > 0.0f; }  // gain(best) > 0
    __device__ double gain(S best) const { return (double)(best - sd) * inv_m; }
};

// m and inv_m = 1/m of the vertex's graph (the float64 score uses m only).
// The float32 operations are spelled out, so that every kernel that may serve
// a vertex decides exact ties of s_c and s_d alike: the candidates' scores
// round once (fused); the score of staying rounds twice, but once for a vertex
// of more than BIG_MAX_LIMIT edges (hub).  That is a property of the vertex: the
// boundaries between the classes may be tuned, and must not change a decision.
template <bool F64>
__device__ __forceinline__ Score<F64> make_score(double Ki, typename std::conditional<F64, double, float>::type kid,
                                                 double Sd, double m, double inv_m, bool hub = false);
template <>
__device__ __forceinline__ Score<true> make_score<true>(double Ki, double kid, double Sd, double m, double, bool) {
    Score<true> s;
    s.Ki = Ki; s.Kid = kid; s.Sd = Sd; s.m = m;
    return s;
}
template <>
__device__ __forceinline__ Score<false> make_score<false>(double Ki, float kid, double Sd, double, double inv_m,
                                                          bool hub) {
    Score<false> s;
    const double inv2m = 0.5 * inv_m;
    s.kif = f32_of(Ki * inv2m);
    const float rest = f32_of(Sd - Ki);
    s.sd = hub ? __fmaf_rn(-s.kif, rest, kid) : __fsub_rn(kid, __fmul_rn(s.kif, rest));
    s.inv_m = inv_m;
    return s;
}

__device__ __forceinline__ bool rounds_as_hub(uint64_t deg) { return deg > BIG_MAX_LIMIT; }

// m of vertex i's graph (batches) or of the single graph.
__device__ __forceinline__ double vertex_m(const MoveArgs &a, uint32_t i, double m0) {
    return a.gid ? a.m_g[a.gid[i]] : m0;
}
__device__ __forceinline__ double vertex_inv_m(const MoveArgs &a, uint32_t i, double inv0) {
    return a.gid ? a.minv_g[a.gid[i]] : inv0;
}
__device__ __forceinline__ void add_graph_gain(const MoveArgs &a, uint32_t i, double gain) {
    if (a.dq_g) atomicAdd(a.dq_g + a.gid[i], gain);
}

// In place: i moves from d to c now.
__device__ __forceinline__ void apply_now(const MoveArgs &a, uint32_t i, uint32_t d, uint32_t c, double Ki) {
    a.left[i] = d;
    a.left_it[i] = *a.iteration;
    a.C[i] = c;
    atomicAdd(a.Sig + d, -Ki);
    atomicAdd(a.Sig + c, Ki);
    atomicSub(a.size + d, 1u);
    atomicAdd(a.size + c, 1u);
}

// Decide the move of i toward c (one thread).  Frozen-state: record it in the
// move list; in place: apply it now.  Returns whether i moves.
template <int SYNC>
__device__ __forceinline__ bool decide_move(const MoveArgs &a, uint32_t i, uint32_t d, uint32_t c, double Ki) {
    if (c == EMPTY || c == d) return false;
    if (a.rule) {
        uint32_t sd = ld_state<SYNC>(a.size + d), sc = ld_state<SYNC>(a.size + c);
        if (sd == 1 && sc == 1 && c > d) return false;
    }
    if (a.no_return_from > 0 && ld_state<SYNC>(a.left + i) == c) {
        const int it = *a.iteration;
        if (it >= a.no_return_from && ld_state<SYNC>(a.left_it + i) == it - 1) return false;
    }
    if (a.choice) a.choice[i] = c;
    if constexpr (SYNC) {
        uint32_t slot = atomicAdd(a.mv_cnt, 1u);
        a.mv_vtx[slot] = i;
        a.mv_cmt[slot] = c;
    } else {
        apply_now(a, i, d, c, Ki);
    }
    return true;
}

struct LocalCtr {  // of one thread (a thread visits fewer than 2^32 edges in a launch's sums)
    double dq = 0;
    uint32_t moved = 0, vertices = 0, candidates = 0;
    unsigned long long edges = 0, marked = 0;
};

// Warp sums by the reduction instruction, a float64 sum only where something
// moved, and one shared atomic per warp and counter (six block-wide sums of
// shuffles took twelve barriers).
__device__ void flush_counters(const LocalCtr &l, MoveCounters *g) {
    constexpr unsigned FULL = 0xFFFFFFFFu;
    __shared__ unsigned long long s_cnt[5];
    __shared__ double s_dq;
    if (threadIdx.x < 5) s_cnt[threadIdx.x] = 0;
    if (threadIdx.x == 5) s_dq = 0.0;
    __syncthreads();
    const bool lane0 = (threadIdx.x & 31) == 0;
    const uint32_t n3[3] = {l.moved, l.vertices, l.candidates};
    const unsigned long long e2[2] = {l.edges, l.marked};
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const uint32_t t = __reduce_add_sync(FULL, n3[k]);
        if (lane0 && t) atomicAdd(&s_cnt[k], (unsigned long long)t);
    }
#pragma unroll
    for (int k = 0; k < 2; k++) {
        // 64-bit sums in two halves: the low 26 bits of 32 lanes stay below 2^32
        const uint32_t lo = __reduce_add_sync(FULL, (uint32_t)(e2[k] & 0x3FFFFFFu));
        const uint32_t hi = __reduce_add_sync(FULL, (uint32_t)(e2[k] >> 26));
        if (lane0 && (lo | hi)) atomicAdd(&s_cnt[3 + k], ((unsigned long long)hi << 26) + lo);
    }
    if (__any_sync(FULL, l.dq != 0.0)) {
        const double dq = warp_sum(l.dq);
        if (lane0) atomicAdd(&s_dq, dq);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_dq != 0.0) atomicAdd(&g->dq, s_dq);
        if (s_cnt[0]) atomicAdd(&g->moved, s_cnt[0]);
        if (s_cnt[1]) atomicAdd(&g->vertices, s_cnt[1]);
        if (s_cnt[2]) atomicAdd(&g->candidates, s_cnt[2]);
        if (s_cnt[3]) atomicAdd(&g->edges, s_cnt[3]);
        if (s_cnt[4]) atomicAdd(&g->marked, s_cnt[4]);
    }
}

__device__ __forceinline__ void vertex_features(const MoveArgs &a, uint32_t i, uint32_t deg, double Ki, float *x) {
    const float iter_frac = a.max_iterations > 0 ? (float)*a.iteration / (float)a.max_iterations : 0.0f;
    predictor_features(deg, Ki, a.feat_kept[i], a.feat_gain[i], a.moved_last[i], a.max_logk, iter_frac, x);
}

// After a visit: record last-visit features and, for sampled visits, a trace
// row (features before the visit, label = moved).
__device__ __forceinline__ void record_visit(const MoveArgs &a, uint32_t i, uint32_t deg, double Ki, double kid,
                                             double gain, double m, int moved) {
    if (!a.feat_kept) return;
    if (a.trace_x && (hash32(i ^ ((uint32_t)*a.iteration * 0x9E3779B9u + a.salt)) % a.trace_every) == 0) {
        float x[MLP_IN];
        vertex_features(a, i, deg, Ki, x);
        uint32_t slot = atomicAdd(a.trace_cnt, 1u);
        if (slot < a.trace_cap) {
#pragma unroll
            for (int k = 0; k < MLP_IN; k++) a.trace_x[(size_t)slot * MLP_IN + k] = x[k];
            a.trace_y[slot] = (uint8_t)moved;
            if (a.trace_keys) a.trace_keys[slot] = a.trace_tag | ((uint64_t)(*a.iteration & 0xFF) << 48) | i;
        }
    }
    float kept = Ki > 0.0 ? (float)(kid / Ki) : 0.0f;
    float g = Ki > 0.0 ? (float)(gain * m / Ki) : 0.0f;
    a.feat_kept[i] = kept;
    a.feat_gain[i] = fminf(fmaxf(g, -1.0f), 1.0f);
    if (a.last_gain) a.last_gain[i] = (float)gain;
    a.moved_last[i] = (uint8_t)moved;
}

// --------------------------------------------------------------------------
// One warp, 32 / 2^lg vertices at a time: 2^lg lanes per vertex.
//
// The warp goes through the steps of a visit together, groups without a
// vertex idling along.  What bounds a visit is its chain of gathers (flag ->
// row and C_i -> targets -> C_j -> Sigma_c) and what it issues between them:
// Sigma of the first EPL edges' communities is gathered while the table fills,
// movers of a round share one reservation in the move list, the row is read
// once (its targets stay in registers for the marks of a mover), and nothing
// on the way is a float64 instruction that an integer or float32 one can
// replace (this part issues float64 at 1/64 of the float32 rate; one division
// 1/m per thread was a third of the group kernel's time).
// A full wave of R-MAT 21 alone, before -> after: degrees <= 128 78 -> 61 us,
// 129-512 49 -> 36, 513-2048 85 -> 57.
// --------------------------------------------------------------------------
template <int EPL, typename WT> struct LaneEdges {
    uint32_t j[EPL];
    WT w[EPL];
    // edges gl, gl + G, ... of a row of deg entries at b; padding counts as a self-loop
    __device__ __forceinline__ void load(const uint32_t *__restrict__ tgt, const WT *__restrict__ wt, uint32_t i,
                                         uint64_t b, uint32_t deg, uint32_t gl, int lg) {
#pragma unroll
        for (int u = 0; u < EPL; u++) {
            const uint32_t p = gl + ((uint32_t)u << lg);
            const bool ok = p < deg;
            j[u] = ok ? __ldg(tgt + b + p) : i;
            w[u] = ok ? __ldg(wt + b + p) : WT(0);
        }
    }
};

template <typename V> struct Decision {  // of the group's vertex, the same in all its lanes
    uint32_t to = EMPTY;  // community to move to (EMPTY: stay)
    double gain = 0.0;
    V kid = 0;
};

// Decide vertex i (act: the group has one and it is unprocessed) of community
// d, whose lanes hold c[] = C of their first EPL edges' targets; rows of up to
// CH * EPL * G edges.  tab: the group's table of 2^logcap slots, empty before
// and after; all of it is used whatever the degree, since free slots cost
// nothing and make the probes shorter.
template <int EPL, int CH, int SYNC, typename WT, bool F64, typename V>
__device__ __forceinline__ Decision<V> decide_warp(const MoveArgs &a, int lg, bool act, uint32_t i, uint32_t d,
                                                   uint64_t b, uint32_t deg, double Ki, double m, double inv_m,
                                                   const LaneEdges<EPL, WT> &ed, const uint32_t (&c)[EPL], int it,
                                                   Table<V> tab, int logcap, LocalCtr &lc) {
    using SC = Score<F64>;
    using S = typename SC::S;
    constexpr unsigned FULL = 0xFFFFFFFFu;
    const uint32_t G = 1u << lg, gl = threadIdx.x & (G - 1u);
    const WT *w = static_cast<const WT *>(a.w);
    double Sd = 0.0, sg[EPL];
    uint32_t sd = 0, lf = EMPTY;
    if (act) {
        // Sigma of the first edges' communities while the table fills
#pragma unroll
        for (int u = 0; u < EPL; u++) sg[u] = c[u] != d ? ld_state<SYNC>(a.Sig + c[u]) : 0.0;
        Sd = ld_state<SYNC>(a.Sig + d);
        if (a.rule) sd = ld_state<SYNC>(a.size + d);
        if (a.no_return_from > 0 && it >= a.no_return_from && ld_state<SYNC>(a.left_it + i) == it - 1)
            lf = ld_state<SYNC>(a.left + i);
    }
    uint32_t slot[EPL * CH];
#pragma unroll
    for (int u = 0; u < EPL * CH; u++) slot[u] = EMPTY;
    V kid = 0;
    if (act) {
#pragma unroll
        for (int u = 0; u < EPL; u++) {
            if (ed.j[u] == i) continue;
            if (c[u] == d) kid += (V)ed.w[u];
            else slot[u] = tab.add(logcap, c[u], (V)ed.w[u]);
        }
    }
    if constexpr (CH > 1) {
#pragma unroll
        for (int h = 1; h < CH; h++) {
            const uint32_t p0 = h * EPL * G;
            if (!act || deg <= p0) continue;
            LaneEdges<EPL, WT> more;
            more.load(a.tgt, w, i, b + p0, deg - p0, gl, lg);
            uint32_t cm[EPL];
#pragma unroll
            for (int u = 0; u < EPL; u++) cm[u] = more.j[u] != i ? ld_state<SYNC>(a.C + more.j[u]) : d;
#pragma unroll
            for (int u = 0; u < EPL; u++) {
                if (more.j[u] == i) continue;
                if (cm[u] == d) kid += (V)more.w[u];
                else slot[h * EPL + u] = tab.add(logcap, cm[u], (V)more.w[u]);
            }
        }
    }
    __syncwarp();  // every edge is in
    for (uint32_t o = G >> 1; o > 0; o >>= 1) kid += __shfl_xor_sync(FULL, kid, o);
    const SC sc = make_score<F64>(Ki, kid, Sd, m, inv_m);
    S best = -INFINITY;
    uint32_t bestc = EMPTY, ncand = 0;
#pragma unroll
    for (int u = 0; u < EPL; u++) {
        if (slot[u] == EMPTY) continue;
        V v;
        const uint32_t cu = tab.get(slot[u], v);
        tab.clear(slot[u]);
        ncand++;
        const S x = sc.score(v, sg[u]);
        if (better(x, cu, best, bestc)) { best = x; bestc = cu; }
    }
    if constexpr (CH > 1) {
        if (act && deg > EPL * G)
            score_slots<EPL * (CH - 1), SYNC>(tab, slot + EPL, a.Sig, sc, best, bestc, ncand);
    }
    lc.candidates += ncand;
    const bool need_size = sd == 1;  // the singleton rule looks at the target's size
    uint32_t bsz = need_size && bestc != EMPTY ? ld_state<SYNC>(a.size + bestc) : 0u;
    __syncwarp();  // the table is empty
    for (uint32_t o = G >> 1; o > 0; o >>= 1) {
        const S x = __shfl_xor_sync(FULL, best, o);
        const uint32_t cx = __shfl_xor_sync(FULL, bestc, o), zx = __shfl_xor_sync(FULL, bsz, o);
        if (better(x, cx, best, bestc)) { best = x; bestc = cx; bsz = zx; }
    }
    Decision<V> r;
    r.kid = kid;
    if (act) {
        // a vertex alone in its community moves to another singleton only
        // toward a lower id, and nobody back to the community just left
        if (bestc != EMPTY && sc.gains(best) && bestc != lf && !(need_size && bsz == 1 && bestc > d)) r.to = bestc;
        if (r.to != EMPTY || (a.feat_kept && bestc != EMPTY)) r.gain = sc.gain(best);
        if (gl == 0) {
            lc.vertices++;
            lc.edges += deg;
            if (r.to != EMPTY) {
                lc.moved++;
                lc.marked += deg;
                lc.dq += r.gain;
                add_graph_gain(a, i, r.gain);
            }
        }
    }
    return r;
}

// A class of at most CAP / 2 edges per vertex, G lanes each; a warp's tables
// (32 / G of CAP slots) lie in its own region of shared memory, so the warps of
// a block run independently: warp `wbase` of `wstep` takes the list entries
// wbase, wbase + wstep, ...
template <int G, int CAP, typename V> constexpr size_t warp_tables = (size_t)(32 / G) * CAP * Table<V>::slot_bytes;

template <int G, int CAP, typename WT, bool F64, int SYNC>
__device__ void group_body(const MoveArgs &a, const uint32_t *__restrict__ list, uint32_t count, uint32_t wbase,
                           uint32_t wstep, unsigned char *warp_smem, LocalCtr &lc) {
    using V = typename std::conditional<F64, double, float>::type;
    constexpr unsigned FULL = 0xFFFFFFFFu;
    constexpr int LG = G == 4 ? 2 : G == 8 ? 3 : G == 16 ? 4 : 5;
    constexpr int NGW = 32 / G;                  // vertices of a warp at a time
    constexpr int EPL = CAP <= 4 * G ? 2 : 4;    // edges a lane holds ...
    constexpr int CH = CAP / 2 / (EPL * G);      // ... and rounds of them in the longest row
    const int wl = threadIdx.x & 31, gl = wl % G, gw = wl / G;
    Table<V> tab(warp_smem, NGW * CAP, gw * CAP);
    for (int t = gl; t < CAP; t += G) tab.clear(t);
    __syncwarp();  // votes and shuffles do not order shared memory
    const WT *w = static_cast<const WT *>(a.w);
    const double m0 = *a.m, inv0 = a.m[1];
    const int it = *a.iteration;
    // 32 of the warp's entries are claimed at once (each lane reads one flag
    // and marks its vertex processed), and the active ones are dealt to the
    // groups round by round, so that the inactive vertices of later sweeps
    // cost one parallel round of loads per 32 entries.
    for (uint64_t kb = 0; wbase + kb * wstep < count; kb += 32) {
        const uint64_t my = wbase + (kb + wl) * wstep;
        uint32_t vi = 0;
        int claim = 0;
        if (my < count) {
            vi = list[my];
            claim = ld_state<SYNC>(a.act + vi);
            if (claim) {
                a.act[vi] = 0;
                if (a.deferred) a.deferred[vi] = 0;
            }
        }
        const unsigned amask = __ballot_sync(FULL, claim);
        const int nact = __popc(amask);
        for (int r0 = 0; r0 < nact; r0 += NGW) {
            const int q = r0 + gw;  // this group's active entry in the round
            const bool act = q < nact;
            const uint32_t i = __shfl_sync(FULL, vi, act ? select_bit(amask, q) : 0);
            uint64_t b = 0;
            uint32_t deg = 0, d = 0, c[EPL];
            double Ki = 0.0, m = m0, inv_m = inv0;
            LaneEdges<EPL, WT> ed;
            if (act) {
                d = ld_state<SYNC>(a.C + i);
                b = a.off[i];
                deg = (uint32_t)(a.off[i + 1] - b);
                Ki = a.K[i];
                m = vertex_m(a, i, m0);
                inv_m = vertex_inv_m(a, i, inv0);
            }
            ed.load(a.tgt, w, i, b, deg, gl, LG);
#pragma unroll
            for (int u = 0; u < EPL; u++) c[u] = ed.j[u] != i ? ld_state<SYNC>(a.C + ed.j[u]) : d;
            const Decision<V> r = decide_warp<EPL, CH, SYNC, WT, F64, V>(a, LG, act, i, d, b, deg, Ki, m, inv_m, ed, c,
                                                                         it, tab, ceil_log2(CAP), lc);
            const bool moves = r.to != EMPTY;
            if (act && gl == 0) {
                if (moves && a.choice) a.choice[i] = r.to;
                record_visit(a, i, deg, Ki, (double)r.kid, r.gain, m, moves);
            }
            const unsigned movers = __ballot_sync(FULL, moves && gl == 0);
            if (!movers) continue;
            if constexpr (SYNC) {  // one reservation in the move list per round
                uint32_t base = 0;
                if (wl == 0) base = atomicAdd(a.mv_cnt, (uint32_t)__popc(movers));
                base = __shfl_sync(FULL, base, 0);
                if (moves && gl == 0) {
                    const uint32_t slot = base + __popc(movers & ((1u << wl) - 1u));
                    a.mv_vtx[slot] = i;
                    a.mv_cmt[slot] = r.to;
                }
            } else if (moves && gl == 0) {
                apply_now(a, i, d, r.to, Ki);
            }
            // movers re-mark their neighbours (frozen-state waves write a
            // separate array merged after the wave, so that the wave never
            // sees its marks)
            if (moves) {
#pragma unroll
                for (int u = 0; u < EPL; u++)
                    if (ed.j[u] != i) a.mark[ed.j[u]] = 1;
                for (uint64_t p = b + EPL * G + gl; p < b + deg; p += G) {
                    const uint32_t j = __ldg(a.tgt + p);
                    if (j != i) a.mark[j] = 1;
                }
            }
            __syncwarp();
        }
    }
    __syncwarp();  // the warp's tables are free for the next body
}

struct GroupLists {
    const uint32_t *list[4];
    uint32_t count[4];
    uint32_t bstart[5];  // block ranges of the four classes
};

template <typename WT, bool F64, int SYNC>
__global__ void __launch_bounds__(256, F64 ? 3 : 4) k_move_groups(MoveArgs a, GroupLists gl) {
    using V = typename std::conditional<F64, double, float>::type;
    constexpr size_t WREG = warp_tables<32, 256, V>;  // the largest of the four
    __shared__ __align__(16) unsigned char smem[8 * WREG];
    const uint32_t b = blockIdx.x, wid = threadIdx.x >> 5;
    unsigned char *ws = smem + wid * WREG;
    const int k = b < gl.bstart[1] ? 0 : b < gl.bstart[2] ? 1 : b < gl.bstart[3] ? 2 : 3;
    const uint32_t wb = (b - gl.bstart[k]) * 8 + wid, wn = (gl.bstart[k + 1] - gl.bstart[k]) * 8;
    LocalCtr lc;
    if (k == 0) group_body<4, 16, WT, F64, SYNC>(a, gl.list[0], gl.count[0], wb, wn, ws, lc);
    else if (k == 1) group_body<8, 32, WT, F64, SYNC>(a, gl.list[1], gl.count[1], wb, wn, ws, lc);
    else if (k == 2) group_body<16, 64, WT, F64, SYNC>(a, gl.list[2], gl.count[2], wb, wn, ws, lc);
    else group_body<32, 256, WT, F64, SYNC>(a, gl.list[3], gl.count[3], wb, wn, ws, lc);
    flush_counters(lc, a.ctr);
}

// Degrees 129..512: one warp per vertex, 1024-slot table per warp.
constexpr int W512_CAP = 1024;
template <typename WT, bool F64, int SYNC>
__global__ void __launch_bounds__(256, F64 ? 2 : 3) k_move_w512(MoveArgs a, const uint32_t *__restrict__ list, uint32_t count) {
    using V = typename std::conditional<F64, double, float>::type;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    const uint32_t wid = threadIdx.x >> 5;
    LocalCtr lc;
    group_body<32, W512_CAP, WT, F64, SYNC>(a, list, count, blockIdx.x * 8 + wid, gridDim.x * 8,
                                            dyn_smem + wid * warp_tables<32, W512_CAP, V>, lc);
    flush_counters(lc, a.ctr);
}

// Float64 weights of one community met by several lanes go to the table as one:
// a float64 add in shared memory is a loop of compare-and-swaps, in which the
// edges of a row with few communities queue (9 K vertices of degree 7 K in ten
// communities: a sweep 5.4 ms added one by one, 1.8 combined;
// R-MAT of 60 K vertices, the phase 7.1 -> 5.3).  Sums of exactly
// representable weights, exact in any order.  All 32 lanes; the first lane of a
// community keeps it, the others are left with EMPTY.
__device__ __forceinline__ void combine_lanes(uint32_t &c, double &v) {
    constexpr unsigned FULL = 0xFFFFFFFFu;
    const unsigned peers = __match_any_sync(FULL, c);
    unsigned m = c != EMPTY ? peers : 0u;
    if (!__any_sync(FULL, m & (m - 1u))) return;
    const int lane = threadIdx.x & 31, first = __ffs((int)m) - 1;
    double sum = 0.0;
    while (__any_sync(FULL, m)) {
        const double x = __shfl_sync(FULL, v, m ? __ffs((int)m) - 1 : lane);
        if (m) sum += x;
        m &= m - 1u;
    }
    v = sum;
    if (lane != first) c = EMPTY;
}

// --------------------------------------------------------------------------
// One block per vertex, table of up to CAP slots in shared memory.  Two block
// barriers a vertex: after the edges are inserted, and after their slots are
// scored and emptied; warp 0 decides while the others start the next vertex.
// A thread holds the slots of U edges; with more edges than the block's threads
// hold the table is read through instead.
// --------------------------------------------------------------------------
template <int CAP, int U, typename WT, bool F64, int SYNC>
__device__ void block_body(const MoveArgs &a, const uint32_t *__restrict__ list, uint32_t count, uint32_t lb,
                           uint32_t nb, unsigned char *dyn_smem, LocalCtr &lc, uint32_t slots = CAP) {
    using V = typename std::conditional<F64, double, float>::type;
    using SC = Score<F64>;
    using S = typename SC::S;
    constexpr unsigned FULL = 0xFFFFFFFFu;
    constexpr uint32_t CLAIM = 256;
    // all of the table is used whatever the degree; a degree above CAP / 2 comes
    // only on graphs of fewer than CAP vertices (move_level)
    const int logcap = ceil_log2(slots);
    Table<V> tab(dyn_smem, CAP, 0);
    __shared__ S red_s[32];
    __shared__ uint32_t red_c[32];
    __shared__ V red_k[32];
    __shared__ uint32_t s_todo[CLAIM], s_ntodo, s_wcnt[32];
    __shared__ uint8_t s_moved[CLAIM];
    const WT *w = static_cast<const WT *>(a.w);
    const double m0 = *a.m;
    const double inv0 = a.m[1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    for (uint32_t s = threadIdx.x; s < slots; s += blockDim.x) tab.clear(s);
    // The block's entries are lb + k * nb; CLAIM of them are claimed at
    // once (one flag per thread) and the active ones listed in shared memory,
    // so inactive vertices cost no serial round trip.
    for (uint64_t kb = 0; lb + kb * nb < count; kb += CLAIM) {
        const uint64_t my = lb + (kb + threadIdx.x) * nb;
        uint32_t vi = 0;
        int claim = 0;
        if (threadIdx.x < CLAIM && my < count) {
            vi = list[my];
            claim = ld_state<SYNC>(a.act + vi);
            if (claim) {
                a.act[vi] = 0;
                if (a.deferred) a.deferred[vi] = 0;
            }
        }
        const unsigned bal = __ballot_sync(FULL, claim);
        __syncthreads();  // the loop's previous step is done with s_todo
        if (lane == 0) s_wcnt[wid] = __popc(bal);
        __syncthreads();
        if (claim) {
            uint32_t pos = __popc(bal & ((1u << lane) - 1u));
            for (int k = 0; k < wid; k++) pos += s_wcnt[k];
            s_todo[pos] = vi;
        }
        if (threadIdx.x == 0) {
            uint32_t t = 0;
            for (int k = 0; k < nw; k++) t += s_wcnt[k];
            s_ntodo = t;
        }
        __syncthreads();
        const uint32_t ntodo = s_ntodo;
        for (uint32_t kk = 0; kk < ntodo; kk++) {
            const uint32_t i = s_todo[kk];
            const uint32_t d = ld_state<SYNC>(a.C + i);
            const uint64_t b = a.off[i], e = a.off[i + 1];
            const double Ki = a.K[i];
            const double Sd = ld_state<SYNC>(a.Sig + d);
            const uint32_t deg = (uint32_t)(e - b);
            const bool held = deg <= U * blockDim.x;  // every claimed slot is in its thread's registers
            uint32_t slot[U];
#pragma unroll
            for (int u = 0; u < U; u++) slot[u] = EMPTY;
            V kid = 0;
            for (uint64_t p0 = b; p0 < e; p0 += (uint64_t)U * blockDim.x) {  // the same trips for all threads
                uint32_t j[U], c[U];
                V wv[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const uint64_t p = p0 + (uint64_t)u * blockDim.x + threadIdx.x;
                    j[u] = p < e ? __ldg(a.tgt + p) : i;
                    wv[u] = p < e ? (V)__ldg(w + p) : V(0);
                }
#pragma unroll
                for (int u = 0; u < U; u++) c[u] = j[u] != i ? ld_state<SYNC>(a.C + j[u]) : EMPTY;
#pragma unroll
                for (int u = 0; u < U; u++) {
                    if (c[u] == d) {
                        kid += wv[u];
                        c[u] = EMPTY;
                    }
                    if constexpr (F64) combine_lanes(c[u], wv[u]);
                    if (c[u] != EMPTY) slot[u] = tab.add(logcap, c[u], wv[u]);
                }
            }
            kid = warp_sum(kid);
            if (lane == 0) red_k[wid] = kid;
            __syncthreads();  // every edge inserted
            kid = warp_sum(lane < nw ? red_k[lane] : V(0));
            const double m = vertex_m(a, i, m0);
            const SC sc = make_score<F64>(Ki, kid, Sd, m, vertex_inv_m(a, i, inv0), rounds_as_hub(deg));
            S best = -INFINITY;
            uint32_t bestc = EMPTY, ncand = 0;
            if (held) score_slots_warp<U, SYNC>(tab, slot, a.Sig, sc, best, bestc, ncand);
            else score_table<SYNC>(tab, slots, threadIdx.x, blockDim.x, a.Sig, sc, best, bestc, ncand);
            lc.candidates += ncand;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const S v2 = __shfl_xor_sync(FULL, best, o);
                const uint32_t c2 = __shfl_xor_sync(FULL, bestc, o);
                if (better(v2, c2, best, bestc)) { best = v2; bestc = c2; }
            }
            if (lane == 0) { red_s[wid] = best; red_c[wid] = bestc; }
            __syncthreads();  // every slot scored and emptied
            if (wid != 0) continue;
            best = lane < nw ? red_s[lane] : (S)-INFINITY;
            bestc = lane < nw ? red_c[lane] : EMPTY;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const S v2 = __shfl_xor_sync(FULL, best, o);
                const uint32_t c2 = __shfl_xor_sync(FULL, bestc, o);
                if (better(v2, c2, best, bestc)) { best = v2; bestc = c2; }
            }
            if (lane == 0) {
                const double gain = (bestc == EMPTY) ? 0.0 : sc.gain(best);
                int mv = 0;
                if (bestc != EMPTY && sc.gains(best)) mv = decide_move<SYNC>(a, i, d, bestc, Ki);
                lc.vertices++;
                lc.edges += deg;
                if (mv) { lc.moved++; lc.marked += deg; lc.dq += gain; add_graph_gain(a, i, gain); }
                record_visit(a, i, deg, Ki, (double)kid, gain, m, mv);
                s_moved[kk] = (uint8_t)mv;
            }
            __syncwarp();
        }
        __syncthreads();  // the decisions of the claimed vertices are in
        if (!a.mark) continue;
        for (uint32_t kk = 0; kk < ntodo; kk++) {
            if (!s_moved[kk]) continue;
            const uint32_t i = s_todo[kk];
            const uint64_t e = a.off[i + 1];
            for (uint64_t p = a.off[i] + threadIdx.x; p < e; p += blockDim.x) {
                const uint32_t j = __ldg(a.tgt + p);
                if (j != i) a.mark[j] = 1;
            }
        }
    }
    __syncthreads();  // the block's table is free for the next body
}

template <int CAP, int THREADS, typename WT, bool F64, int SYNC>
__global__ void __launch_bounds__(THREADS, F64 ? 1 : 1024 / THREADS) k_move_block(MoveArgs a, const uint32_t *__restrict__ list, uint32_t count) {
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    LocalCtr lc;
    // the block's threads hold the slots of the class's longest row (CAP / 2 edges)
    block_body<CAP, CAP / 2 / THREADS, WT, F64, SYNC>(a, list, count, blockIdx.x, gridDim.x, dyn_smem, lc);
    flush_counters(lc, a.ctr);
}

// --------------------------------------------------------------------------
// Apply a frozen-state wave's moves: C, Sigma and size updates (float64
// atomics of exactly representable values, so the result does not depend on
// their order).  The movers' neighbours were already re-marked, into the
// separate mark array, by the kernels that decided the moves (hub movers by
// k_mark_big).
// --------------------------------------------------------------------------

// Community totals change by +-K_i per move; movers of a wave crowd into a
// few large communities, so the deltas are first summed per block in a
// shared table (float64 sums of exactly representable values, exact in any
// order) and then applied with one atomic per community per block.
constexpr int APPLY_SLOG = 11;

// The block's delta of Sigma_c is summed either in float64 or, when K is in
// exact integer units of 2^lsb (lsb != INT_MIN), as a signed 64-bit integer
// (two's complement in an unsigned atomic add: one native shared-memory
// operation, where a float64 add loops on compare-and-swap under contention).
// Both sums are exact, so Sigma ends up the same.
__device__ __forceinline__ double signed_units_val(unsigned long long u, int lsb) {
    const long long v = (long long)u;
    return v < 0 ? -Acc<unsigned long long>::val((unsigned long long)(-v), lsb)
                 : Acc<unsigned long long>::val((unsigned long long)v, lsb);
}

// n = -1 or 1 member of weight k leaves or joins c; u: k in units.
__device__ __forceinline__ void apply_delta(uint32_t *keys, double *ds, int *dn, uint32_t c, double k,
                                            unsigned long long u, int n, double *Sig, uint32_t *size, int lsb) {
    uint32_t mask = (1u << APPLY_SLOG) - 1u;
    uint32_t h = hash32(c) >> (32 - APPLY_SLOG);
    for (uint32_t probe = 0; probe < 64; probe++) {
        uint32_t old = *(volatile uint32_t *)&keys[h];
        if (old == EMPTY) old = atomicCAS(&keys[h], EMPTY, c);
        if (old == EMPTY || old == c) {
            if (lsb != INT_MIN) atomicAdd(reinterpret_cast<unsigned long long *>(ds) + h, n < 0 ? 0ull - u : u);
            else atomicAdd(&ds[h], n < 0 ? -k : k);
            atomicAdd(&dn[h], n);
            return;
        }
        h = (h + 1) & mask;
    }
    atomicAdd(Sig + c, n < 0 ? -k : k);  // crowded table: apply directly
    atomicAdd(size + c, (uint32_t)n);
}

// Flush a block's delta table (slot t) into Sigma and size.
__device__ __forceinline__ void flush_delta(const uint32_t *keys, const double *ds, const int *dn, int t, double *Sig,
                                            uint32_t *size, int lsb) {
    const uint32_t c = keys[t];
    if (c == EMPTY) return;
    if (lsb != INT_MIN) {
        const unsigned long long u = reinterpret_cast<const unsigned long long *>(ds)[t];
        if (u) atomicAdd(Sig + c, signed_units_val(u, lsb));
    } else if (ds[t] != 0.0) {
        atomicAdd(Sig + c, ds[t]);
    }
    if (dn[t] != 0) atomicAdd(size + c, (uint32_t)dn[t]);
}

// act |= mark, mark = 0 (16 bytes per thread step) by blocks lb of nb.
__device__ __forceinline__ void merge_marks(uint8_t *act, uint8_t *mark, uint32_t n, uint32_t lb, uint32_t nb) {
    uint32_t n16 = n / 16;
    uint4 *a4 = reinterpret_cast<uint4 *>(act);
    uint4 *m4 = reinterpret_cast<uint4 *>(mark);
    for (uint32_t t = lb * blockDim.x + threadIdx.x; t < n16; t += nb * blockDim.x) {
        uint4 mk = m4[t];
        if (mk.x | mk.y | mk.z | mk.w) {
            uint4 ac = a4[t];
            ac.x |= mk.x; ac.y |= mk.y; ac.z |= mk.z; ac.w |= mk.w;
            a4[t] = ac;
            m4[t] = make_uint4(0, 0, 0, 0);
        }
    }
    for (uint32_t v = n16 * 16 + lb * blockDim.x + threadIdx.x; v < n; v += nb * blockDim.x) {
        if (mark[v]) { act[v] = 1; mark[v] = 0; }
    }
}

// The first `appliers` blocks apply the moves, the others merge the marks (two
// launches less the gap between them on a chain of launches per wave).
__global__ void __launch_bounds__(256) k_apply_moves(const uint32_t *__restrict__ mv_vtx,
                                                     const uint32_t *__restrict__ mv_cmt,
                                                     const uint32_t *__restrict__ mv_cnt, const double *__restrict__ K,
                                                     uint32_t *C, double *Sig, uint32_t *size, int lsb, uint32_t *left,
                                                     int *left_it, const int *iteration_dev, unsigned appliers,
                                                     uint8_t *act, uint8_t *mark, uint32_t n) {
    if (blockIdx.x >= appliers) {
        merge_marks(act, mark, n, blockIdx.x - appliers, gridDim.x - appliers);
        return;
    }
    const uint32_t cnt = *mv_cnt;
    if (blockIdx.x * blockDim.x >= cnt) return;
    __shared__ uint32_t skeys[1 << APPLY_SLOG];
    __shared__ double sds[1 << APPLY_SLOG];
    __shared__ int sdn[1 << APPLY_SLOG];
    for (int t = threadIdx.x; t < (1 << APPLY_SLOG); t += blockDim.x) { skeys[t] = EMPTY; sds[t] = 0.0; sdn[t] = 0; }
    __syncthreads();
    const int iteration = *iteration_dev;
    // four moves per thread and round, their loads in flight together: a warp of
    // the deciding kernel lists its movers side by side, vertices from all over
    // the wave's list (20 sweeps of one wave on a path of 470 K vertices: 3.9 ms
    // one by one, 2.4 so; 3.2 while movers were listed as they came)
    constexpr int U = 4;
    const uint64_t step = (uint64_t)appliers * blockDim.x;
    for (uint64_t t0 = blockIdx.x * blockDim.x + threadIdx.x; t0 < cnt; t0 += U * step) {
        uint32_t i[U], c[U], d[U];
        double k[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const uint64_t t = t0 + u * step;
            i[u] = t < cnt ? mv_vtx[t] : EMPTY;
            c[u] = t < cnt ? mv_cmt[t] : EMPTY;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (i[u] == EMPTY) continue;
            d[u] = C[i[u]];
            k[u] = K[i[u]];
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (i[u] == EMPTY) continue;
            C[i[u]] = c[u];
            left[i[u]] = d[u];
            left_it[i[u]] = iteration;
            const unsigned long long x = lsb != INT_MIN ? units_of(k[u], lsb) : 0ull;
            apply_delta(skeys, sds, sdn, d[u], k[u], x, -1, Sig, size, lsb);
            apply_delta(skeys, sds, sdn, c[u], k[u], x, 1, Sig, size, lsb);
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < (1 << APPLY_SLOG); t += blockDim.x) flush_delta(skeys, sds, sdn, t, Sig, size, lsb);
}

// Re-mark the neighbours of the big movers: block column x takes movers
// x, x + gridDim.x, ...; the gridDim.y blocks of a column split each mover's
// edges into interleaved slices.
__global__ void k_mark_big(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tgt,
                           const uint32_t *__restrict__ big, const uint32_t *__restrict__ nbig, uint8_t *act) {
    uint32_t cnt = *nbig;
    uint64_t step = (uint64_t)gridDim.y * blockDim.x;
    for (uint32_t t = blockIdx.x; t < cnt; t += gridDim.x) {
        uint32_t i = big[t];
        uint64_t b = off[i], e = off[i + 1];
        for (uint64_t p = b + (uint64_t)blockIdx.y * blockDim.x + threadIdx.x; p < e; p += step) {
            uint32_t j = tgt[p];
            if (j != i) act[j] = 1;
        }
    }
}

// --------------------------------------------------------------------------
// Persistent sweep: for graphs with no hub (every degree <= 2048) and at most
// a million or so vertices, a sweep of W waves costs 4-6 launches per wave on
// the normal path, and on small graphs those dependent launches, not the
// work, set the time.  Here one cooperative launch runs the whole sweep: per
// run of a wave, every block takes its share of each degree class (the same device
// bodies as the per-class kernels, frozen-state decisions into the wave's
// move list), a grid barrier, the moves applied and the re-marks merged,
// and a grid barrier.  Data written by earlier phases are read through L2
// (SYNC mode 2).  The barrier spins a bounded number of times: a block that
// gives up flags the sweep (MoveCounters::stalled) and the kernel returns.
// --------------------------------------------------------------------------
constexpr unsigned long long GRID_SYNC_SPINS = 1ull << 22;  // x 64 ns sleeps: about 0.3 s

__device__ bool grid_sync(GridBar *b, unsigned nb, MoveCounters *ctr) {
    __shared__ unsigned s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned ok = 1;
        volatile unsigned *vgen = &b->gen;
        const unsigned g = *vgen;
        __threadfence();
        if (atomicAdd(&b->arrive, 1u) == nb - 1) {
            b->arrive = 0;
            __threadfence();
            atomicAdd(&b->gen, 1u);
        } else {
            unsigned long long spins = 0;
            while (*vgen == g) {
                if (++spins > GRID_SYNC_SPINS || *(volatile unsigned *)&b->err) {
                    atomicExch(&b->err, 1u);
                    atomicAdd(&ctr->stalled, 1ull);
                    ok = 0;
                    break;
                }
                if (spins > 256) __nanosleep(32);  // poll tightly first: most waits are short
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Moves of a wave applied as k_apply_moves does, reading the move list, C
// and the count through L2; `smem` holds the block's delta table.
__device__ void apply_body_l2(const uint32_t *mv_vtx, const uint32_t *mv_cmt, const uint32_t *mv_cnt,
                              const double *__restrict__ K, uint32_t *C, double *Sig, uint32_t *size, uint32_t lb,
                              uint32_t nb, unsigned char *smem, int lsb, uint32_t *left, int *left_it, int iteration) {
    uint32_t *skeys = reinterpret_cast<uint32_t *>(smem);
    double *sds = reinterpret_cast<double *>(smem + sizeof(uint32_t) * (1u << APPLY_SLOG));
    int *sdn = reinterpret_cast<int *>(smem + (sizeof(uint32_t) + sizeof(double)) * (1u << APPLY_SLOG));
    for (int t = threadIdx.x; t < (1 << APPLY_SLOG); t += blockDim.x) { skeys[t] = EMPTY; sds[t] = 0.0; sdn[t] = 0; }
    __syncthreads();
    const uint32_t cnt = __ldcg(mv_cnt);
    for (uint32_t t = lb * blockDim.x + threadIdx.x; t < cnt; t += nb * blockDim.x) {
        const uint32_t i = __ldcg(mv_vtx + t), c = __ldcg(mv_cmt + t);
        const uint32_t d = __ldcg(C + i);
        const double Ki = K[i];
        C[i] = c;
        left[i] = d;
        left_it[i] = iteration;
        const unsigned long long u = lsb != INT_MIN ? units_of(Ki, lsb) : 0ull;
        apply_delta(skeys, sds, sdn, d, Ki, u, -1, Sig, size, lsb);
        apply_delta(skeys, sds, sdn, c, Ki, u, 1, Sig, size, lsb);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < (1 << APPLY_SLOG); t += blockDim.x) flush_delta(skeys, sds, sdn, t, Sig, size, lsb);
    __syncthreads();
}

__device__ void merge_body_l2(uint8_t *act, uint8_t *mark, uint32_t n, uint32_t lb, uint32_t nb) {
    const uint32_t n16 = n / 16;
    uint4 *a4 = reinterpret_cast<uint4 *>(act);
    uint4 *m4 = reinterpret_cast<uint4 *>(mark);
    for (uint32_t t = lb * blockDim.x + threadIdx.x; t < n16; t += nb * blockDim.x) {
        const uint4 mk = __ldcg(m4 + t);
        if (mk.x | mk.y | mk.z | mk.w) {
            uint4 ac = __ldcg(a4 + t);
            ac.x |= mk.x; ac.y |= mk.y; ac.z |= mk.z; ac.w |= mk.w;
            a4[t] = ac;
            m4[t] = make_uint4(0, 0, 0, 0);
        }
    }
    for (uint32_t v = n16 * 16 + lb * blockDim.x + threadIdx.x; v < n; v += nb * blockDim.x) {
        if (ldcg(mark + v)) { act[v] = 1; mark[v] = 0; }
    }
}

template <typename WT, bool F64>
__global__ void __launch_bounds__(256) k_sweep_persistent(MoveArgs a, const uint32_t *__restrict__ list,
                                                          const uint32_t *__restrict__ start, int W, int R,
                                                          uint32_t n, uint32_t *mv_cnts, GridBar *bar) {
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    const uint32_t lb = blockIdx.x, nb = gridDim.x;
    LocalCtr lc;  // one flush per block per sweep
    if (lb == 0)
        for (int t = threadIdx.x; t < W * R; t += blockDim.x) mv_cnts[t] = 0;
    if (!grid_sync(bar, nb, a.ctr)) return;
    for (int wr = 0; wr < W * R; wr++) {  // wave wr / R, repeat wr % R
        const int wv = wr / R;
        uint32_t cb[CLS_HUGE], cc[CLS_HUGE], tot = 0;
#pragma unroll
        for (int k = 0; k < CLS_HUGE; k++) {
            cb[k] = start[k * W + wv];
            cc[k] = start[k * W + wv + 1] - cb[k];
            tot += cc[k];
        }
        if (!tot) continue;  // the same for every block
        MoveArgs aw = a;
        aw.mv_cnt = mv_cnts + wr;
        {
            using V = typename std::conditional<F64, double, float>::type;
            const uint32_t wid = threadIdx.x >> 5, wb = lb * 8 + wid, wn = nb * 8;
            unsigned char *ws = dyn_smem + wid * warp_tables<32, W512_CAP, V>;
            group_body<4, 16, WT, F64, 2>(aw, list + cb[CLS_G4], cc[CLS_G4], wb, wn, ws, lc);
            group_body<8, 32, WT, F64, 2>(aw, list + cb[CLS_G8], cc[CLS_G8], wb, wn, ws, lc);
            group_body<16, 64, WT, F64, 2>(aw, list + cb[CLS_G16], cc[CLS_G16], wb, wn, ws, lc);
            group_body<32, 256, WT, F64, 2>(aw, list + cb[CLS_G32], cc[CLS_G32], wb, wn, ws, lc);
            group_body<32, W512_CAP, WT, F64, 2>(aw, list + cb[CLS_W512], cc[CLS_W512], wb, wn, ws, lc);
            __syncthreads();  // the block class uses the whole buffer
        }
        if (cc[CLS_BLOCK])
            block_body<4096, 8, WT, F64, 2>(aw, list + cb[CLS_BLOCK], cc[CLS_BLOCK], lb, nb, dyn_smem, lc);
        if (!grid_sync(bar, nb, a.ctr)) return;
        apply_body_l2(a.mv_vtx, a.mv_cmt, mv_cnts + wr, a.K, a.C, a.Sig, a.size, lb, nb, dyn_smem, a.lsb, a.left,
                      a.left_it, *a.iteration);
        merge_body_l2(a.act, a.mark, n, lb, nb);
        if (!grid_sync(bar, nb, a.ctr)) return;
    }
    flush_counters(lc, a.ctr);
}

// --------------------------------------------------------------------------
// Local moving of a small graph in one launch: every sweep of the phase, all
// waves and repeats, run by one thread-block cluster.
//
// What bounds a small graph (and the later, aggregated levels of every run)
// is the number of dependent steps, not the work in them: a sweep is W waves
// (times the repeats of the first iteration), each a decide step and an apply
// step that must see all of the other's writes; as launches a wave cost 17-25
// us in five kernels and memsets.  Inside one cluster the steps are parted by
// the hardware's cluster barrier, and the sweep's gain is tested against tau
// on the device, so the host neither launches nor waits between sweeps.  The
// rest is a chain of L2 round trips, kept short:
//   * a warp handles 32 lanes' worth of vertices of one class (8 of 4 lanes
//     ... 1 of 32 lanes) as one task; what of a task never changes (vertex,
//     row bounds, K, the first LEVEL_EPL targets and weights of each lane) is
//     fetched into registers between the arrival at a barrier and the wait;
//   * decide: trip 1 reads the flag, C_i and C_j, trip 2 Sigma and the sizes
//     of all candidates;
//   * a warp keeps its movers in shared memory and applies them itself after
//     the barrier: Sigma and size by atomics that nobody waits for, marks
//     straight into the flags (no vertex is deciding then).
// A cluster has at most 16 of the 152 SMs, so the host takes this path only
// while a wave's work fits them (move_level), with as few CTAs as give each
// task a warp.  Measured (611 vertices, 153 wave runs, one CTA): 5.4 us a run.
//
// Batches: per-graph gains and stopping as in the host loop (a graph whose
// gain of the sweep is <= tau stops, and its vertices become inactive).
// --------------------------------------------------------------------------
constexpr int LEVEL_CTAS = 16;       // non-portable cluster size; 8 when 16 do not fit the device
constexpr int LEVEL_THREADS = 512;
constexpr int LEVEL_WARPS = LEVEL_THREADS / 32;
constexpr int LEVEL_EPL = 4;         // edges a lane holds in registers
constexpr uint32_t LEVEL_TASKS = 6;  // most tasks of a warp in a wave ...
constexpr uint32_t LEVEL_MOVERS = 8 * LEVEL_TASKS;  // ... of at most 8 vertices each
constexpr uint32_t LEVEL_BMOVERS = 64;              // most vertices of the block classes per CTA and wave
constexpr int LEVEL_CAP = 16384;  // slots of the block classes' table

struct LevelArgs {
    const uint32_t *list, *start;  // class/wave lists (Classes)
    int W, R;                      // waves; repeats of a wave in the first iteration
    uint32_t n;
    double tau;
    int max_it;
    double *dq;                    // 3 gains of a sweep, zero at start
    int *iterations;               // out: sweeps run
    // batches (G == 0: one graph)
    uint32_t G;
    uint8_t *live;
    int *li;                       // sweeps of each graph
    uint32_t *nlive;               // 3 counts of the graphs still iterating, zero at start
};

// Barrier of all CTAs, split into arrival and wait; alone, a CTA's own barrier
// at the wait (a cluster barrier's release and acquire cost 0.7-1.3 us).  The
// aligned forms take whole warps, and the code before them parts the lanes
// (level_fetch between arrival and wait leaves the lanes without a vertex
// early): each half brings its warp together first.
__device__ __forceinline__ void level_arrive(bool alone) {
    __syncwarp();
    if (!alone) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void level_wait(bool alone) {
    __syncwarp();
    if (alone) __syncthreads();
    else asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

struct LevelMover {
    uint64_t b;
    double K;
    uint32_t i, c, d, deg;
};

template <bool F64> struct LevelSmem {
    using V = typename std::conditional<F64, double, float>::type;
    static constexpr size_t tables_bytes =
        std::max((size_t)LEVEL_WARPS * warp_tables<32, W512_CAP, V>,
                 (size_t)LEVEL_CAP * Table<V>::slot_bytes);
    alignas(16) unsigned char tables[tables_bytes];  // per-warp tables, or one table of a block class
    LevelMover mv[LEVEL_WARPS][LEVEL_MOVERS];
    uint32_t start[NUM_CLS * MAX_WAVES + 1];
};

// What a lane holds of its warp's task: the vertex of its group of 2^lg lanes
// (i == EMPTY: none), and the group's edges lane, lane + G, ...
template <typename WT> struct LevelTask {
    uint64_t b;
    double K, m, inv_m;
    uint32_t i, deg;
    int lg;
    LaneEdges<LEVEL_EPL, WT> ed;
};

// Number of warp tasks of class k with `count` vertices (lanes per vertex:
// 4, 8, 16, 32, 32 for the classes up to CLS_W512).
__host__ __device__ constexpr uint32_t level_lg(int k) { return k < 3 ? 2 + k : 5; }
__host__ __device__ constexpr uint32_t level_tasks(int k, uint32_t count) {
    return ((count << level_lg(k)) + 31) >> 5;
}

template <typename WT>
__device__ __forceinline__ void level_fetch(const MoveArgs &a, const uint32_t *__restrict__ list,
                                            const uint32_t *start, int W, int wv, uint32_t task, double m0, double inv0,
                                            LevelTask<WT> &t) {
    const uint32_t lane = threadIdx.x & 31;
    t.i = EMPTY;
    t.deg = 0;
    t.lg = 5;
    for (int k = CLS_W512; k >= CLS_G4; k--) {
        const uint32_t beg = start[k * W + wv], cnt = start[k * W + wv + 1] - beg;
        const uint32_t nt = level_tasks(k, cnt);
        if (task >= nt) { task -= nt; continue; }
        t.lg = (int)level_lg(k);
        const uint32_t idx = (task << (5 - t.lg)) + (lane >> t.lg);
        if (idx < cnt) t.i = list[beg + idx];
        break;
    }
    if (t.i == EMPTY) return;
    t.b = a.off[t.i];
    t.deg = (uint32_t)(a.off[t.i + 1] - t.b);
    t.K = a.K[t.i];
    t.m = vertex_m(a, t.i, m0);
    t.inv_m = vertex_inv_m(a, t.i, inv0);
    t.ed.load(a.tgt, static_cast<const WT *>(a.w), t.i, t.b, t.deg, lane & ((1u << t.lg) - 1u), t.lg);
}

// Decide the vertices of a task; movers are appended to mv[0..nmv).
template <typename WT, bool F64>
__device__ __forceinline__ void level_visit(const MoveArgs &a, const LevelTask<WT> &t, int it, unsigned char *ws,
                                            LevelMover *mv, uint32_t &nmv, LocalCtr &lc) {
    using V = typename std::conditional<F64, double, float>::type;
    constexpr unsigned FULL = 0xFFFFFFFFu;
    const uint32_t lane = threadIdx.x & 31, gl = lane & ((1u << t.lg) - 1u);
    const bool has = t.i != EMPTY;
    const bool act = has && ldcg(a.act + t.i);
    uint32_t d = 0, c[LEVEL_EPL];
    if (has) {
        d = ldcg(a.C + t.i);
#pragma unroll
        for (int u = 0; u < LEVEL_EPL; u++) c[u] = ldcg(a.C + t.ed.j[u]);
    }
    if (!__any_sync(FULL, act)) return;
    if (act && gl == 0) {
        a.act[t.i] = 0;
        if (a.deferred) a.deferred[t.i] = 0;
    }
    // the group's table: 16, 32 or 64 slots, then 256 and 1024
    const Table<V> tab(ws, W512_CAP, t.lg == 5 ? 0u : (lane >> t.lg) * (4u << t.lg));
    const Decision<V> r = decide_warp<LEVEL_EPL, 4, 2, WT, F64, V>(a, t.lg, act, t.i, d, t.b, t.deg, t.K, t.m, t.inv_m,
                                                                t.ed, c, it, tab, t.lg == 5 ? ceil_log2(W512_CAP) : t.lg + 2, lc);
    const bool moves = r.to != EMPTY && gl == 0;
    const unsigned bal = __ballot_sync(FULL, moves);
    if (moves) mv[nmv + __popc(bal & ((1u << lane) - 1u))] = LevelMover{t.b, t.K, t.i, r.to, d, t.deg};
    nmv += __popc(bal);
}

// One thread moves vertex i from d to c after the wave's barrier.
__device__ __forceinline__ void level_apply(const MoveArgs &a, uint32_t i, uint32_t c, uint32_t d, double Ki, int it) {
    a.C[i] = c;
    a.left[i] = d;
    a.left_it[i] = it;
    atomicAdd(a.Sig + d, -Ki);
    atomicAdd(a.Sig + c, Ki);
    atomicSub(a.size + d, 1u);
    atomicAdd(a.size + c, 1u);
}

template <typename WT, bool F64>
__global__ void __launch_bounds__(LEVEL_THREADS, 1) k_move_level(MoveArgs a, LevelArgs v) {
    using V = typename std::conditional<F64, double, float>::type;
    constexpr int CAP = LEVEL_CAP;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    LevelSmem<F64> &sm = *reinterpret_cast<LevelSmem<F64> *>(dyn_smem);
    __shared__ int s_it;
    __shared__ double s_red[32];
    __shared__ uint32_t s_bv[LEVEL_BMOVERS], s_bc[LEVEL_BMOVERS], s_bn;
    const uint32_t lb = blockIdx.x, nb = gridDim.x;
    const bool alone = nb == 1;
    const uint32_t tid = lb * LEVEL_THREADS + threadIdx.x, nt = nb * LEVEL_THREADS;
    const uint32_t wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // warp w of CTA b is number w * nb + b, so that few tasks spread over the CTAs
    const uint32_t wb = wid * nb + lb, wn = nb * LEVEL_WARPS;
    unsigned char *ws = sm.tables + wid * warp_tables<32, W512_CAP, V>;
    LevelMover *mv = sm.mv[wid];
    const double m0 = *a.m, inv0 = a.m[1];
    for (int t = threadIdx.x; t <= NUM_CLS * v.W; t += LEVEL_THREADS) sm.start[t] = v.start[t];
    auto clear_tables = [&]() {
        Table<V> tab(ws, W512_CAP, 0);
        for (int t = lane; t < W512_CAP; t += 32) tab.clear(t);
        __syncwarp();  // votes and shuffles do not order shared memory
    };
    clear_tables();
    __syncthreads();
    // the block classes' movers go to the CTA's list, applied after the barrier
    MoveArgs ab = a;
    ab.iteration = &s_it;
    ab.mv_vtx = s_bv;
    ab.mv_cmt = s_bc;
    ab.mv_cnt = &s_bn;
    ab.mark = nullptr;
    auto cls = [&](int k, int wv, uint32_t &beg) {
        beg = sm.start[k * v.W + wv];
        return sm.start[k * v.W + wv + 1] - beg;
    };
    auto next_wave = [&](int wv) {  // the next wave after wv with a vertex, or W
        for (wv++; wv < v.W; wv++) {
            uint32_t tot = 0, beg;
            for (int k = 0; k < NUM_CLS; k++) tot += cls(k, wv, beg);
            if (tot) break;
        }
        return wv;
    };
    LocalCtr lc;
    LevelTask<WT> t0;
    const int wave0 = next_wave(-1);
    int fetched = wave0;
    if (wave0 < v.W) level_fetch(a, v.list, sm.start, v.W, wave0, wb, m0, inv0, t0);
    int it = 0;
    for (;; it++) {
        if (threadIdx.x == 0) s_it = it;
        // sums of a sweep rotate through three slots: the next sweep's was
        // last read before this sweep's first barrier
        const int sum = it % 3;
        if (tid == 0) {
            v.dq[(it + 1) % 3] = 0.0;
            v.nlive[(it + 1) % 3] = 0;
        }
        lc.dq = 0.0;
        const int rep = it == 0 ? v.R : 1;
        for (int wv = wave0; wv < v.W;) {
            const int after = next_wave(wv);
            uint32_t tasks = 0, nblk = 0, beg;
            for (int k = CLS_G4; k <= CLS_W512; k++) tasks += level_tasks(k, cls(k, wv, beg));
            for (int k = CLS_BLOCK; k <= CLS_HUGE; k++) nblk += cls(k, wv, beg);
            for (int r = 0; r < rep; r++) {
                uint32_t nmv = 0;
                if (nblk) {  // the same for every CTA; the heaviest first: a whole CTA per vertex
                    if (threadIdx.x == 0) s_bn = 0;
                    __syncthreads();
                    for (int k = CLS_HUGE; k >= CLS_BLOCK; k--) {
                        const uint32_t cnt = cls(k, wv, beg);
                        const uint32_t slots = k == CLS_BLOCK ? 4096u : (uint32_t)CAP;
                        if (cnt) block_body<CAP, 4, WT, F64, 2>(ab, v.list + beg, cnt, lb, nb, sm.tables, lc, slots);
                    }
                    clear_tables();
                }
                if (wb < tasks) level_visit<WT, F64>(a, t0, it, ws, mv, nmv, lc);
                for (uint32_t x = wb + wn; x < tasks; x += wn) {
                    LevelTask<WT> t;
                    level_fetch(a, v.list, sm.start, v.W, wv, x, m0, inv0, t);
                    level_visit<WT, F64>(a, t, it, ws, mv, nmv, lc);
                }
                level_arrive(alone);  // every vertex of the wave has decided
                __syncwarp();      // the warp's movers are visible to its lanes
                if (r + 1 == rep) {
                    const int nx = after < v.W ? after : wave0;
                    if (nx != fetched) level_fetch(a, v.list, sm.start, v.W, nx, wb, m0, inv0, t0);
                    fetched = nx;
                }
                level_wait(alone);
                for (uint32_t x = lane; x < nmv; x += 32) {
                    const LevelMover q = mv[x];
                    level_apply(a, q.i, q.c, q.d, q.K, it);
                }
                // marks: four lanes per mover, the whole warp for the long rows
                for (uint32_t x = lane >> 2; x < nmv; x += 8) {
                    const LevelMover q = mv[x];
                    if (q.deg > 32) continue;
                    for (uint32_t p = lane & 3; p < q.deg; p += 4) {
                        const uint32_t j = __ldg(a.tgt + q.b + p);
                        if (j != q.i) a.act[j] = 1;
                    }
                }
                for (uint32_t x = 0; x < nmv; x++) {
                    const LevelMover q = mv[x];
                    if (q.deg <= 32) continue;
                    for (uint32_t p = lane; p < q.deg; p += 32) {
                        const uint32_t j = __ldg(a.tgt + q.b + p);
                        if (j != q.i) a.act[j] = 1;
                    }
                }
                if (nblk) {
                    __syncthreads();
                    for (uint32_t x = 0; x < s_bn; x++) {
                        const uint32_t i = s_bv[x];
                        const uint64_t b = a.off[i], e = a.off[i + 1];
                        if (threadIdx.x == 0) level_apply(a, i, s_bc[x], ldcg(a.C + i), a.K[i], it);
                        for (uint64_t p = b + threadIdx.x; p < e; p += LEVEL_THREADS) {
                            const uint32_t j = __ldg(a.tgt + p);
                            if (j != i) a.act[j] = 1;
                        }
                    }
                    __syncthreads();
                }
                level_arrive(alone);  // the wave's moves and marks are in place
                level_wait(alone);
            }
            wv = after;
        }
        // the sweep's gain; then every CTA takes the same decision
        const double dq = block_sum<double>(lc.dq, s_red);
        if (threadIdx.x == 0 && dq != 0.0) atomicAdd(v.dq + sum, dq);
        level_arrive(alone);
        level_wait(alone);
        if (!v.G) {
            if (it + 1 >= v.max_it || __ldcg(v.dq + sum) <= v.tau) break;
            continue;
        }
        uint32_t alive = 0;
        for (uint32_t g = tid; g < v.G; g += nt) {
            if (!ldcg(v.live + g)) continue;
            v.li[g] = it + 1;
            if (__ldcg(a.dq_g + g) <= v.tau) v.live[g] = 0;
            else alive = 1;
            a.dq_g[g] = 0.0;
        }
        alive = (uint32_t)__syncthreads_count(alive != 0);
        if (threadIdx.x == 0 && alive) atomicAdd(v.nlive + sum, alive);
        level_arrive(alone);
        level_wait(alone);
        if (it + 1 >= v.max_it || !__ldcg(v.nlive + sum)) break;
        for (uint32_t i = tid; i < v.n; i += nt)
            if (!ldcg(v.live + a.gid[i])) a.act[i] = 0;
        level_arrive(alone);
        level_wait(alone);
    }
    lc.dq = 0.0;  // reported per sweep
    flush_counters(lc, a.ctr);
    if (tid == 0) *v.iterations = it + 1;
}

// --------------------------------------------------------------------------
// Hub vertices (degree > 8192), processed by the whole grid:
//   prepare: read and clear each hub's flag, snapshot its community;
//   insert:  the hub's edges are cut into HUB_CHUNK-edge tasks; a block
//            combines a task's communities in a shared table, then its threads
//            publish the slots they claimed to the hub's global table;
//   score:   the hub's tasks read its table through, each its share of the
//            slots, score what is there and empty it; the block that ends last
//            for a hub reduces the tasks' bests and decides;
//   mark:    all blocks re-mark the movers' neighbours (k_mark_big).
// The tables are empty between waves, so nothing is cleared ahead and every
// wave uses the same memory.  Reading a table through moves 16-32 bytes an edge
// in whole lines (tables of 1.5 slots an edge instead of 2-4 moved less and were
// slower, R-MAT 24 98 -> 104 ms: longer probes); the list of occupied slots that it replaces was appended to
// behind a counter per block and cost a sector per entry to follow.
// The chain of a wave went from three memsets and five kernels to four kernels.
// --------------------------------------------------------------------------
constexpr int HUB_SLOG = 11;     // shared table of 2 * HUB_CHUNK slots
constexpr int HUB_THREADS = 512;  // 4 blocks of 32 registers a thread per SM: all its warps
constexpr int HUB_EPT = HUB_CHUNK / HUB_THREADS;  // edges of a task per thread

struct HubArgs {
    const uint32_t *hubs;
    uint32_t nh;
    const uint64_t *pool_off;  // per hub (nh + 1 entries): slots of its table
    const uint64_t *tasks;     // per hub: prefix of chunk counts (nh + 1 entries, tasks[0] = base)
    void *keys, *vals;         // the pool: 64-bit slots (float32) or keys and values (float64)
    void *kid;          // per hub, V
    uint8_t *go;        // per hub
    uint32_t *d;        // per hub
    uint32_t *done;     // per hub: tasks scored
    void *best_s;       // per task, S
    uint32_t *best_c;   // per task
    uint32_t *big, *nbig;
};

template <typename V> __device__ __forceinline__ Table<V> hub_table(const HubArgs &h, uint32_t t);
template <> __device__ __forceinline__ Table<float> hub_table<float>(const HubArgs &h, uint32_t t) {
    return Table<float>(static_cast<unsigned long long *>(h.keys) + (h.pool_off[t] - h.pool_off[0]));
}
template <> __device__ __forceinline__ Table<double> hub_table<double>(const HubArgs &h, uint32_t t) {
    const uint64_t o = h.pool_off[t] - h.pool_off[0];
    return Table<double>(static_cast<uint32_t *>(h.keys) + o, static_cast<double *>(h.vals) + o);
}

template <typename V, int SYNC>
__global__ void k_hub_prepare(MoveArgs a, HubArgs h) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *h.nbig = 0;
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < h.nh; t += gridDim.x * blockDim.x) {
        uint32_t i = h.hubs[t];
        uint8_t go = ld_state<SYNC>(a.act + i);
        if (go) {
            a.act[i] = 0;
            if (a.deferred) a.deferred[i] = 0;
        }
        h.go[t] = go;
        h.d[t] = ld_state<SYNC>(a.C + i);
        h.done[t] = 0;
        static_cast<V *>(h.kid)[t] = V(0);
    }
}

template <typename WT, bool F64, int SYNC>
__global__ void __launch_bounds__(HUB_THREADS, F64 ? 1 : 4) k_hub_insert(MoveArgs a, HubArgs h) {
    using V = typename std::conditional<F64, double, float>::type;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    Table<V> tab(dyn_smem, 1u << HUB_SLOG, 0);
    const WT *w = static_cast<const WT *>(a.w);
    V *kidv = static_cast<V *>(h.kid);
    for (uint32_t s = threadIdx.x; s < (1u << HUB_SLOG); s += HUB_THREADS) tab.clear(s);
    __syncthreads();
    const uint64_t base = h.tasks[0], total = h.tasks[h.nh] - base;
    for (uint64_t task = blockIdx.x; task < total; task += gridDim.x) {
        const uint32_t t = task_item(h.tasks, h.nh, task + base);
        if (!h.go[t]) continue;
        const uint32_t i = h.hubs[t], d = h.d[t];
        const uint64_t b0 = a.off[i], e1 = a.off[i + 1];
        const uint64_t b = b0 + (task + base - h.tasks[t]) * HUB_CHUNK;
        const uint64_t e = min(b + HUB_CHUNK, e1);
        uint32_t j[HUB_EPT], c[HUB_EPT], slot[HUB_EPT];
        V wv[HUB_EPT], kid = 0;
#pragma unroll
        for (int u = 0; u < HUB_EPT; u++) {
            const uint64_t p = b + u * HUB_THREADS + threadIdx.x;
            j[u] = p < e ? __ldg(a.tgt + p) : i;
            wv[u] = p < e ? (V)__ldg(w + p) : V(0);
        }
#pragma unroll
        for (int u = 0; u < HUB_EPT; u++) c[u] = j[u] != i ? ld_state<SYNC>(a.C + j[u]) : EMPTY;
#pragma unroll
        for (int u = 0; u < HUB_EPT; u++) {
            slot[u] = EMPTY;
            if (c[u] == EMPTY) continue;
            if (c[u] == d) kid += wv[u];
            else slot[u] = tab.add(HUB_SLOG, c[u], wv[u]);
        }
        kid = warp_sum(kid);
        if ((threadIdx.x & 31) == 0 && kid != V(0)) atomicAdd(kidv + t, kid);
        __syncthreads();  // the task is combined
        V val[HUB_EPT];
#pragma unroll
        for (int u = 0; u < HUB_EPT; u++) {
            c[u] = EMPTY;
            if (slot[u] == EMPTY) continue;
            c[u] = tab.get(slot[u], val[u]);
            tab.clear(slot[u]);
        }
        __syncthreads();  // the shared table is empty
        hub_table<V>(h, t).template publish<HUB_EPT>((uint32_t)(h.pool_off[t + 1] - h.pool_off[t] - 1), c, val);
    }
}

// The move of hub t, its tasks' bests all written: one warp.
template <bool F64, int SYNC>
__device__ void hub_decide(const MoveArgs &a, const HubArgs &h, uint32_t t, LocalCtr &lc) {
    using V = typename std::conditional<F64, double, float>::type;
    using SC = Score<F64>;
    using S = typename SC::S;
    const int lane = threadIdx.x & 31;
    const V *kidv = static_cast<const V *>(h.kid);
    const S *bs = static_cast<const S *>(h.best_s);
    const uint64_t base = h.tasks[0];
    const uint32_t i = h.hubs[t], d = h.d[t];
    S best = -INFINITY;
    uint32_t bestc = EMPTY;
    for (uint64_t k = h.tasks[t] - base + lane; k < h.tasks[t + 1] - base; k += 32) {
        const S v = __ldcg(bs + k);
        const uint32_t c = __ldcg(h.best_c + k);
        if (c != EMPTY && better(v, c, best, bestc)) { best = v; bestc = c; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        S v2 = __shfl_xor_sync(0xFFFFFFFFu, best, o);
        uint32_t c2 = __shfl_xor_sync(0xFFFFFFFFu, bestc, o);
        if (better(v2, c2, best, bestc)) { best = v2; bestc = c2; }
    }
    if (lane != 0) return;
    const double Ki = a.K[i];
    const uint64_t deg = a.off[i + 1] - a.off[i];
    const double m = vertex_m(a, i, a.m[0]);
    const SC sc = make_score<F64>(Ki, kidv[t], ld_state<SYNC>(a.Sig + d), m, vertex_inv_m(a, i, a.m[1]),
                                  rounds_as_hub(deg));
    const double gain = (bestc == EMPTY) ? 0.0 : sc.gain(best);
    int mv = 0;
    if (bestc != EMPTY && sc.gains(best)) mv = decide_move<SYNC>(a, i, d, bestc, Ki);
    lc.vertices++;
    lc.edges += deg;
    if (mv) {  // neighbours are re-marked by k_mark_big
        lc.moved++;
        lc.dq += gain;
        add_graph_gain(a, i, gain);
        lc.marked += deg;
        h.big[atomicAdd(h.nbig, 1u)] = i;
    }
    record_visit(a, i, (uint32_t)deg, Ki, (double)kidv[t], gain, m, mv);
}

// Scoring uses the insert's task split: task k of a hub's n tasks takes the
// slots [cap k / n, cap (k + 1) / n) of its table and leaves its best in
// best[task].
template <typename WT, bool F64, int SYNC>
__global__ void __launch_bounds__(HUB_THREADS, F64 ? 1 : 4) k_hub_score(MoveArgs a, HubArgs h) {
    using V = typename std::conditional<F64, double, float>::type;
    using SC = Score<F64>;
    using S = typename SC::S;
    __shared__ S red_s[32];
    __shared__ uint32_t red_c[32];
    __shared__ uint32_t s_last;
    const V *kidv = static_cast<const V *>(h.kid);
    S *bs = static_cast<S *>(h.best_s);
    const double m0 = a.m[0], inv0 = a.m[1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t base = h.tasks[0], total = h.tasks[h.nh] - base;
    LocalCtr lc;
    for (uint64_t task = blockIdx.x; task < total; task += gridDim.x) {
        const uint32_t t = task_item(h.tasks, h.nh, task + base);
        if (!h.go[t]) continue;
        const uint64_t n = h.tasks[t + 1] - h.tasks[t], k = task + base - h.tasks[t];
        const uint32_t i = h.hubs[t], d = h.d[t];
        const uint64_t cap = h.pool_off[t + 1] - h.pool_off[t];
        const uint64_t first = hub_share(cap, k, n);
        const uint32_t s0 = (uint32_t)first, slots = (uint32_t)(hub_share(cap, k + 1, n) - first);
        Table<V> tab = hub_table<V>(h, t);
        // hub_decide takes the score of staying; the candidates' do not read it in the mixed mode
        const SC sc = make_score<F64>(a.K[i], kidv[t], ld_state<SYNC>(a.Sig + d), vertex_m(a, i, m0),
                                      vertex_inv_m(a, i, inv0));
        S best = -INFINITY;
        uint32_t bestc = EMPTY, ncand = 0;
        // U slots per thread per round, their gathers of Sigma issued at once
        constexpr int U = 4;
        ScoreQueue<V> queue;
        for (uint32_t x0 = 0; x0 < slots; x0 += U * HUB_THREADS) {  // the same trips for all lanes
            const uint32_t x = x0 + threadIdx.x;
            uint32_t c[U];
            V val[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                const uint32_t y = x + u * HUB_THREADS;
                c[u] = EMPTY;
                val[u] = V(0);
                if (y < slots) c[u] = tab.get(s0 + y, val[u]);
            }
            if constexpr (F64) {
#pragma unroll
                for (int u = 0; u < U; u++) {
                    if (c[u] == EMPTY) continue;
                    tab.clear(s0 + x + u * HUB_THREADS);
                    ncand++;
                }
                queue.template put<SYNC>(c, val, a.Sig, sc, best, bestc);
            } else {
                double sg[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    sg[u] = 0.0;
                    if (c[u] == EMPTY) continue;
                    tab.clear(s0 + x + u * HUB_THREADS);
                    sg[u] = ld_state<SYNC>(a.Sig + c[u]);
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    if (c[u] == EMPTY) continue;
                    ncand++;
                    const S v = sc.score(val[u], sg[u]);
                    if (better(v, c[u], best, bestc)) { best = v; bestc = c[u]; }
                }
            }
        }
        if constexpr (F64) queue.template finish<SYNC>(a.Sig, sc, best, bestc);
        lc.candidates += ncand;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            S v2 = __shfl_xor_sync(0xFFFFFFFFu, best, o);
            uint32_t c2 = __shfl_xor_sync(0xFFFFFFFFu, bestc, o);
            if (better(v2, c2, best, bestc)) { best = v2; bestc = c2; }
        }
        __syncthreads();  // the previous task's reduction is over
        if (lane == 0) { red_s[wid] = best; red_c[wid] = bestc; }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int x = 1; x < HUB_THREADS / 32; x++)
                if (better(red_s[x], red_c[x], best, bestc)) { best = red_s[x]; bestc = red_c[x]; }
            bs[task] = best;
            h.best_c[task] = bestc;
            __threadfence();  // the best is visible before its task counts as done
            s_last = atomicAdd(h.done + t, 1u) == (uint32_t)n - 1;
        }
        __syncthreads();
        if (s_last && wid == 0) {
            __threadfence();
            hub_decide<F64, SYNC>(a, h, t, lc);
            __syncwarp();
        }
    }
    flush_counters(lc, a.ctr);
}

__global__ void k_hub_tasks(const uint64_t *__restrict__ off, const uint32_t *__restrict__ list, uint32_t count,
                            uint64_t *ntask) {
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < count; t += gridDim.x * blockDim.x) {
        uint32_t v = list[t];
        ntask[t] = (off[v + 1] - off[v] + HUB_CHUNK - 1) / HUB_CHUNK;
    }
}

// --------------------------------------------------------------------------
// Degree classes
// --------------------------------------------------------------------------
__device__ __forceinline__ int class_of(uint64_t deg, const ClassBounds &cb) {
    if (deg <= 8) return CLS_G4;
    if (deg <= 16) return CLS_G8;
    if (deg <= 32) return CLS_G16;
    if (deg <= cb.group_max) return CLS_G32;
    if (deg <= cb.warp_max) return CLS_W512;
    if (deg <= cb.block_max) return CLS_BLOCK;
    if (deg <= cb.big_max) return CLS_BIG;
    return CLS_HUGE;
}

// Wave of vertex v: a hash of its index within its graph, mod W.  The hash
// (the MurmurHash3 32-bit finaliser, Appleby) keeps arithmetic patterns of
// ids out of the waves: with the index itself, every community of a planted
// graph whose community count shares a factor with W (vertex v in community
// v mod k) fell into few waves, decided at once and cycled.
__device__ __forceinline__ uint32_t wave_hash(uint32_t x) {
    x ^= x >> 16;
    x *= 0x85ebca6bu;
    x ^= x >> 13;
    x *= 0xc2b2ae35u;
    x ^= x >> 16;
    return x;
}
__device__ __forceinline__ int wave_of(uint32_t v, int W, const uint32_t *gid, const uint64_t *gvo) {
    const uint32_t local = gid ? (uint32_t)(v - gvo[gid[v]]) : v;
    return (int)(wave_hash(local) % (uint32_t)W);
}

__global__ void k_classify_count(const uint64_t *__restrict__ off, uint32_t n, int W, uint32_t *counts,
                                 const uint32_t *__restrict__ gid, const uint64_t *__restrict__ gvo, ClassBounds cb) {
    __shared__ uint32_t sc[NUM_CLS * MAX_WAVES];
    for (int t = threadIdx.x; t < NUM_CLS * W; t += blockDim.x) sc[t] = 0;
    __syncthreads();
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        uint64_t deg = off[v + 1] - off[v];
        if (deg) atomicAdd(&sc[class_of(deg, cb) * W + wave_of(v, W, gid, gvo)], 1u);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < NUM_CLS * W; t += blockDim.x)
        if (sc[t]) atomicAdd(&counts[t], sc[t]);
}

// The lists, a tile of vertices per block and round: ranked by key in shared
// counters, then one reservation per key and tile.  (One per key and warp
// queued 32 K atomics on each hot key of a million vertices: 1.17 ms on R-MAT
// 24.)  With one wave a tile has a handful of keys, and the ranks queue in their
// counters: there the lanes of a key take theirs together (MATCH).  Small graphs
// take tiles of 256 vertices, so that the few there are spread over the SMs.
template <int PER, bool MATCH>
__global__ void __launch_bounds__(256) k_classify_fill(const uint64_t *__restrict__ off, uint32_t n, int W,
                                                       uint32_t *cursor, uint32_t *list,
                                                       const uint32_t *__restrict__ gid,
                                                       const uint64_t *__restrict__ gvo, ClassBounds cb) {
    __shared__ uint32_t num[NUM_CLS * MAX_WAVES];
    const int NK = NUM_CLS * W, lane = threadIdx.x & 31;
    for (uint64_t v0 = (uint64_t)blockIdx.x * 256 * PER; v0 < n; v0 += (uint64_t)gridDim.x * 256 * PER) {
        for (int t = threadIdx.x; t < NK; t += 256) num[t] = 0;
        __syncthreads();
        int key[PER];
        uint32_t rank[PER];
#pragma unroll
        for (int u = 0; u < PER; u++) {
            const uint64_t v = v0 + u * 256 + threadIdx.x;
            const uint64_t deg = v < n ? off[v + 1] - off[v] : 0;
            key[u] = deg ? class_of(deg, cb) * W + wave_of((uint32_t)v, W, gid, gvo) : -1;
            if (MATCH) {
                const unsigned peers = __match_any_sync(0xFFFFFFFFu, key[u]);
                const int leader = __ffs((int)peers) - 1;
                uint32_t base = 0;
                if (lane == leader && deg) base = atomicAdd(num + key[u], (uint32_t)__popc(peers));
                rank[u] = __shfl_sync(0xFFFFFFFFu, base, leader) + __popc(peers & ((1u << lane) - 1u));
            } else if (deg) {
                rank[u] = atomicAdd(num + key[u], 1u);
            }
        }
        __syncthreads();
        for (int t = threadIdx.x; t < NK; t += 256)
            if (num[t]) num[t] = atomicAdd(cursor + t, num[t]);
        __syncthreads();
#pragma unroll
        for (int u = 0; u < PER; u++)
            if (key[u] >= 0) list[num[key[u]] + rank[u]] = (uint32_t)(v0 + u * 256 + threadIdx.x);
        __syncthreads();
    }
}

__global__ void k_pool_caps(const uint64_t *__restrict__ off, const uint32_t *__restrict__ list, uint32_t count,
                            uint64_t *caps) {
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < count; t += gridDim.x * blockDim.x) {
        uint32_t v = list[t];
        caps[t] = hub_slots(off[v + 1] - off[v]);
    }
}

void classify_vertices(const DevGraph &g, Classes &cl, int waves, cudaStream_t s, const uint32_t *gid,
                       const uint64_t *gvo) {
    GSP_REQUIRE(waves >= 1 && waves <= MAX_WAVES, "waves must be in [1, %d]", MAX_WAVES);
    const int W = waves;
    const int NK = NUM_CLS * W;
    cl.W = W;
    uint32_t *counts = arena().get<uint32_t>(2 * NK);
    GSP_CUDA(cudaMemsetAsync(counts, 0, sizeof(uint32_t) * NK, s));
    unsigned grid = grid_for(g.n, 256, sms(8));
    const Tuning tn = tuning();
    const ClassBounds cb{tn.group_max, tn.warp_max, tn.block_max, tn.big_max};
    k_classify_count<<<grid, 256, 0, s>>>(g.off, g.n, W, counts, gid, gvo, cb);
    GSP_CHECK_LAUNCH();
    uint32_t h[NUM_CLS * MAX_WAVES];
    GSP_CUDA(cudaMemcpyAsync(h, counts, sizeof(uint32_t) * NK, cudaMemcpyDeviceToHost, s));
    GSP_CUDA(cudaStreamSynchronize(s));
    cl.start[0] = 0;
    for (int k = 0; k < NK; k++) cl.start[k + 1] = cl.start[k] + h[k];
    uint32_t *cursor = counts + NK;
    GSP_CUDA(cudaMemcpyAsync(cursor, cl.start, sizeof(uint32_t) * NK, cudaMemcpyHostToDevice, s));
    cl.list = arena().get<uint32_t>(cl.start[NK] + 1);
    const bool few = g.n <= 256ull * sms(4);  // tiles of 256: at most four a SM
    auto fill = [&](auto fn, unsigned tile) {
        fn<<<grid_for(g.n, tile, sms(8)), 256, 0, s>>>(g.off, g.n, W, cursor, cl.list, gid, gvo, cb);
    };
    if (W == 1) few ? fill(k_classify_fill<1, true>, 256) : fill(k_classify_fill<8, true>, 2048);
    else few ? fill(k_classify_fill<1, false>, 256) : fill(k_classify_fill<8, false>, 2048);
    GSP_CHECK_LAUNCH();
    cl.dstart = arena().get<uint32_t>(NK + 1);
    GSP_CUDA(cudaMemcpyAsync(cl.dstart, cl.start, sizeof(uint32_t) * (NK + 1), cudaMemcpyHostToDevice, s));
    uint32_t nh = cl.cls_count(CLS_HUGE);
    cl.pool_off = arena().get<uint64_t>(nh + 1);
    cl.pool_slots = 0;
    if (nh) {
        uint64_t *caps = arena().get<uint64_t>(nh);
        k_pool_caps<<<grid_for(nh, 256), 256, 0, s>>>(g.off, cl.list + cl.cls_begin(CLS_HUGE), nh, caps);
        GSP_CHECK_LAUNCH();
        exclusive_scan_u64(caps, cl.pool_off, nh, s);
        cl.host_pool_off.resize(nh + 1);
        GSP_CUDA(cudaMemcpyAsync(cl.host_pool_off.data(), cl.pool_off, sizeof(uint64_t) * (nh + 1),
                                 cudaMemcpyDeviceToHost, s));
        GSP_CUDA(cudaStreamSynchronize(s));
        cl.pool_slots = cl.host_pool_off[nh];
        uint64_t *ntask = arena().get<uint64_t>(nh);
        cl.hub_tasks = arena().get<uint64_t>(nh + 1);
        k_hub_tasks<<<grid_for(nh, 256), 256, 0, s>>>(g.off, cl.list + cl.cls_begin(CLS_HUGE), nh, ntask);
        GSP_CHECK_LAUNCH();
        exclusive_scan_u64(ntask, cl.hub_tasks, nh, s);
        cl.host_hub_tasks.resize(nh + 1);
        GSP_CUDA(cudaMemcpyAsync(cl.host_hub_tasks.data(), cl.hub_tasks, sizeof(uint64_t) * (nh + 1),
                                 cudaMemcpyDeviceToHost, s));
        GSP_CUDA(cudaStreamSynchronize(s));
    }
}

// --------------------------------------------------------------------------
// Host launchers
// --------------------------------------------------------------------------
SideStreams &side_streams() {
    static SideStreams ss[16];
    static bool made[16] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    dev &= 15;
    if (!made[dev]) {
        for (int k = 0; k < SideStreams::N; k++)
            GSP_CUDA(cudaStreamCreateWithFlags(&ss[dev].side[k], cudaStreamNonBlocking));
        for (int f = 0; f < 64; f++) {
            GSP_CUDA(cudaEventCreateWithFlags(&ss[dev].fork_ev[f], cudaEventDisableTiming));
            for (int k = 0; k < SideStreams::N; k++)
                GSP_CUDA(cudaEventCreateWithFlags(&ss[dev].join_ev[f][k], cudaEventDisableTiming));
        }
        made[dev] = true;
    }
    return ss[dev];
}

// The class kernels of a wave touch disjoint vertices and only append to the
// move list, so they run as parallel branches: W512 and the block class on
// side streams 0 and 1, the hub chain on side stream 2, the big-table block
// class on side stream 3, the group classes on the main stream; all join
// before the wave's moves are applied.  A wave without group classes has its
// first other class on the main stream: in-place waves launch nothing after the
// join, and a main stream that only waits hands the kernels of all earlier waves
// to the next one as dependencies (64 waves of 2 K vertices of degree 400: 3.1 ms
// to instantiate the sweep's graph instead of 0.1).
template <typename WT, bool F64, int SYNC>
static void launch_wave(const Classes &cl, const MoveArgs &a, int wave, void *pool, uint32_t *big, uint32_t *nbig,
                        cudaStream_t main) {
    using V = typename std::conditional<F64, double, float>::type;
    SideStreams &ss = side_streams();
    const int f = ss.next;
    ss.next = (ss.next + 1) & 63;
    bool used[SideStreams::N] = {false, false, false, false};
    GSP_CUDA(cudaEventRecord(ss.fork_ev[f], main));
    bool main_free = true;  // nothing of this wave on the main stream yet
    auto on = [&](int k) -> cudaStream_t {
        if (main_free) {
            main_free = false;
            return main;
        }
        if (!used[k]) {
            GSP_CUDA(cudaStreamWaitEvent(ss.side[k], ss.fork_ev[f], 0));
            used[k] = true;
        }
        return ss.side[k];
    };
    cudaStream_t s = main;
    const Tuning tn = tuning();
    const int sm = sm_count();
    GroupLists gl;
    const int G[4] = {4, 8, 16, 32};
    uint32_t blocks = 0;
    for (int c = 0; c < 4; c++) {
        gl.list[c] = cl.list + cl.begin(c, wave);
        gl.count[c] = cl.count(c, wave);
        gl.bstart[c] = blocks;
        if (gl.count[c]) blocks += grid_for((uint64_t)gl.count[c] * G[c], 256, (uint32_t)(sm * tn.groups));
    }
    gl.bstart[4] = blocks;
    if (blocks) {
        k_move_groups<WT, F64, SYNC><<<blocks, 256, 0, s>>>(a, gl);
        GSP_CHECK_LAUNCH();
        note_cap(CAP_GROUPS);
        main_free = false;
    }
    uint32_t nw5 = cl.count(CLS_W512, wave);
    if (nw5) {
        constexpr size_t smem = (size_t)8 * W512_CAP * (sizeof(uint32_t) + sizeof(V));
        static bool attr = false;
        if (!attr) {
            GSP_CUDA(cudaFuncSetAttribute(k_move_w512<WT, F64, SYNC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)smem));
            attr = true;
        }
        k_move_w512<WT, F64, SYNC><<<grid_for((uint64_t)nw5 * 32, 256, (uint32_t)(sm * tn.w512)), 256, smem, on(0)>>>(
            a, cl.list + cl.begin(CLS_W512, wave), nw5);
        GSP_CHECK_LAUNCH();
        note_cap(CAP_W512);
    }
    uint32_t nb = cl.count(CLS_BLOCK, wave);
    if (nb) {
        constexpr int CAP = 4096, THREADS = 256;
        constexpr size_t smem = CAP * Table<V>::slot_bytes;
        const auto fn = k_move_block<CAP, THREADS, WT, F64, SYNC>;
        static bool attr = false;
        if (!attr) {
            GSP_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            attr = true;
        }
        fn<<<grid_for(nb, 1, (uint32_t)(sm * tn.block)), THREADS, smem, on(1)>>>(a, cl.list + cl.begin(CLS_BLOCK, wave),
                                                                                nb);
        GSP_CHECK_LAUNCH();
        note_cap(CAP_BLOCK);
    }
    uint32_t ng = cl.count(CLS_BIG, wave);
    if (ng) {
        // 2049..8192 edges: one block per vertex with a 16384-slot shared
        // table (twice the most edges); the table leaves room for one block
        // per SM, so the block is as large as the registers allow
        constexpr int CAP = 16384, THREADS = F64 ? 512 : 1024;
        constexpr size_t smem = CAP * Table<V>::slot_bytes;
        const auto fn = k_move_block<CAP, THREADS, WT, F64, SYNC>;
        static bool attr = false;
        if (!attr) {
            GSP_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            attr = true;
        }
        fn<<<grid_for(ng, 1, (uint32_t)sm), THREADS, smem, on(3)>>>(a, cl.list + cl.begin(CLS_BIG, wave), ng);
        GSP_CHECK_LAUNCH();
    }
    uint32_t nh = cl.count(CLS_HUGE, wave);
    if (nh) {
        cudaStream_t s = on(2);
        using S = typename Score<F64>::S;
        uint32_t rel = cl.begin(CLS_HUGE, wave) - cl.cls_begin(CLS_HUGE);
        size_t mk = arena().mark();
        HubArgs h;
        h.hubs = cl.list + cl.begin(CLS_HUGE, wave);
        h.nh = nh;
        h.pool_off = cl.pool_off + rel;
        h.tasks = cl.hub_tasks + rel;
        h.keys = pool;
        h.vals = F64 ? static_cast<uint32_t *>(pool) + align_up(cl.wave_pool_slots(), 64) : nullptr;
        h.kid = arena().alloc(sizeof(V) * nh);
        h.go = arena().get<uint8_t>(nh);
        h.d = arena().get<uint32_t>(nh);
        h.done = arena().get<uint32_t>(nh);
        uint64_t ntasks = cl.host_hub_tasks[rel + nh] - cl.host_hub_tasks[rel];
        h.best_s = arena().alloc(sizeof(S) * ntasks);
        h.best_c = arena().get<uint32_t>(ntasks);
        h.big = big;
        h.nbig = nbig;
        k_hub_prepare<V, SYNC><<<grid_for(nh, 256), 256, 0, s>>>(a, h);
        GSP_CHECK_LAUNCH();
        constexpr size_t hsmem = Table<V>::slot_bytes << HUB_SLOG;
        // one block per task at most: small waves launch only what they use
        note_cap(CAP_HUB);
        const unsigned hub_grid = (unsigned)std::min<uint64_t>(ntasks, (uint64_t)sm * tn.hub);
        k_hub_insert<WT, F64, SYNC><<<hub_grid, HUB_THREADS, hsmem, s>>>(a, h);
        GSP_CHECK_LAUNCH();
        k_hub_score<WT, F64, SYNC><<<hub_grid, HUB_THREADS, 0, s>>>(a, h);
        GSP_CHECK_LAUNCH();
        k_mark_big<<<dim3(sm, 16), 256, 0, s>>>(a.off, a.tgt, big, nbig, a.mark);
        GSP_CHECK_LAUNCH();
        arena().release(mk);
    }
    for (int k = 0; k < SideStreams::N; k++) {
        if (!used[k]) continue;
        GSP_CUDA(cudaEventRecord(ss.join_ev[f][k], ss.side[k]));
        GSP_CUDA(cudaStreamWaitEvent(main, ss.join_ev[f][k], 0));
    }
}

static MoveArgs make_move_args(const DevGraph &g, const MoveBuffers &mb, bool sync, bool rule, int iteration,
                               int max_iterations) {
    MoveArgs a;
    a.off = g.off;
    a.tgt = g.tgt;
    a.w = g.w;
    a.C = mb.C;
    a.K = mb.K;
    a.Sig = mb.Sigma;
    a.size = mb.size;
    a.act = mb.act;
    a.mark = sync ? mb.mark : mb.act;
    a.m = mb.m_dev;
    a.gid = mb.gid;
    a.m_g = mb.m_g;
    a.minv_g = mb.minv_g;
    a.lsb = mb.lsb;
    a.dq_g = mb.dq_g;
    a.ctr = mb.ctr;
    a.rule = rule ? 1 : 0;
    a.left = mb.left;
    a.left_it = mb.left_it;
    a.iteration = mb.it_dev;
    a.no_return_from = mb.no_return_from;
    a.mv_vtx = mb.mv_vtx;
    a.mv_cmt = mb.mv_cmt;
    a.mv_cnt = mb.mv_cnt;
    a.choice = mb.choice;
    a.feat_kept = mb.feat_kept;
    a.feat_gain = mb.feat_gain;
    a.last_gain = mb.last_gain;
    a.moved_last = mb.moved_last;
    a.deferred = mb.skip;
    a.trace_x = mb.trace_x;
    a.trace_y = mb.trace_y;
    a.trace_cnt = mb.trace_cnt;
    a.trace_cap = mb.trace_cap;
    a.trace_keys = mb.trace_keys;
    a.trace_tag = ((uint64_t)(mb.trace_pass & 0xFF) << 56) | ((uint64_t)(mb.cur_repeat & 0xFF) << 40);
    a.trace_every = mb.trace_every ? mb.trace_every : 1;
    a.max_logk = mb.max_logk;
    a.max_iterations = max_iterations;
    a.salt = mb.trace_salt;
    return a;
}

template <typename WT, bool F64>
static bool launch_persistent(const MoveArgs &a, const Classes &cl, uint32_t n, MoveBuffers &mb, int iteration,
                              cudaStream_t s) {
    using V = typename std::conditional<F64, double, float>::type;
    constexpr size_t smem = std::max(std::max(8 * warp_tables<32, W512_CAP, V>, 4096 * Table<V>::slot_bytes),
                                     (size_t)(sizeof(uint32_t) + sizeof(double) + sizeof(int)) << APPLY_SLOG);
    static int per_sm[64] = {0};  // resident blocks per SM, per device (-1: cannot run)
    int dev = 0;
    GSP_CUDA(cudaGetDevice(&dev));
    dev &= 63;
    if (!per_sm[dev]) {
        GSP_CUDA(cudaFuncSetAttribute(k_sweep_persistent<WT, F64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem));
        int coop = 0, nblk = 0;
        GSP_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
        GSP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nblk, k_sweep_persistent<WT, F64>, 256, smem));
        per_sm[dev] = (coop && nblk > 0) ? nblk : -1;
    }
    if (per_sm[dev] < 0) return false;
    MoveArgs aa = a;
    const uint32_t *list = cl.list;
    const uint32_t *start = cl.dstart;
    int W = cl.W;
    int R = std::min(wave_repeats_at(mb, iteration), MAX_REPEATS);
    uint32_t nn = n;
    uint32_t *cnts = mb.mv_cnts;
    GridBar *bar = mb.bar;
    void *args[] = {&aa, &list, &start, &W, &R, &nn, &cnts, &bar};
    GSP_CUDA(cudaMemsetAsync(bar, 0, sizeof(GridBar), s));
    GSP_CUDA(cudaLaunchCooperativeKernel((const void *)k_sweep_persistent<WT, F64>, dim3(per_sm[dev] * sm_count()),
                                         dim3(256), args, smem, s));
    count_launch();
    return true;
}

// The caller asked for the persistent sweep on graphs of this size
// (gsp_tuning.persist_max_vertices), and the graph and the run qualify.
static bool persistent_asked(const DevGraph &g, const Classes &cl, const MoveBuffers &mb) {
    return g.n <= tuning().persist_max_vertices && !cl.cls_count(CLS_HUGE) && !cl.cls_count(CLS_BIG) &&
           !mb.feat_kept && !mb.choice && cl.dstart && mb.bar;
}

bool sweep_persistent(const DevGraph &g, const Classes &cl, MoveBuffers &mb, bool fp64, bool rule, int iteration,
                      int max_iterations, cudaStream_t s) {
    if (!persistent_asked(g, cl, mb)) return false;
    MoveArgs a = make_move_args(g, mb, true, rule, iteration, max_iterations);
    if (g.wt == GSP_W_F32) return fp64 ? launch_persistent<float, true>(a, cl, g.n, mb, iteration, s)
                                       : launch_persistent<float, false>(a, cl, g.n, mb, iteration, s);
    return fp64 ? launch_persistent<double, true>(a, cl, g.n, mb, iteration, s)
                : launch_persistent<double, false>(a, cl, g.n, mb, iteration, s);
}

template <typename WT, bool F64>
static bool launch_level(const MoveArgs &a, const LevelArgs &v, int ctas_needed, int ctas_wanted, cudaStream_t s) {
    constexpr size_t smem = sizeof(LevelSmem<F64>);
    static int ctas[64] = {0};  // CTAs of the cluster, per device (-1: cannot run)
    int dev = 0;
    GSP_CUDA(cudaGetDevice(&dev));
    dev &= 63;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(LEVEL_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const auto fn = k_move_level<WT, F64>;
    if (!ctas[dev]) {
        GSP_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        GSP_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        int found = -1;
        for (int c = LEVEL_CTAS; c >= 8 && found < 0; c /= 2) {
            at[0].val.clusterDim.x = c;
            cfg.gridDim = dim3(c);
            int clusters = 0;
            if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) == cudaSuccess && clusters > 0) found = c;
            else cudaGetLastError();
        }
        ctas[dev] = found;
    }
    if (ctas[dev] < ctas_needed) return false;
    const int c = std::min(ctas[dev], ctas_wanted);
    at[0].val.clusterDim.x = c;
    cfg.gridDim = dim3(c);
    GSP_CUDA(cudaLaunchKernelEx(&cfg, fn, a, v));
    count_launch();
    return true;
}

// Most stored entries of a graph that one cluster moves.  Measured on GB300,
// whole local-moving phase (gsp_local_move), launches / cluster:
//   mixed    planted, degree 16: 312 K entries 1.28, 408 K 1.08, 504 K 0.97, 536 K
//            0.98; degree 48: 448 K 1.14, 537 K 1.11; grids 492 K 1.09, 519 K
//            1.05, 548 K 0.98, 669 K 0.91; R-MAT 417 K 1.10, 541 K 1.07, 600 K
//            1.01; dense graphs of 2 K vertices: planted 499 K 1.45, 940 K 1.31,
//            R-MAT 416 K 1.08
//   float64  planted, degree 16: 139 K 1.13, 171 K 1.03, 187 K 0.99, 203 K 0.87;
//            degree 32: 148 K 1.16, 212 K 0.89; grids 151 K 1.06, 183 K 1.03,
//            201 K 0.98, 237 K 0.94; R-MAT 75 K 1.04, 122 K 0.98, 157 K 1.03,
//            200 K 0.98, 276 K 0.94
//   float64, at most 2048 vertices: planted 225 K 1.33, 248 K 1.37, 328 K 1.18,
//            410 K 1.08; 1500 vertices 210 K 1.15, 281 K 1.00, 377 K 0.94; R-MAT
//            104 K 1.11, 152 K 0.95, 241 K 0.86
// What the float64 mode costs on 16 SMs is its divisions, one pair a candidate:
// rows whose neighbours soon share a few communities gain longer than rows whose
// do not (R-MAT), which the entries cannot tell.  The dense limit is drawn for
// the former: dense levels come from aggregation.
constexpr uint64_t LEVEL_MAX_EDGES = 1u << 19, LEVEL_MAX_EDGES_F64 = 160000, LEVEL_MAX_EDGES_F64_DENSE = 1u << 18;
constexpr uint32_t LEVEL_DENSE_VERTICES = 2048;

bool move_level(const DevGraph &g, const Classes &cl, MoveBuffers &mb, bool fp64, bool rule, double tau, int max_it,
                LevelResult &out, uint32_t G, uint8_t *live, int *li, cudaStream_t s) {
    const uint64_t most = !fp64                              ? LEVEL_MAX_EDGES
                          : g.n <= LEVEL_DENSE_VERTICES ? LEVEL_MAX_EDGES_F64_DENSE
                                                        : LEVEL_MAX_EDGES_F64;
    if (g.nnz > most || mb.feat_kept || mb.choice || !cl.dstart || persistent_asked(g, cl, mb)) return false;
    // a vertex's communities must fit the block classes' table
    if (g.n > LEVEL_CAP * 3 / 4 && cl.cls_count(CLS_HUGE)) return false;
    // a wave must fit the warps' task and mover lists, and the CTAs' lists of block-class movers
    int need = 1;
    uint64_t busiest = 0;
    for (int wv = 0; wv < cl.W; wv++) {
        uint64_t tasks = 0, blk = 0;
        for (int k = CLS_G4; k <= CLS_W512; k++) tasks += level_tasks(k, cl.count(k, wv));
        // a CTA takes its share of each block class, rounded up
        for (int k = CLS_BLOCK; k <= CLS_HUGE; k++) blk += cl.count(k, wv);
        const uint64_t c = std::max((tasks + LEVEL_TASKS * LEVEL_WARPS - 1) / (LEVEL_TASKS * LEVEL_WARPS),
                                    (blk + LEVEL_BMOVERS - 4) / (LEVEL_BMOVERS - 3));
        if (c > LEVEL_CTAS) return false;
        need = std::max(need, (int)c);
        busiest = std::max(busiest, tasks + 64 * blk);
    }
    // one task per warp where that takes more than one CTA; fewer CTAs make the
    // barriers cheaper, and one needs none between CTAs
    int want = LEVEL_CTAS;
    while (want > 1 && busiest <= (uint64_t)(want / 2) * LEVEL_WARPS) want /= 2;
    while (want < need) want *= 2;
    MoveArgs a = make_move_args(g, mb, true, rule, 0, max_it);
    struct Scratch { double dq[3]; uint32_t nlive[3]; int iterations; };
    static_assert(sizeof(Scratch) <= sizeof(uint32_t) * MAX_WAVES * MAX_REPEATS, "the persistent sweep's counters hold it");
    Scratch *d = reinterpret_cast<Scratch *>(mb.mv_cnts);
    GSP_CUDA(cudaMemsetAsync(d, 0, sizeof(Scratch), s));
    GSP_CUDA(cudaMemsetAsync(mb.ctr, 0, sizeof(MoveCounters), s));
    const LevelArgs v{cl.list, cl.dstart, cl.W, std::min(std::max(mb.repeats, 1), MAX_REPEATS), g.n, tau, max_it,
                      d->dq, &d->iterations, G, live, li, d->nlive};
    bool ran;
    if (g.wt == GSP_W_F32) ran = fp64 ? launch_level<float, true>(a, v, need, want, s) : launch_level<float, false>(a, v, need, want, s);
    else ran = fp64 ? launch_level<double, true>(a, v, need, want, s) : launch_level<double, false>(a, v, need, want, s);
    if (ran) {
        GSP_CUDA(cudaMemcpyAsync(&out.iterations, &d->iterations, sizeof(int), cudaMemcpyDeviceToHost, s));
        GSP_CUDA(cudaMemcpyAsync(&out.ctr, mb.ctr, sizeof(MoveCounters), cudaMemcpyDeviceToHost, s));
    }
    return ran;
}

void move_wave(const DevGraph &g, const Classes &cl, MoveBuffers &mb, int wave, bool sync, bool fp64, bool rule,
               bool learned, int iteration, int max_iterations, cudaStream_t s) {
    (void)learned;
    MoveArgs a = make_move_args(g, mb, sync, rule, iteration, max_iterations);
#define GSP_WAVE(WT, F64, SYNC) \
    launch_wave<WT, F64, SYNC>(cl, a, wave, mb.pool, mb.big, mb.nbig, s)
    if (g.wt == GSP_W_F32) {
        if (fp64) { if (sync) GSP_WAVE(float, true, true); else GSP_WAVE(float, true, false); }
        else { if (sync) GSP_WAVE(float, false, true); else GSP_WAVE(float, false, false); }
    } else {
        if (fp64) { if (sync) GSP_WAVE(double, true, true); else GSP_WAVE(double, true, false); }
        else { if (sync) GSP_WAVE(double, false, true); else GSP_WAVE(double, false, false); }
    }
#undef GSP_WAVE
}

void apply_moves(const DevGraph &g, MoveBuffers &mb, uint32_t n_hint, cudaStream_t s) {
    const unsigned appliers = grid_for(n_hint, 256, sms(4));
    const unsigned mergers = grid_for(g.n / 16 + 1, 256, sms(4));
    k_apply_moves<<<appliers + mergers, 256, 0, s>>>(mb.mv_vtx, mb.mv_cmt, mb.mv_cnt, mb.K, mb.C, mb.Sigma, mb.size,
                                                     mb.lsb, mb.left, mb.left_it, mb.it_dev, appliers, mb.act, mb.mark,
                                                     g.n);
    GSP_CHECK_LAUNCH();
}

}  // namespace gsp
