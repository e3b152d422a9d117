// misc.cu -- vertex weights (Section 3), modularity (Equation 1), community
// renumbering and dendrogram lookup (Algorithm 1), the final numbering, and
// the disconnected-community count (Algorithm 6).
//
// Row sums use one thread per row up to 64 entries, one warp per row up to
// 8192 and one block per longer row.  Their sums of weights are exact and so
// do not depend on the order: in integer units of the weights' lowest set bit
// when the total fits 2^52 such units (exact_lsb), otherwise in float64 over
// float32-representable weights whose partial sums stay representable.
#include <cmath>
#include <cstring>
#include <type_traits>

#include "internal.cuh"

namespace gsp {

constexpr uint32_t SHORT_ROW = 64;

// f(x) for every x[i], i < n, 16 bytes at a time and four of them in flight;
// x need only be aligned to its elements (the ends are read one by one).  Grids
// have a thread per 16 bytes up to eight blocks an SM: with four of them per
// thread also on small inputs, 40 K entries took 5.0 us instead of 2.8.
template <typename T, typename F> __device__ __forceinline__ void for_each_16b(const T *__restrict__ x, uint64_t n, F &&f) {
    constexpr int PER = 16 / sizeof(T);
    const uint64_t tid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, nt = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t head = min(n, (uint64_t)((16 - (reinterpret_cast<uintptr_t>(x) & 15)) & 15) / sizeof(T));
    const uint64_t vecs = (n - head) / PER;
    const uint4 *v = reinterpret_cast<const uint4 *>(x + head);
    auto each = [&](const uint4 &q) {
        T e[PER];
        memcpy(e, &q, 16);
#pragma unroll
        for (int k = 0; k < PER; k++) f(e[k]);
    };
    uint64_t i = tid;
    for (; i + 3 * nt < vecs; i += 4 * nt) {
        uint4 q[4];
#pragma unroll
        for (int u = 0; u < 4; u++) q[u] = __ldg(v + i + u * nt);
#pragma unroll
        for (int u = 0; u < 4; u++) each(q[u]);
    }
    for (; i < vecs; i += nt) each(__ldg(v + i));
    const uint64_t tail = head + vecs * PER;
    if (tid < head) f(x[tid]);
    if (tid < n - tail) f(x[tail + tid]);
}

// Smallest lowest-set-bit exponent over the weights and their (rounded) sum.
template <typename WT>
__global__ void k_weight_range(const WT *__restrict__ w, uint64_t nnz, int *minlow, double *sum) {
    int lo = INT_MAX;
    float acc = 0.0f;  // an estimate for the range test (float64 is slow here)
    for_each_16b(w, nnz, [&](WT x) {
        lo = min(lo, low_bit_exp(x));
        acc += (float)x;
    });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lo = min(lo, __shfl_xor_sync(0xFFFFFFFFu, lo, o));
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(minlow, lo);
        atomicAdd(sum, (double)acc);
    }
}

// exact_lsb: the exponent lsb such that every weight is a multiple of 2^lsb
// and the total weight is below 2^52 * 2^lsb, so that every sum of weights is
// an integer number of units below 2^52, exact both as uint64 and as float64;
// INT_MIN when no such exponent in [-1000, 1000] exists (zero, negative or
// non-finite weights, or too wide a range of magnitudes).  The total is
// estimated with float32 partial sums (relative error far below the factor 2
// of margin kept under 2^53).
template <typename WT>
static WeightUnit exact_unit_t(const DevGraph &g, cudaStream_t s) {
    const WeightUnit none{INT_MIN, false};
    if (!g.nnz || !g.w) return none;
    size_t mk = arena().mark();
    int *dlo = arena().get<int>(1);
    double *dsum = arena().get<double>(1);
    const int init = INT_MAX;
    GSP_CUDA(cudaMemcpyAsync(dlo, &init, sizeof(int), cudaMemcpyHostToDevice, s));
    GSP_CUDA(cudaMemsetAsync(dsum, 0, sizeof(double), s));
    k_weight_range<WT><<<grid_for(g.nnz, 256 * 16 / sizeof(WT), sms(8)), 256, 0, s>>>(static_cast<const WT *>(g.w), g.nnz, dlo,
                                                                                   dsum);
    GSP_CHECK_LAUNCH();
    int lo = 0;
    double sum = 0.0;
    GSP_CUDA(cudaMemcpyAsync(&lo, dlo, sizeof(int), cudaMemcpyDeviceToHost, s));
    GSP_CUDA(cudaMemcpyAsync(&sum, dsum, sizeof(double), cudaMemcpyDeviceToHost, s));
    GSP_CUDA(cudaStreamSynchronize(s));
    arena().release(mk);
    if (lo < -1000 || lo > 1000) return none;
    // the sum is an estimate: keep a factor 2 of margin below 2^53 (and 2^32)
    if (!(sum > 0.0) || !(sum < std::ldexp(1.0, 52 + lo))) return none;
    return {lo, sum < std::ldexp(1.0, 31 + lo)};
}

WeightUnit exact_unit(const DevGraph &g, cudaStream_t s) {
    return g.wt == GSP_W_F64 ? exact_unit_t<double>(g, s) : exact_unit_t<float>(g, s);
}
int exact_lsb(const DevGraph &g, cudaStream_t s) { return exact_unit(g, s).lsb; }


__global__ void k_iota(uint32_t *p, uint32_t n) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) p[i] = i;
}
void iota_u32(uint32_t *p, uint32_t n, cudaStream_t s) {
    if (!n) return;
    k_iota<<<grid_for(n, 256), 256, 0, s>>>(p, n);
    GSP_CHECK_LAUNCH();
}

// Owner of every task of a chunked work split: one warp per item writes the
// item's index over its task range.
__global__ void k_task_items(const uint64_t *__restrict__ prefix, uint32_t nitems, uint32_t *out) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t base = prefix[0];
    for (uint32_t t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < nitems;
         t += (gridDim.x * blockDim.x) >> 5) {
        const uint64_t b = prefix[t] - base, e = prefix[t + 1] - base;
        for (uint64_t k = b + lane; k < e; k += 32) out[k] = t;
    }
}
void task_items(const uint64_t *prefix, uint32_t nitems, uint32_t *out, cudaStream_t s) {
    if (!nitems) return;
    k_task_items<<<grid_for((uint64_t)nitems * 32, 256), 256, 0, s>>>(prefix, nitems, out);
    GSP_CHECK_LAUNCH();
}

// Sigma of the communities that a block's rows belong to, summed in a shared
// table before the global adds: a few communities hold most rows, and one
// float64 atomic per row on their totals took 1.4 of the 1.55 ms of the row
// sums of a 2 M vertex graph (R-MAT, star partition).  Integer units only (the
// sums are exact, so their grouping does not show); float64 sums go out as they
// come, and so do those of graphs below SIGMA_MIN vertices, where too few rows
// queue on a community to pay for the table (gsp_modularity, one atomic a row
// against the table, us: planted 500 vertices 120 and 123, 8 K 125 and 128, 50 K
// 139 and 142; R-MAT 1 K 132 and 137, 8 K 149 and 151, 16 K 169 and 168, 50 K
// 251 and 206, 200 K 413 and 230; power laws of 60 to 80 K vertices whose
// communities are all cold 213 and 221).
constexpr uint32_t SIGMA_MIN = 16384;
struct SigmaSums {
    static constexpr int LOG = 10;
    static constexpr uint32_t SLOTS = 1u << LOG;
    uint32_t keys[SLOTS];
    unsigned long long sums[SLOTS];
    __device__ void clear() {
        for (uint32_t s = threadIdx.x; s < SLOTS; s += blockDim.x) { keys[s] = EMPTY; sums[s] = 0; }
        __syncthreads();
    }
    __device__ void add(double *Sig, uint32_t c, unsigned long long k, int lsb) {
        uint32_t h = hash32(c) >> (32 - LOG);
        for (int probe = 0; probe < 4; probe++) {
            uint32_t old = *(volatile uint32_t *)(keys + h);
            if (old == EMPTY) old = atomicCAS(keys + h, EMPTY, c);
            if (old == EMPTY || old == c) {
                atomicAdd(sums + h, k);
                return;
            }
            h = (h + 1) & (SLOTS - 1);
        }
        atomicAdd(Sig + c, Acc<unsigned long long>::val(k, lsb));  // crowded
    }
    __device__ void flush(double *Sig, int lsb) {
        __syncthreads();
        for (uint32_t s = threadIdx.x; s < SLOTS; s += blockDim.x)
            if (sums[s]) atomicAdd(Sig + keys[s], Acc<unsigned long long>::val(sums[s], lsb));
    }
};

// Per row i: K_i, and the intra-community part sum_{j: C_j = C_i} w_ij when C
// is given; Sigma_c += K_i when Sig is given (GROUPED: through a table, and Sig
// must be).  Long rows are deferred to a
// list for the block kernel.
template <typename WT, typename AV, bool GROUPED>
__global__ void k_row_sums(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tgt,
                           const WT *__restrict__ w, uint32_t n, const uint32_t *__restrict__ C, double *K,
                           double *Sig, AV *acc /* [0]=2m, [1]=intra */, uint32_t *longlist,
                           uint32_t *nlong, int lsb) {
    __shared__ AV red[32];
    __shared__ typename std::conditional<GROUPED, SigmaSums, char>::type sig;
    if constexpr (GROUPED) sig.clear();
    AV two_m = 0, intra = 0;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        uint64_t b = off[i], e = off[i + 1];
        if (e - b > SHORT_ROW) {
            longlist[atomicAdd(nlong, 1u)] = i;
            continue;
        }
        AV k = 0, in = 0;
        uint32_t ci = C ? C[i] : 0;
        uint64_t p = b;
        for (; p + 4 <= e; p += 4) {  // four independent loads in flight
            AV wv[4];
            uint32_t cj[4];
#pragma unroll
            for (int u = 0; u < 4; u++) wv[u] = Acc<AV>::of(w[p + u], lsb);
            if (C) {
#pragma unroll
                for (int u = 0; u < 4; u++) cj[u] = C[tgt[p + u]];
            }
#pragma unroll
            for (int u = 0; u < 4; u++) {
                k += wv[u];
                if (C && cj[u] == ci) in += wv[u];
            }
        }
        for (; p < e; p++) {
            const AV wv = Acc<AV>::of(w[p], lsb);
            k += wv;
            if (C && C[tgt[p]] == ci) in += wv;
        }
        if (K) K[i] = Acc<AV>::val(k, lsb);
        if constexpr (GROUPED) sig.add(Sig, ci, k, lsb);
        else if (Sig) atomicAdd(Sig + ci, Acc<AV>::val(k, lsb));
        two_m += k;
        intra += in;
    }
    if constexpr (GROUPED) sig.flush(Sig, lsb);
    two_m = block_sum(two_m, red);
    intra = block_sum(intra, red);
    if (threadIdx.x == 0) {
        atomicAdd(acc, two_m);
        if (C) atomicAdd(acc + 1, intra);
    }
}

// Long rows: one warp per row up to 8192 entries, one block per longer row.
constexpr uint32_t WARP_ROW = 8192;

template <typename WT, typename AV, bool GROUPED>
__global__ void k_row_sums_long(const uint64_t *__restrict__ off, const uint32_t *__restrict__ tgt,
                                const WT *__restrict__ w, const uint32_t *__restrict__ C, double *K, double *Sig,
                                AV *acc, const uint32_t *longlist, const uint32_t *nlong, int lsb) {
    __shared__ AV red[32];
    __shared__ typename std::conditional<GROUPED, SigmaSums, char>::type sig;
    uint32_t cnt = *nlong;
    if (!cnt) return;
    if constexpr (GROUPED) sig.clear();
    const int lane = threadIdx.x & 31;
    uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    AV wk = 0, win = 0;
    for (uint32_t t = warp; t < cnt; t += nwarps) {
        uint32_t i = longlist[t];
        uint64_t b = off[i], e = off[i + 1];
        if (e - b > WARP_ROW) continue;
        uint32_t ci = C ? C[i] : 0;
        AV k = 0, in = 0;
        uint64_t p = b + lane;
        for (; p + 96 < e; p += 128) {  // four independent loads per lane in flight
            AV wv[4];
            uint32_t cj[4];
#pragma unroll
            for (int u = 0; u < 4; u++) wv[u] = Acc<AV>::of(w[p + 32 * u], lsb);
            if (C) {
#pragma unroll
                for (int u = 0; u < 4; u++) cj[u] = C[tgt[p + 32 * u]];
            }
#pragma unroll
            for (int u = 0; u < 4; u++) {
                k += wv[u];
                if (C && cj[u] == ci) in += wv[u];
            }
        }
        for (; p < e; p += 32) {
            const AV wv = Acc<AV>::of(w[p], lsb);
            k += wv;
            if (C && C[tgt[p]] == ci) in += wv;
        }
        k = warp_sum(k);
        in = warp_sum(in);
        if (lane == 0) {
            if (K) K[i] = Acc<AV>::val(k, lsb);
            if constexpr (GROUPED) sig.add(Sig, ci, k, lsb);
            else if (Sig) atomicAdd(Sig + ci, Acc<AV>::val(k, lsb));
            wk += k;
            win += in;
        }
    }
    // rows longer than WARP_ROW: one block each
    for (uint32_t t = blockIdx.x; t < cnt; t += gridDim.x) {
        uint32_t i = longlist[t];
        uint64_t b = off[i], e = off[i + 1];
        if (e - b <= WARP_ROW) continue;
        uint32_t ci = C ? C[i] : 0;
        AV k = 0, in = 0;
        uint64_t p = b + threadIdx.x;
        const uint64_t st = blockDim.x;
        for (; p + 3 * st < e; p += 4 * st) {
            AV wv[4];
            uint32_t cj[4];
#pragma unroll
            for (int u = 0; u < 4; u++) wv[u] = Acc<AV>::of(w[p + st * u], lsb);
            if (C) {
#pragma unroll
                for (int u = 0; u < 4; u++) cj[u] = C[tgt[p + st * u]];
            }
#pragma unroll
            for (int u = 0; u < 4; u++) {
                k += wv[u];
                if (C && cj[u] == ci) in += wv[u];
            }
        }
        for (; p < e; p += st) {
            const AV wv = Acc<AV>::of(w[p], lsb);
            k += wv;
            if (C && C[tgt[p]] == ci) in += wv;
        }
        k = block_sum(k, red);
        in = block_sum(in, red);
        if (threadIdx.x == 0) {
            if (K) K[i] = Acc<AV>::val(k, lsb);
            if constexpr (GROUPED) sig.add(Sig, ci, k, lsb);
            else if (Sig) atomicAdd(Sig + ci, Acc<AV>::val(k, lsb));
            wk += k;
            win += in;
        }
    }
    if constexpr (GROUPED) sig.flush(Sig, lsb);
    wk = block_sum(wk, red);
    win = block_sum(win, red);
    if (threadIdx.x == 0) {
        if (wk != AV(0)) atomicAdd(acc, wk);
        if (C && win != AV(0)) atomicAdd(acc + 1, win);
    }
}

template <typename WT, typename AV, bool GROUPED = false>
static void row_sums(const DevGraph &g, const uint32_t *C, double *K, double *Sig, AV *acc, int lsb, cudaStream_t s) {
    if constexpr (std::is_same<AV, unsigned long long>::value && !GROUPED)
        if (Sig && g.n >= SIGMA_MIN) return row_sums<WT, AV, true>(g, C, K, Sig, acc, lsb, s);
    size_t mk = arena().mark();
    uint32_t *longlist = arena().get<uint32_t>(g.n + 1);
    uint32_t *nlong = arena().get<uint32_t>(1);
    GSP_CUDA(cudaMemsetAsync(nlong, 0, sizeof(uint32_t), s));
    const WT *w = static_cast<const WT *>(g.w);
    k_row_sums<WT, AV, GROUPED><<<grid_for(g.n, 256), 256, 0, s>>>(g.off, g.tgt, w, g.n, C, K, Sig, acc, longlist,
                                                                   nlong, lsb);
    GSP_CHECK_LAUNCH();
    // as many warps as fit: each long row is a chain of loads per lane
    const auto long_rows = k_row_sums_long<WT, AV, GROUPED>;
    long_rows<<<resident_grid((const void *)long_rows, 256, 0, 8), 256, 0, s>>>(g.off, g.tgt, w, C, K, Sig, acc,
                                                                                longlist, nlong, lsb);
    GSP_CHECK_LAUNCH();
    arena().release(mk);
}

// x[k] = u[k] units of 2^lsb as float64 (exact: u < 2^52).
__global__ void k_units_to_f64(const unsigned long long *u, int cnt, int lsb, double *x) {
    if ((int)threadIdx.x < cnt) x[threadIdx.x] = Acc<unsigned long long>::val(u[threadIdx.x], lsb);
}

// Row sums into float64 accumulators (acc: [0] = 2m, [1] = intra), or, when
// lsb != INT_MIN, in integer units accumulated in acc_u and converted here
// (exactly) into the same float64 values.
static void row_sums_any(const DevGraph &g, const uint32_t *C, double *K, double *Sig, double *acc,
                         unsigned long long *acc_u, int lsb, cudaStream_t s) {
    if (lsb != INT_MIN) {
        if (g.wt == GSP_W_F64) row_sums<double, unsigned long long>(g, C, K, Sig, acc_u, lsb, s);
        else row_sums<float, unsigned long long>(g, C, K, Sig, acc_u, lsb, s);
        k_units_to_f64<<<1, 32, 0, s>>>(acc_u, 2, lsb, acc);
        GSP_CHECK_LAUNCH();
        return;
    }
    if (g.wt == GSP_W_F64) row_sums<double, double>(g, C, K, Sig, acc, INT_MIN, s);
    else row_sums<float, double>(g, C, K, Sig, acc, INT_MIN, s);
}

__global__ void k_half(const double *acc, double *m_dev) {
    m_dev[0] = acc[0] / 2.0;
    m_dev[1] = 1.0 / m_dev[0];
}

double vertex_weights(const DevGraph &g, double *K, double *m_dev, cudaStream_t s, int lsb) {
    size_t mk = arena().mark();
    double *acc = arena().get<double>(2);
    unsigned long long *acc_u = arena().get<unsigned long long>(2);
    GSP_CUDA(cudaMemsetAsync(acc, 0, 2 * sizeof(double), s));
    GSP_CUDA(cudaMemsetAsync(acc_u, 0, 2 * sizeof(unsigned long long), s));
    row_sums_any(g, nullptr, K, nullptr, acc, acc_u, lsb, s);
    if (m_dev) {
        k_half<<<1, 1, 0, s>>>(acc, m_dev);
        GSP_CHECK_LAUNCH();
    }
    double h[2];
    GSP_CUDA(cudaMemcpyAsync(h, acc, sizeof(h), cudaMemcpyDeviceToHost, s));
    GSP_CUDA(cudaStreamSynchronize(s));
    arena().release(mk);
    return h[0] / 2.0;
}

__global__ void k_sum_sq(const double *Sig, uint32_t n, double *out) {
    __shared__ double red[32];
    double t = 0;
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        double x = Sig[c];
        t += x * x;
    }
    t = block_sum(t, red);
    if (threadIdx.x == 0) atomicAdd(out, t);
}

// Equation 1, second form: Q = sum_c sigma_c / 2m - sum_c (Sigma_c / 2m)^2,
// with sum_c sigma_c = the weight of all intra-community entries.
double modularity(const DevGraph &g, const uint32_t *C, cudaStream_t s, int lsb) {
    size_t mk = arena().mark();
    double *acc = arena().get<double>(4);
    unsigned long long *acc_u = arena().get<unsigned long long>(2);
    double *Sig = arena().get<double>(g.n);
    GSP_CUDA(cudaMemsetAsync(acc, 0, 4 * sizeof(double), s));
    GSP_CUDA(cudaMemsetAsync(acc_u, 0, 2 * sizeof(unsigned long long), s));
    GSP_CUDA(cudaMemsetAsync(Sig, 0, sizeof(double) * g.n, s));
    row_sums_any(g, C, nullptr, Sig, acc, acc_u, lsb, s);
    k_sum_sq<<<grid_for(g.n, 256), 256, 0, s>>>(Sig, g.n, acc + 2);
    GSP_CHECK_LAUNCH();
    double h[4];
    GSP_CUDA(cudaMemcpyAsync(h, acc, sizeof(h), cudaMemcpyDeviceToHost, s));
    GSP_CUDA(cudaStreamSynchronize(s));
    arena().release(mk);
    double two_m = h[0];
    if (!(two_m > 0.0)) return 0.0;
    return h[1] / two_m - h[2] / (two_m * two_m);
}

// Equation 1 with caller-provided scratch instead of the workspace: Sig (n
// doubles), acc (4 doubles), longlist (n entries) and nlong (1 entry).
// Allocates nothing.
template <typename WT>
static double modularity_scratch_t(const DevGraph &g, const uint32_t *C, double *Sig, double *acc, uint32_t *longlist,
                                   uint32_t *nlong, cudaStream_t s) {
    const WT *w = static_cast<const WT *>(g.w);
    GSP_CUDA(cudaMemsetAsync(acc, 0, 4 * sizeof(double), s));
    GSP_CUDA(cudaMemsetAsync(Sig, 0, sizeof(double) * g.n, s));
    GSP_CUDA(cudaMemsetAsync(nlong, 0, sizeof(uint32_t), s));
    k_row_sums<WT, double, false><<<grid_for(g.n, 256), 256, 0, s>>>(g.off, g.tgt, w, g.n, C, nullptr, Sig, acc, longlist,
                                                              nlong, INT_MIN);
    GSP_CHECK_LAUNCH();
    k_row_sums_long<WT, double, false><<<sms(4), 256, 0, s>>>(g.off, g.tgt, w, C, nullptr, Sig, acc, longlist, nlong,
                                                       INT_MIN);
    GSP_CHECK_LAUNCH();
    k_sum_sq<<<grid_for(g.n, 256), 256, 0, s>>>(Sig, g.n, acc + 2);
    GSP_CHECK_LAUNCH();
    double h[4];
    GSP_CUDA(cudaMemcpyAsync(h, acc, sizeof(h), cudaMemcpyDeviceToHost, s));
    GSP_CUDA(cudaStreamSynchronize(s));
    double two_m = h[0];
    if (!(two_m > 0.0)) return 0.0;
    return h[1] / two_m - h[2] / (two_m * two_m);
}

double modularity_scratch(const DevGraph &g, const uint32_t *C, double *Sig, double *acc, uint32_t *longlist,
                          uint32_t *nlong, cudaStream_t s) {
    if (g.wt == GSP_W_F64) return modularity_scratch_t<double>(g, C, Sig, acc, longlist, nlong, s);
    return modularity_scratch_t<float>(g, C, Sig, acc, longlist, nlong, s);
}

__global__ void k_count_ge(const uint32_t *__restrict__ x, uint64_t n, uint32_t bound, unsigned long long *out) {
    unsigned long long b = 0;
    for_each_16b(x, n, [&](uint32_t v) { b += v >= bound; });
    if (b) atomicAdd(out, b);
}

// Number of entries x[i] >= bound (i < n), counted in *counter
// (caller-provided, no allocation).
unsigned long long count_out_of_range(const uint32_t *x, uint64_t n, uint32_t bound, unsigned long long *counter,
                                      cudaStream_t s) {
    GSP_CUDA(cudaMemsetAsync(counter, 0, sizeof(*counter), s));
    if (n) {
        k_count_ge<<<grid_for(n, 256 * 4, sms(8)), 256, 0, s>>>(x, n, bound, counter);
        GSP_CHECK_LAUNCH();
    }
    unsigned long long h = 0;
    GSP_CUDA(cudaMemcpyAsync(&h, counter, sizeof(h), cudaMemcpyDeviceToHost, s));
    GSP_CUDA(cudaStreamSynchronize(s));
    return h;
}

__global__ void k_count_bad_offsets(const uint64_t *__restrict__ off, uint32_t n, uint64_t nnz,
                                    unsigned long long *out) {
    unsigned long long b = 0;
    const uint64_t tid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    for (uint64_t i = tid; i < n; i += (uint64_t)gridDim.x * blockDim.x)
        if (off[i + 1] < off[i]) b++;
    if (tid == 0 && (off[0] != 0 || off[n] != nnz)) b++;
    if (b) atomicAdd(out, b);
}

// CSR structure for the phase entry points: offsets rise from 0 to nnz and
// every target is < n; raises GSP_ERR_INVALID otherwise.  *counter is
// caller-provided scratch (no allocation).
void check_csr(const uint64_t *off, const uint32_t *tgt, uint32_t n, uint64_t nnz, unsigned long long *counter,
               cudaStream_t s) {
    GSP_CUDA(cudaMemsetAsync(counter, 0, sizeof(*counter), s));
    k_count_bad_offsets<<<grid_for(n, 256), 256, 0, s>>>(off, n, nnz, counter);
    GSP_CHECK_LAUNCH();
    unsigned long long h = 0;
    GSP_CUDA(cudaMemcpyAsync(&h, counter, sizeof(h), cudaMemcpyDeviceToHost, s));
    GSP_CUDA(cudaStreamSynchronize(s));
    GSP_REQUIRE(h == 0, "invalid graph: offsets must rise from 0 to nnz");
    h = count_out_of_range(tgt, nnz, n, counter, s);
    GSP_REQUIRE(h == 0, "invalid graph: %llu targets out of range (must be < %u)", h, n);
}

// ---------------------------------------------------------------- renumber
__global__ void k_mark_used(const uint32_t *__restrict__ C, uint32_t n, uint8_t *used) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) used[C[i]] = 1;
}
__global__ void k_apply_rank(const uint32_t *__restrict__ C, uint32_t n, const uint32_t *__restrict__ rank,
                             uint32_t *out) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[i] = rank[C[i]];
}

uint32_t renumber(uint32_t n, const uint32_t *C, uint32_t *C_dense, cudaStream_t s) {
    size_t mk = arena().mark();
    uint8_t *used = arena().get<uint8_t>(n);
    uint32_t *rank = arena().get<uint32_t>((size_t)n + 1);
    GSP_CUDA(cudaMemsetAsync(used, 0, n, s));
    k_mark_used<<<grid_for(n, 256), 256, 0, s>>>(C, n, used);
    GSP_CHECK_LAUNCH();
    exclusive_scan_u8_to_u32(used, rank, n, s);
    k_apply_rank<<<grid_for(n, 256), 256, 0, s>>>(C, n, rank, C_dense);
    GSP_CHECK_LAUNCH();
    uint32_t k;
    GSP_CUDA(cudaMemcpyAsync(&k, rank + n, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    GSP_CUDA(cudaStreamSynchronize(s));
    arena().release(mk);
    return k;
}

__global__ void k_lookup(uint32_t *Ctop, uint32_t n, const uint32_t *__restrict__ Cp) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) Ctop[i] = Cp[Ctop[i]];
}
void lookup(uint32_t n_top, uint32_t *C_top, const uint32_t *C_pass, cudaStream_t s) {
    if (!n_top) return;
    k_lookup<<<grid_for(n_top, 256), 256, 0, s>>>(C_top, n_top, C_pass);
    GSP_CHECK_LAUNCH();
}

// ------------------------------------------------------- final numbering
__global__ void k_first_vertex(const uint32_t *__restrict__ C, uint32_t n, uint32_t *first) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        atomicMin(first + C[i], i);
}
__global__ void k_is_first(const uint32_t *__restrict__ C, uint32_t n, const uint32_t *__restrict__ first,
                           uint8_t *flag) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        flag[i] = first[C[i]] == i;
}
__global__ void k_apply_first(uint32_t *C, uint32_t n, const uint32_t *__restrict__ first,
                              const uint32_t *__restrict__ rank) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        C[i] = rank[first[C[i]]];
}

uint32_t canonical_numbering(uint32_t n, uint32_t *C, cudaStream_t s) {
    size_t mk = arena().mark();
    uint32_t *first = arena().get<uint32_t>(n);
    uint8_t *flag = arena().get<uint8_t>(n);
    uint32_t *rank = arena().get<uint32_t>((size_t)n + 1);
    GSP_CUDA(cudaMemsetAsync(first, 0xFF, sizeof(uint32_t) * n, s));
    unsigned gr = grid_for(n, 256);
    k_first_vertex<<<gr, 256, 0, s>>>(C, n, first);
    GSP_CHECK_LAUNCH();
    k_is_first<<<gr, 256, 0, s>>>(C, n, first, flag);
    GSP_CHECK_LAUNCH();
    exclusive_scan_u8_to_u32(flag, rank, n, s);
    k_apply_first<<<gr, 256, 0, s>>>(C, n, first, rank);
    GSP_CHECK_LAUNCH();
    uint32_t k;
    GSP_CUDA(cudaMemcpyAsync(&k, rank + n, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    GSP_CUDA(cudaStreamSynchronize(s));
    arena().release(mk);
    return k;
}

// ------------------------------------------ Algorithm 6 (disconnected count)
// A community is disconnected exactly when its vertices fall in more than
// one connected component of the intra-community subgraph.
__global__ void k_count_roots(const uint32_t *__restrict__ C, const uint32_t *__restrict__ lab, uint32_t n,
                              uint32_t *ncomp) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        if (lab[i] == i) atomicAdd(ncomp + C[i], 1u);
}
__global__ void k_flag_disconnected(const uint32_t *__restrict__ ncomp, uint32_t n, uint8_t *flags,
                                    unsigned long long *count) {
    __shared__ unsigned long long red[32];
    unsigned long long t = 0;
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        uint8_t f = ncomp[c] > 1;
        if (flags) flags[c] = f;
        t += f;
    }
    t = block_sum(t, red);
    if (threadIdx.x == 0 && t) atomicAdd(count, t);
}

uint32_t count_disconnected(const DevGraph &g, const uint32_t *C, uint8_t *flags, cudaStream_t s) {
    size_t mk = arena().mark();
    uint32_t *lab = arena().get<uint32_t>(g.n);
    uint32_t *ncomp = arena().get<uint32_t>(g.n);
    unsigned long long *cnt = arena().get<unsigned long long>(1);
    split_labels(g, Classes(), C, GSP_SPLIT_SV, lab, s);  // every technique gives the same labels
    GSP_CUDA(cudaMemsetAsync(ncomp, 0, sizeof(uint32_t) * g.n, s));
    GSP_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), s));
    unsigned gr = grid_for(g.n, 256);
    k_count_roots<<<gr, 256, 0, s>>>(C, lab, g.n, ncomp);
    GSP_CHECK_LAUNCH();
    k_flag_disconnected<<<gr, 256, 0, s>>>(ncomp, g.n, flags, cnt);
    GSP_CHECK_LAUNCH();
    unsigned long long h;
    GSP_CUDA(cudaMemcpyAsync(&h, cnt, sizeof(h), cudaMemcpyDeviceToHost, s));
    GSP_CUDA(cudaStreamSynchronize(s));
    arena().release(mk);
    return (uint32_t)h;
}

}  // namespace gsp
