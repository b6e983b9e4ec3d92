// graph.cu -- device-side graph preprocessing: drop self loops, insert both
// directions, sort, deduplicate, optionally relabel by degree, and lay the
// result out as CSR with sorted neighbour lists (GraphPi Section IV-E).
//
// Each directed pair (u, v) travels as one key with u above v, so a single
// radix sort orders the pairs by source and then by target, which is exactly
// the CSR order. The sorts, the unique pass and the scan are CUB library calls.
#include <algorithm>

#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_scan.cuh>
#include <cub/device/device_select.cuh>

#include "engine.h"

namespace gp {

namespace {

constexpr int kThreads = 256;

inline int blocks_for(int64_t n) {
    int64_t b = (n + kThreads - 1) / kThreads;
    return (int)(b < 1 ? 1 : (b > (1 << 30) ? (1 << 30) : b));
}

int bits_for(uint64_t x) {     // bits needed to represent x
    int b = 0;
    while (b < 64 && (x >> b)) ++b;
    return b;
}

// What the host reads back of the pairs: kInfoBad is set by an id outside
// [0, n), kInfoLoop by a self loop, kInfoUnique receives the number of
// distinct keys.
enum { kInfoBad, kInfoLoop, kInfoUnique, kInfoPairs };

// Pair i yields keys 2i (u -> v) and 2i + 1 (v -> u), written as one 16-byte
// store; a key is (u << shift) | v, with `shift` the bits of the largest id,
// so that the sort sees no dead bits between the two. A self loop or an id out
// of range yields two copies of the sentinel n << shift, which sorts after
// every real key.
__global__ void k_make_keys(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                            int64_t m, int32_t n, int shift, ulonglong2* __restrict__ keys,
                            int64_t* __restrict__ info) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t u = src[i], v = dst[i];
        const bool ok = u >= 0 && u < n && v >= 0 && v < n;
        if (!ok) info[kInfoBad] = 1;
        else if (u == v) info[kInfoLoop] = 1;
        const uint64_t a = (uint32_t)u, b = (uint32_t)v, none = (uint64_t)(uint32_t)n << shift;
        keys[i] = (ok && u != v) ? make_ulonglong2((a << shift) | b, (b << shift) | a) : make_ulonglong2(none, none);
    }
}

// row_ptr[u] = first key whose source is >= u (binary search in sorted keys).
__global__ void k_row_ptr(const uint64_t* __restrict__ keys, int64_t nnz, int32_t n, int shift,
                          int64_t* __restrict__ row_ptr) {
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u <= n;
         u += (int64_t)gridDim.x * blockDim.x) {
        uint64_t target = (uint64_t)u << shift;
        int64_t lo = 0, hi = nnz;
        while (lo < hi) {
            int64_t mid = lo + ((hi - lo) >> 1);
            if (keys[mid] < target) lo = mid + 1; else hi = mid;
        }
        row_ptr[u] = lo;
    }
}

__global__ void k_col(const uint64_t* __restrict__ keys, int64_t nnz, int shift, int32_t* __restrict__ col) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nnz;
         i += (int64_t)gridDim.x * blockDim.x)
        col[i] = (int32_t)(keys[i] & (((uint64_t)1 << shift) - 1));
}

__global__ void k_max_deg(const int64_t* __restrict__ row_ptr, int32_t n, int* __restrict__ out) {
    int best = 0;
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n;
         u += (int64_t)gridDim.x * blockDim.x)
        best = max(best, (int)(row_ptr[u + 1] - row_ptr[u]));
    for (int o = 16; o; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, best);
}

// Degree and id of every vertex, to sort by degree (the sort is stable, so
// ties keep the id order).
__global__ void k_degrees(const int64_t* __restrict__ row_ptr, int32_t n, int32_t* __restrict__ deg,
                          int32_t* __restrict__ ids) {
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n;
         u += (int64_t)gridDim.x * blockDim.x) {
        deg[u] = (int32_t)(row_ptr[u + 1] - row_ptr[u]);
        ids[u] = (int32_t)u;
    }
}

// The inverse of new2old, and the new degrees in 64 bits with a zero behind
// them (their exclusive sum is the new row_ptr).
__global__ void k_inverse(const int32_t* __restrict__ new2old, const int32_t* __restrict__ sorted_deg, int32_t n,
                          int32_t* __restrict__ old2new, int64_t* __restrict__ deg64) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= n;
         i += (int64_t)gridDim.x * blockDim.x) {
        deg64[i] = i < n ? sorted_deg[i] : 0;
        if (i < n) old2new[new2old[i]] = (int32_t)i;
    }
}

// The entries (u, v) of the old graph in the order of the new id of u: entry
// e of old row u goes to its place in the new row of u, as the pair (target =
// new id of v, source = new id of u). The graph is symmetric, so these are
// also the entries of every new row `target`, and a stable sort by target
// alone leaves each row's sources ascending: half the key bits of sorting
// whole relabelled entries. The key itself names u and v (no row search:
// 0.53 -> 0.16 ms for 31 M entries).
__global__ void k_relabel(const uint64_t* __restrict__ keys, int64_t nnz, int shift,
                          const int64_t* __restrict__ old_row, const int64_t* __restrict__ new_row,
                          const int32_t* __restrict__ old2new, int32_t* __restrict__ target,
                          int32_t* __restrict__ source) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t key = keys[e];
        const int32_t u = (int32_t)(key >> shift), v = (int32_t)(key & (((uint64_t)1 << shift) - 1));
        const int32_t nu = old2new[u];
        const int64_t at = new_row[nu] + (e - old_row[u]);
        target[at] = old2new[v];
        source[at] = nu;
    }
}

__global__ void k_pairs_from_csr(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                                 int32_t n, int64_t nnz, int32_t* __restrict__ src,
                                 int32_t* __restrict__ dst) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = n;
        while (hi - lo > 1) {
            int64_t mid = (lo + hi) >> 1;
            if (row_ptr[mid] <= e) lo = mid; else hi = mid;
        }
        src[e] = (int32_t)lo;
        dst[e] = col[e];
    }
}

// Stream-ordered scratch that is released on every exit path.
struct Scratch {
    cudaStream_t st;
    void* p = nullptr;
    explicit Scratch(cudaStream_t s) : st(s) {}
    ~Scratch() { if (p) cudaFreeAsync(p, st); }
    cudaError_t alloc(size_t bytes) { return cudaMallocAsync(&p, bytes ? bytes : 16, st); }
    template <class T> T* as() const { return static_cast<T*>(p); }
};

// One block per core vertex u: set bit x of row u for every neighbour x of u
// below core_n (a prefix of u's sorted list; up to core_n entries, so a warp
// would walk it for 0.1 ms).
__global__ void k_core_bits(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                            int32_t core_n, int32_t words, uint32_t* __restrict__ bits) {
    for (int64_t u = blockIdx.x; u < core_n; u += gridDim.x) {
        const int64_t b = row_ptr[u], e = row_ptr[u + 1];
        for (int64_t i = b + threadIdx.x; i < e; i += blockDim.x) {
            const int32_t x = col[i];
            if (x >= core_n) break;
            atomicOr(bits + u * words + (x >> 5), 1u << (x & 31));
        }
    }
}

// What the host keeps about the finished graph.
struct GraphInfo {
    int64_t roots_ge[32];     // entries of the non-increasing `sorted` that are >= 2^i
    int64_t heavy_end;        // degree-ordered graphs: first entry of the first row shorter than kHeavyDegree
    int64_t n_hubs;           // degree-ordered graphs: rows longer than kHubDegree
    unsigned long long max_root_words;
    double dplus_pairs;       // sum of dplus (dplus - 1) / 2
    double sum_deg2;          // sum of squared degrees
    int32_t max_dplus;
    int32_t max_deg;
};

// dplus[u]: entries of row u below u (a prefix of the sorted row); the keys
// and ids to sort by it; the facts that are sums or maxima over all vertices.
__global__ void k_dplus(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int32_t n,
                        int32_t* __restrict__ dplus, int32_t* __restrict__ ids, GraphInfo* __restrict__ out) {
    __shared__ unsigned long long s_best[kThreads / 32];
    __shared__ double s_pairs[kThreads / 32], s_deg2[kThreads / 32];
    unsigned long long best = 0;
    double pairs = 0, deg2 = 0;
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n;
         u += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = row_ptr[u];
        int64_t lo = b, hi = row_ptr[u + 1];
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (col[mid] < u) lo = mid + 1; else hi = mid;
        }
        const int64_t below = lo - b, deg = row_ptr[u + 1] - b;
        dplus[u] = (int32_t)below;
        ids[u] = (int32_t)u;
        best = max(best, (unsigned long long)below * (4 * (unsigned long long)((deg + 127) >> 7)));
        pairs += 0.5 * (double)below * (double)(below - 1);
        deg2 += (double)deg * (double)deg;
    }
    for (int o = 16; o; o >>= 1) {
        best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
        pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
        deg2 += __shfl_xor_sync(0xffffffffu, deg2, o);
    }
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) { s_best[warp] = best; s_pairs[warp] = pairs; s_deg2[warp] = deg2; }
    __syncthreads();
    if (threadIdx.x) return;
    for (int w = 1; w < kThreads / 32; ++w) { best = max(best, s_best[w]); pairs += s_pairs[w]; deg2 += s_deg2[w]; }
    if (best) atomicMax(&out->max_root_words, best);
    if (pairs > 0) atomicAdd(&out->dplus_pairs, pairs);
    if (deg2 > 0) atomicAdd(&out->sum_deg2, deg2);
}

// One thread per fact; max_deg arrives from k_max_deg unless the rows are
// ordered by degree.
__global__ void k_graph_info(const int32_t* __restrict__ sorted, const int64_t* __restrict__ row_ptr, int32_t n,
                             bool ordered, GraphInfo* __restrict__ out) {
    const int i = threadIdx.x;
    if (i > 33) return;
    if (i == 32) {
        out->max_dplus = sorted[0];
        if (ordered) out->max_deg = (int32_t)(row_ptr[1] - row_ptr[0]);
    }
    int32_t lo = 0, hi = (i >= 32 && !ordered) ? 0 : n;
    while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1);
        const int64_t deg = i >= 32 ? row_ptr[mid + 1] - row_ptr[mid] : 0;
        const bool in = i == 32 ? deg >= kHeavyDegree : i == 33 ? deg > kHubDegree
                                : (int64_t)sorted[mid] >= ((int64_t)1 << i);
        if (in) lo = mid + 1; else hi = mid;
    }
    if (i == 32) out->heavy_end = ordered ? row_ptr[lo] : 0;
    else if (i == 33) out->n_hubs = lo;
    else out->roots_ge[i] = lo;
}

inline size_t padded(size_t bytes) { return (bytes + 255) & ~(size_t)255; }

}  // namespace

gp_status alloc_graph(gp_graph* g, int32_t n, int64_t nnz, bool ordered) {
    // one allocation for all arrays: each costs a synchronising driver call
    const int32_t core_n = ordered ? std::min(n, kCoreMax) : 0;
    const int32_t words = (((core_n + 31) / 32) + 3) & ~3;   // rows of whole 16-byte groups
    const size_t rows_b = padded(sizeof(int64_t) * ((size_t)n + 1)), col_b = padded(sizeof(int32_t) * (size_t)(nnz + 1));
    const size_t vert_b = padded(sizeof(int32_t) * (size_t)n), core_b = sizeof(uint32_t) * (size_t)core_n * (size_t)words;
    char* p = nullptr;
    const cudaError_t e = cudaMalloc((void**)&p, rows_b + col_b + (ordered ? 3 : 2) * vert_b + core_b);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("cudaMalloc of a graph with %lld entries failed: %s", (long long)nnz, cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? GP_ERR_NOMEM : GP_ERR_CUDA;
    }
    g->mem = p;
    g->n = n;
    g->nnz = nnz;
    g->row_ptr = reinterpret_cast<int64_t*>(p);
    g->col = reinterpret_cast<int32_t*>(p += rows_b);
    g->dplus = reinterpret_cast<int32_t*>(p += col_b);
    g->roots = reinterpret_cast<int32_t*>(p += vert_b);
    p += vert_b;
    if (ordered) {
        g->perm = reinterpret_cast<int32_t*>(p);
        g->core_bits = reinterpret_cast<uint32_t*>(p + vert_b);
        g->core_n = core_n;
        g->core_words = words;
    }
    return GP_OK;
}

gp_status finish_graph(gp_graph* g, cudaStream_t st) {
    const int32_t n = g->n;
    if (n == 0) return GP_OK;
    const bool ordered = g->perm != nullptr;
    Scratch ids(st), keys(st), temp(st), info(st);
    GP_CUDA_TRY(ids.alloc(sizeof(int32_t) * (size_t)n));
    GP_CUDA_TRY(keys.alloc(sizeof(int32_t) * (size_t)n));
    GP_CUDA_TRY(info.alloc(sizeof(GraphInfo)));
    GraphInfo* d_info = info.as<GraphInfo>();
    GP_CUDA_TRY(cudaMemsetAsync(d_info, 0, sizeof(GraphInfo), st));
    k_dplus<<<blocks_for(n), kThreads, 0, st>>>(g->row_ptr, g->col, n, g->dplus, ids.as<int32_t>(), d_info);
    size_t tb = 0;
    const int bits = std::max(1, bits_for((uint64_t)n - 1));
    GP_CUDA_TRY(cub::DeviceRadixSort::SortPairsDescending(nullptr, tb, g->dplus, keys.as<int32_t>(), ids.as<int32_t>(),
                                                          g->roots, n, 0, bits, st));
    GP_CUDA_TRY(temp.alloc(tb));
    GP_CUDA_TRY(cub::DeviceRadixSort::SortPairsDescending(temp.p, tb, g->dplus, keys.as<int32_t>(), ids.as<int32_t>(),
                                                          g->roots, n, 0, bits, st));
    if (!ordered) k_max_deg<<<std::min(blocks_for(n), 4096), kThreads, 0, st>>>(g->row_ptr, n, &d_info->max_deg);
    k_graph_info<<<1, 64, 0, st>>>(keys.as<int32_t>(), g->row_ptr, n, ordered, d_info);
    count_launch(ordered ? 3 : 4);
    if (g->core_n > 0) {
        GP_CUDA_TRY(cudaMemsetAsync(g->core_bits, 0, sizeof(uint32_t) * (size_t)g->core_n * (size_t)g->core_words, st));
        k_core_bits<<<g->core_n, kThreads, 0, st>>>(g->row_ptr, g->col, g->core_n, g->core_words, g->core_bits);
        count_launch();
    }
    GP_CUDA_TRY(cudaGetLastError());
    GraphInfo h;
    GP_CUDA_TRY(cudaMemcpyAsync(&h, d_info, sizeof(h), cudaMemcpyDeviceToHost, st));
    GP_CUDA_TRY(cudaStreamSynchronize(st));
    for (int i = 0; i < 32; ++i) g->roots_ge[i] = h.roots_ge[i];
    g->max_dplus = h.max_dplus;
    g->max_deg = h.max_deg;
    g->heavy_end = h.heavy_end;
    g->n_hubs = h.n_hubs;
    g->max_root_words = (int64_t)h.max_root_words;
    g->dplus_pairs = h.dplus_pairs;
    g->sum_deg2 = h.sum_deg2;
    return GP_OK;
}

gp_status csr_to_pairs(const int64_t* d_row_ptr, const int32_t* d_col, int32_t n, int64_t nnz,
                       int32_t* d_src, int32_t* d_dst, cudaStream_t st) {
    if (nnz == 0) return GP_OK;
    k_pairs_from_csr<<<blocks_for(nnz), kThreads, 0, st>>>(d_row_ptr, d_col, n, nnz, d_src, d_dst);
    count_launch();
    GP_CUDA_TRY(cudaGetLastError());
    return GP_OK;
}

gp_status build_graph(const int32_t* d_src, const int32_t* d_dst, int64_t m, int32_t n,
                      bool degree_order, cudaStream_t st, gp_graph* g) {
    const int64_t nkeys = 2 * m;
    const int id_bits = std::max(1, n > 0 ? bits_for((uint64_t)n - 1) : 0);
    const int end_bit = id_bits + bits_for((uint64_t)(uint32_t)n);
    Scratch keys_a(st), keys_b(st), info(st), temp(st);
    GP_CUDA_TRY(keys_a.alloc(sizeof(uint64_t) * (size_t)nkeys));
    GP_CUDA_TRY(keys_b.alloc(sizeof(uint64_t) * (size_t)nkeys));
    cub::DoubleBuffer<uint64_t> keys(keys_a.as<uint64_t>(), keys_b.as<uint64_t>());
    int64_t h[kInfoPairs] = {};
    if (m > 0) {
        // both directions as keys, sorted (CUB), each kept once
        GP_CUDA_TRY(info.alloc(sizeof(h)));
        GP_CUDA_TRY(cudaMemsetAsync(info.p, 0, sizeof(h), st));
        k_make_keys<<<blocks_for(m), kThreads, 0, st>>>(d_src, d_dst, m, n, id_bits,
                                                        reinterpret_cast<ulonglong2*>(keys.Current()), info.as<int64_t>());
        count_launch();
        GP_CUDA_TRY(cudaGetLastError());
        size_t tb = 0, tb2 = 0;
        GP_CUDA_TRY(cub::DeviceRadixSort::SortKeys(nullptr, tb, keys, nkeys, 0, end_bit, st));
        GP_CUDA_TRY(cub::DeviceSelect::Unique(nullptr, tb2, keys.Current(), keys.Alternate(),
                                              info.as<int64_t>() + kInfoUnique, nkeys, st));
        GP_CUDA_TRY(temp.alloc(std::max(tb, tb2)));
        GP_CUDA_TRY(cub::DeviceRadixSort::SortKeys(temp.p, tb, keys, nkeys, 0, end_bit, st));
        GP_CUDA_TRY(cub::DeviceSelect::Unique(temp.p, tb2, keys.Current(), keys.Alternate(),
                                              info.as<int64_t>() + kInfoUnique, nkeys, st));
        keys.selector ^= 1;
        count_launch(2);
        GP_CUDA_TRY(cudaMemcpyAsync(h, info.p, sizeof(h), cudaMemcpyDeviceToHost, st));
        GP_CUDA_TRY(cudaStreamSynchronize(st));
        if (h[kInfoBad]) { set_error("edge endpoint outside [0, %d)", n); return GP_ERR_ARG; }
    }
    const int64_t nnz = h[kInfoUnique] - (h[kInfoLoop] ? 1 : 0);    // without the sentinel
    const bool ordered = degree_order && n > 0;
    gp_status rc = alloc_graph(g, n, nnz, ordered);
    if (rc != GP_OK) return rc;
    if (!ordered) {
        k_row_ptr<<<blocks_for((int64_t)n + 1), kThreads, 0, st>>>(keys.Current(), nnz, n, id_bits, g->row_ptr);
        if (nnz) k_col<<<blocks_for(nnz), kThreads, 0, st>>>(keys.Current(), nnz, id_bits, g->col);
        count_launch(nnz ? 2 : 1);
        GP_CUDA_TRY(cudaGetLastError());
        if (n == 0) GP_CUDA_TRY(cudaStreamSynchronize(st));
        return finish_graph(g, st);
    }

    // relabel by non-increasing degree (ties by id)
    Scratch old_row(st), vert(st), deg64(st), temp2(st);
    GP_CUDA_TRY(old_row.alloc(sizeof(int64_t) * ((size_t)n + 1)));
    GP_CUDA_TRY(vert.alloc(4 * sizeof(int32_t) * (size_t)n));
    GP_CUDA_TRY(deg64.alloc(sizeof(int64_t) * ((size_t)n + 1)));
    int32_t* deg = vert.as<int32_t>();
    int32_t *sorted_deg = deg + n, *ids = deg + 2 * (size_t)n, *old2new = deg + 3 * (size_t)n;
    k_row_ptr<<<blocks_for((int64_t)n + 1), kThreads, 0, st>>>(keys.Current(), nnz, n, id_bits, old_row.as<int64_t>());
    k_degrees<<<blocks_for(n), kThreads, 0, st>>>(old_row.as<int64_t>(), n, deg, ids);
    count_launch(2);
    GP_CUDA_TRY(cudaGetLastError());
    // the pairs to sort: targets and sources in the free key buffer. The
    // sources of the last pass land in g->col whichever number of passes
    // the sort makes (it swaps its buffers once per 8 bits).
    const bool odd = ((id_bits + 7) / 8) & 1;
    int32_t* free_b = reinterpret_cast<int32_t*>(keys.Alternate());
    cub::DoubleBuffer<int32_t> target(free_b, reinterpret_cast<int32_t*>(keys.Current()));
    cub::DoubleBuffer<int32_t> source(odd ? free_b + nnz : g->col, odd ? g->col : free_b + nnz);
    size_t tb = 0, tb2 = 0, tb3 = 0;
    GP_CUDA_TRY(cub::DeviceRadixSort::SortPairsDescending(nullptr, tb, deg, sorted_deg, ids, g->perm, n, 0, id_bits, st));
    GP_CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb2, deg64.as<int64_t>(), g->row_ptr, (int64_t)n + 1, st));
    if (nnz > 0) GP_CUDA_TRY(cub::DeviceRadixSort::SortPairs(nullptr, tb3, target, source, nnz, 0, id_bits, st));
    GP_CUDA_TRY(temp2.alloc(std::max(std::max(tb, tb2), tb3)));
    GP_CUDA_TRY(cub::DeviceRadixSort::SortPairsDescending(temp2.p, tb, deg, sorted_deg, ids, g->perm, n, 0, id_bits, st));
    k_inverse<<<blocks_for((int64_t)n + 1), kThreads, 0, st>>>(g->perm, sorted_deg, n, old2new, deg64.as<int64_t>());
    GP_CUDA_TRY(cub::DeviceScan::ExclusiveSum(temp2.p, tb2, deg64.as<int64_t>(), g->row_ptr, (int64_t)n + 1, st));
    count_launch(3);
    if (nnz > 0) {
        k_relabel<<<blocks_for(nnz), kThreads, 0, st>>>(keys.Current(), nnz, id_bits, old_row.as<int64_t>(), g->row_ptr,
                                                        old2new, target.Current(), source.Current());
        GP_CUDA_TRY(cudaGetLastError());
        GP_CUDA_TRY(cub::DeviceRadixSort::SortPairs(temp2.p, tb3, target, source, nnz, 0, id_bits, st));
        count_launch(2);
        if (source.Current() != g->col)
            GP_CUDA_TRY(cudaMemcpyAsync(g->col, source.Current(), sizeof(int32_t) * (size_t)nnz, cudaMemcpyDeviceToDevice, st));
    }
    GP_CUDA_TRY(cudaGetLastError());
    return finish_graph(g, st);
}

}  // namespace gp
