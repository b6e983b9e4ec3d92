// wedge.cu -- the House's two-loop inclusion-exclusion count with its sums
// exchanged.
//
// The plan binds an edge (v0, v1) and a neighbour v2 of one end p; the inner
// sets are F = N(v_q) ∩ N(v2), q the other end, and O = N(v0) ∩ N(v1)
// (Section IV-D). Written out, with t = |O| and W(a, b) = |N(a) ∩ N(b)|, the
// sum over v2 of (|F| - 1)(t - [v2 in O]) - |F ∩ O| needs W(v_q, v2) for all
// wedges v_q - v_p - v2, which the general kernel intersects anew for every
// one of them. Here a block takes one vertex a, counts W(a, .) for all
// vertices at once by walking the lists of its neighbours into an array of
// counters, and reads off, for each neighbour b above a,
//   t = W(a, b),  P = sum of W(a, x) over the neighbours x of b.
// Over the whole graph the terms |F ∩ O| add up to the same sum of supports
// from both ends of every triangle's edges, so that
//   total = sum over edges of t (P - d(a) - d(b) + 3) - 2 t^2.
//
// The 4-cycle is counted from the same counters (k_cycle4): with v0 its
// largest vertex, the last level sums |N(v1) ∩ N(v2)| below v0 over the pairs of
// smaller neighbours of v0, which is the sum over w < v0 of C(y_w, 2), y_w the
// number of smaller neighbours of v0 adjacent to w.
//
// What bounds it: the counter updates, sum of squared degrees in all for the
// House (shared memory atomics where n counters fit, L2 atomics otherwise).
// Taking b above a reads the shorter lists of a degree-ordered graph.
#include <algorithm>

#include "acc.cuh"
#include "bits.cuh"
#include "engine.h"

namespace gp {

namespace {

// Lists longer than this are walked by the whole block, shorter ones by a
// warp each (in a degree-ordered graph the long ones come first in a row).
constexpr int kLongList = 1024;

struct WedgeArgs {
    DeviceGraph g;
    int32_t n;
    bool ordered;
    uint32_t* counters;        // n per block, zero (null: in shared memory)
    ResultWords* words;        // cursor: vertices
};

template <bool kShared>
__global__ void __launch_bounds__(1024)
k_wedge(const __grid_constant__ WedgeArgs a) {
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ unsigned long long s_item;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const long long t_start = clock64();
    uint32_t* const y = kShared ? smem : a.counters + (size_t)blockIdx.x * a.n;
    Acc acc;
    for (;;) {
        __syncthreads();                             // the last vertex's counters are done with
        if (threadIdx.x == 0) s_item = atomicAdd(&a.words->cursor[0], 1ull);
        if (kShared)
            for (int i = 4 * threadIdx.x; i < a.n; i += 4 * blockDim.x)
                *reinterpret_cast<uint4*>(y + i) = make_uint4(0, 0, 0, 0);
        __syncthreads();
        if (s_item >= (unsigned long long)a.n) break;
        const int v = (int)s_item;
        const int64_t rb = __ldg(a.g.row_ptr + v);
        const int d = (int)(__ldg(a.g.row_ptr + v + 1) - rb), above = __ldg(a.g.dplus + v);
        if (d < 2) continue;
        if (above == d) continue;                    // no neighbour above: nothing to read off
        // the lists of the neighbours, in two passes where counters are global
        // (count, then back to zero)
        auto walk = [&](auto touch) {
            int first = 0;
            for (; a.ordered && first < d; ++first) {
                const int u = __ldg(a.g.col + rb + first);
                const int64_t b = __ldg(a.g.row_ptr + u), e = __ldg(a.g.row_ptr + u + 1);
                if (e - b <= kLongList) break;
                for (int64_t i = b + threadIdx.x; i < e; i += blockDim.x) touch(__ldg(a.g.col + i));
            }
            // lane l holds the l-th of this warp's next 32 neighbours
            for (int base = first + warp; base < d; base += 32 * nwarps) {
                const int mine = base + lane * nwarps;
                int64_t b = 0;
                int len = 0;
                if (mine < d) {
                    const int u = __ldg(a.g.col + rb + mine);
                    b = __ldg(a.g.row_ptr + u);
                    len = (int)(__ldg(a.g.row_ptr + u + 1) - b);
                }
                const int count = min(32, (d - base + nwarps - 1) / nwarps);
                for (int q = 0; q < count; ++q) {
                    const int64_t qb = __shfl_sync(kAllLanes, b, q);
                    const int ql = __shfl_sync(kAllLanes, len, q);
                    for (int i = lane; i < ql; i += 32) touch(__ldg(a.g.col + qb + i));
                }
            }
        };
        walk([&](int w) { atomicAdd(y + w, 1u); });
        __syncthreads();
        // the neighbours above v, eight lanes each
        const int sub = threadIdx.x & 7, groups = blockDim.x >> 3;
        for (int base = above; base < d; base += groups) {
            const int i = base + (threadIdx.x >> 3);
            unsigned t = 0;
            unsigned long long P = 0;
            int db = 0;
            if (i < d) {
                const int b = __ldg(a.g.col + rb + i);
                t = kShared ? y[b] : __ldcg(y + b);
                if (t) {
                    const int64_t e0 = __ldg(a.g.row_ptr + b);
                    db = (int)(__ldg(a.g.row_ptr + b + 1) - e0);
                    for (int x = sub; x < db; x += 8) {
                        const int w = __ldg(a.g.col + e0 + x);
                        P += kShared ? y[w] : __ldcg(y + w);
                    }
                }
            }
            for (int o = 4; o; o >>= 1) P += __shfl_xor_sync(kAllLanes, P, o);
            if (sub == 0 && t) {
                const unsigned long long more = P + 3, less = (unsigned long long)d + (unsigned)db + 2ull * t;
                const unsigned __int128 plus = (unsigned __int128)t * more, minus = (unsigned __int128)t * less;
                const unsigned __int128 diff = plus - minus;
                acc.add128((unsigned long long)diff, (unsigned long long)(diff >> 64));
            }
        }
        if (!kShared) {
            __syncthreads();
            walk([&](int w) { __stcg(y + w, 0u); });
        }
    }
    flush(acc, a.words->total);
    if (lane == 0) atomicAdd(&a.words->busy, (unsigned long long)(clock64() - t_start));
}

constexpr size_t kSharedCounters = 224 * 1024;

size_t counter_bytes(const gp_graph* g) { return ((size_t)g->n * sizeof(uint32_t) + 15) & ~(size_t)15; }

// Lists longer than this are set aside by the warps and shared out in the
// block afterwards (k_cycle4): one warp takes 270 cycles for 32 elements, and
// under a hub the others wait for it (two hubs joined to 30 K vertices: 12.8 ->
// 1.3 ms, Chung-Lu of 1 M vertices 500 -> 171; 500 hubs of 3000 neighbours lose
// 6 % to the barrier).
constexpr int kSetAside = 512;
constexpr int kMostAside = 256;

// C(y, 2) is the sum of the counts found at each increment, so the walk of the
// smaller neighbours' lists, each up to v0, is all there is. kLong: the graph
// has lists to set aside (the extra barrier costs the others 3 %).
template <bool kShared, bool kLong>
__global__ void __launch_bounds__(1024)
k_cycle4(const __grid_constant__ WedgeArgs a) {
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ unsigned long long s_item;
    __shared__ int s_aside[kLong ? kMostAside : 1], s_n_aside;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const long long t_start = clock64();
    uint32_t* const y = kShared ? smem : a.counters + (size_t)blockIdx.x * a.n;
    Acc acc;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) { s_item = atomicAdd(&a.words->cursor[0], 1ull); s_n_aside = 0; }
        __syncthreads();
        if (s_item >= (unsigned long long)a.n) break;
        const int v = __ldg(a.g.roots + s_item);     // by the number of smaller neighbours, largest first
        const int d = __ldg(a.g.dplus + v);
        if (d < 2) break;                            // and so have all that follow
        const int64_t rb = __ldg(a.g.row_ptr + v);
        if (kShared) {
            for (int i = 4 * threadIdx.x; i < v; i += 4 * blockDim.x)
                *reinterpret_cast<uint4*>(y + i) = make_uint4(0, 0, 0, 0);
            __syncthreads();
        }
        // lane l holds the l-th of this warp's next 32 neighbours
        auto walk = [&](auto touch) {
            for (int base = warp; base < d; base += 32 * nwarps) {
                const int mine = base + lane * nwarps;
                int64_t b = 0;
                int len = 0;
                if (mine < d) {
                    const int u = __ldg(a.g.col + rb + mine);
                    b = __ldg(a.g.row_ptr + u);
                    len = (int)(__ldg(a.g.row_ptr + u + 1) - b);
                    if (kLong && len > kSetAside) {
                        const int at = atomicAdd(&s_n_aside, 1);
                        if (at < kMostAside) { s_aside[at] = u; len = 0; }
                    }
                }
                const int count = min(32, (d - base + nwarps - 1) / nwarps);
                for (int q = 0; q < count; ++q) {
                    const int64_t qb = __shfl_sync(kAllLanes, b, q);
                    const int ql = __shfl_sync(kAllLanes, len, q);
                    for (int i = lane; i < ql; i += 32) {
                        const int w = __ldg(a.g.col + qb + i);
                        if (w >= v) break;
                        touch(w);
                    }
                }
            }
            if constexpr (kLong) {
                __syncthreads();
                // a warp each where they are enough to go around, the block
                // one after the other where they are few
                const int n_aside = min(s_n_aside, kMostAside);
                const bool each = n_aside >= nwarps;
                const int step = each ? 32 : (int)blockDim.x;
                for (int q = each ? warp : 0; q < n_aside; q += each ? nwarps : 1) {
                    const int64_t b = __ldg(a.g.row_ptr + s_aside[q]), e = __ldg(a.g.row_ptr + s_aside[q] + 1);
                    for (int64_t i = b + (each ? lane : (int)threadIdx.x); i < e; i += step) {
                        const int w = __ldg(a.g.col + i);
                        if (w >= v) break;
                        touch(w);
                    }
                }
            }
        };
        unsigned long long sum = 0;
        walk([&](int w) { sum += atomicAdd(y + w, 1u); });
        acc.add(sum);
        if (!kShared) {
            __syncthreads();
            if (kLong) {
                if (threadIdx.x == 0) s_n_aside = 0;
                __syncthreads();
            }
            walk([&](int w) { __stcg(y + w, 0u); });
        }
    }
    flush(acc, a.words->total);
    if (lane == 0) atomicAdd(&a.words->busy, (unsigned long long)(clock64() - t_start));
}

// The 4-cycle under restrictions that keep exactly one of its eight maps onto
// every cycle, whatever the order of the ids. Their number over all 24 orders
// (what gp_schedule_explicit validates) does not say so: 0 > 1 > 2, 0 > 3 keeps
// two maps for some orders and none for others, and then the count is the
// plan's own.
bool is_cycle4(const GpPlan& P) {
    if (P.labeled || P.k != 4 || P.iep) return false;
    uint8_t adj[4] = {};                       // depths joined to depth d
    for (int d = 1; d < 4; ++d)
        for (int j = 0; j < d; ++j)
            if (P.lvl[d].op_mask >> j & 1) { adj[d] |= 1 << j; adj[j] |= 1 << d; }
    for (int d = 0; d < 4; ++d)
        if (__builtin_popcount(adj[d]) != 2) return false;
    // four ids form three cycles, each named by the id opposite id 3 and the
    // image of 8 of the 24 orders: how many of those are kept?
    int maps[3] = {0, 0, 0};
    int id[4] = {0, 1, 2, 3};
    const int across = __builtin_ctz(0xf & ~(adj[0] | 1));
    do {
        bool ok = true;
        for (int d = 1; d < 4; ++d)
            for (int j = 0; j < d; ++j) {
                if (P.lvl[d].lo_mask >> j & 1) ok &= id[d] > id[j];
                if (P.lvl[d].hi_mask >> j & 1) ok &= id[d] < id[j];
            }
        if (!ok) continue;
        int other = 0, at = 0;
        for (int d = 0; d < 4; ++d)
            if (id[d] == 3) at = d;
        if (at == 0 || at == across) other = id[at ^ across];
        else for (int d = 1; d < 4; ++d)
            if (d != at && d != across) other = id[d];
        ++maps[other];
    } while (std::next_permutation(id, id + 4));
    return maps[0] == 1 && maps[1] == 1 && maps[2] == 1;
}

// The House as an inclusion-exclusion plan: v2 joined to one end of the edge
// (v0, v1), one inner vertex to the other end and v2, the other to both ends;
// the only restriction left orders v0 and v1.
bool is_house_plan(const GpPlan& P) {
    if (P.labeled || P.k != 5 || P.iep != 2) return false;
    if (P.lvl[1].op_mask != 1 || (P.lvl[1].lo_mask | P.lvl[1].hi_mask) != 1) return false;
    for (int d = 2; d < 5; ++d)
        if (P.lvl[d].lo_mask || P.lvl[d].hi_mask) return false;
    const int far = P.lvl[2].op_mask == 1 ? 2 : P.lvl[2].op_mask == 2 ? 1 : 0;   // bit of the end not joined to v2
    const int f = far | 4, o = 3;
    return far && ((P.lvl[3].op_mask == f && P.lvl[4].op_mask == o) || (P.lvl[3].op_mask == o && P.lvl[4].op_mask == f));
}

}  // namespace

namespace {

// Blocks of a launch with counters in global memory: four of 512 threads an SM,
// halved until clearing the counters costs no more than a fraction of the walks
// that use them.
int64_t global_blocks(const gp_graph* g, int64_t nsm) {
    int64_t blocks = nsm * 4;
    const size_t most = std::max<size_t>((size_t)64 << 20, 64 * (size_t)g->nnz);
    while (blocks > 1 && counter_bytes(g) * (size_t)blocks > most) blocks = (blocks + 1) / 2;
    return blocks;
}

// Is the House worth counters in global memory in this many blocks? The general
// kernel takes about 0.15 ns per wedge (sum of squared degrees), a block 2 to 3
// us per vertex, more where all counters together exceed the L2. Measured on
// uniform graphs (general : counters, ms): 100 K vertices of mean degree 4
// 1.35 : 1.28, 8 1.72 : 1.46; 200 K of 8 2.4 : 5.5, 12 4.1 : 4.0; 1 M of 8
// 10.0 : 38, 12 18.8 : 25, 16 31.8 : 29.7, 20 50 : 22.
bool house_pays(const gp_graph* g, int64_t blocks) {
    const double line = g->n <= 128 * 1024 ? 2800.0 : counter_bytes(g) * (double)blocks <= 128e6 ? 22000.0 : 38000.0;
    return (double)blocks * g->sum_deg2 >= line * (double)g->n;
}

}  // namespace

bool wedge_applies(const CountJob& job, const gp_graph* g, const LaunchOpts& opt) {
    if (opt.stats || opt.no_core || opt.bitmap_mode != 2 || opt.budget_cycles > 0 || opt.task_cycles > 0) return false;
    // the exchanged sums hold for all tasks together
    if (!g->dplus || job.task_begin != 0 || job.ntasks != g->nnz) return false;
    const bool global = counter_bytes(g) > kSharedCounters;
    // On sparse graphs of many vertices the block's turn per vertex (clearing,
    // barriers) outweighs the lists: House at mean degree 2, 50 K vertices 0.73
    // against 0.52 ms; 4-cycles with counters in global memory at mean degree 8,
    // 100 K vertices 1.57 against 1.42 ms (at 20, 200 K: 2.9 against 5.6); at 16,
    // where the counters outgrow the L2 and the blocks are not all there, 1 M
    // vertices 25 against 13 ms (at 20: 17 against 20; Chung-Lu, 1 M: 170 against
    // 254)
    const bool cycle = is_cycle4(job.plan);
    if (!cycle && !is_house_plan(job.plan)) return false;
    if (!global) return cycle || g->n <= 16 * 1024 || g->nnz >= 4 * (int64_t)g->n - g->n / 4;
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return false;
    const int64_t blocks = global_blocks(g, nsm);
    if (!cycle) return house_pays(g, blocks);
    return g->nnz >= 14 * (int64_t)g->n &&
           (g->max_deg > kSetAside || blocks >= (int64_t)nsm * 2 || counter_bytes(g) * (double)blocks <= 128e6);
}

gp_status launch_wedge(const CountJob& job, const gp_graph* g, cudaStream_t st, ResultWords* words, int64_t* warps) {
    const bool cycle = is_cycle4(job.plan);
    int dev = 0, nsm = 0;
    GP_CUDA_TRY(cudaGetDevice(&dev));
    GP_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    WedgeArgs a = {};
    a.g = device_graph(g);
    a.n = g->n;
    a.ordered = g->perm != nullptr;
    // counters in shared memory up to 56 K vertices: several blocks an SM
    // while they fit, one of 1024 threads beyond
    const size_t bytes = counter_bytes(g);
    const bool shared = bytes <= kSharedCounters;
    const int threads = shared && bytes > 110 * 1024 ? 1024 : 512;
    const bool aside = g->max_deg > kSetAside;
    auto fn = cycle ? (shared ? (aside ? k_cycle4<true, true> : k_cycle4<true, false>)
                              : (aside ? k_cycle4<false, true> : k_cycle4<false, false>))
                    : (shared ? k_wedge<true> : k_wedge<false>);
    const size_t smem = shared ? bytes : 0;
    if (smem > kDefaultShared) {
        const gp_status rc = raise_shared_limit((const void*)fn, kSharedCounters);
        if (rc != GP_OK) return rc;
    }
    int64_t blocks = 0;
    size_t extra = 0;
    if (shared) {
        int occ = 0;
        GP_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem));
        blocks = std::max<int64_t>(1, std::min<int64_t>((int64_t)nsm * std::max(occ, 1), g->n));
    } else {
        size_t free_b = 0, total_b = 0;
        GP_CUDA_TRY(cudaMemGetInfo(&free_b, &total_b));
        blocks = global_blocks(g, nsm);
        const int64_t wanted = blocks;
        while (blocks > 1 && bytes * (size_t)blocks > free_b / 4) blocks = (blocks + 1) / 2;
        if (bytes * (size_t)blocks > free_b / 4 || (cycle ? 4 * blocks < wanted : !house_pays(g, blocks))) {
            set_error("counters of %zu bytes per block; %zu free", bytes, free_b);
            return GP_ERR_SCRATCH;
        }
        extra = sizeof(uint32_t) * (size_t)g->n * (size_t)blocks;
    }
    LaunchScratch mem(st);
    const gp_status rc = mem.alloc(extra);
    if (rc != GP_OK) return rc;
    if (extra) GP_CUDA_TRY(cudaMemsetAsync(mem.p, 0, extra, st));
    a.words = words;
    a.counters = reinterpret_cast<uint32_t*>(mem.p);
    fn<<<(unsigned)blocks, threads, smem, st>>>(a);
    count_launch();
    GP_CUDA_TRY(cudaGetLastError());
    *warps = blocks * (threads / 32);
    return GP_OK;
}

}  // namespace gp
