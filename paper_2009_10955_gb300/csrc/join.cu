// join.cu -- inclusion-exclusion counts of a clique joined to independent
// vertices: m = 2..4 mutually adjacent outer vertices, restricted to one
// order, and kk inner vertices each adjacent to all of them (the diamond, the
// 5- and the 6-clique minus an edge, ...).
//
// Every inner set is then the common neighbourhood S of the clique, and the
// inclusion-exclusion sum over kk equal sets is the falling factorial
// |S| (|S| - 1) ... (|S| - kk + 1) (Section IV-D). For a root v0 (the clique's
// largest id) the kernel builds the bit matrix F of the graph with a row for
// each neighbour below v0 and a column for every neighbour of v0; the columns
// are sorted by id, so the rows are the first columns. |S| of {v0, x} is the
// population count of x's row, of {v0, x, y} that of two rows' AND; for
// m = 4 the matrix is compacted to the neighbours of x first, so that the
// AND of the rows of y and z there runs on words that hold little else.
//
// What bounds it: building F (one bit probe of the core matrix, or a binary
// search, per row and column: sum over edges of the smaller degree), then the
// AND/popcount passes. The general kernel intersects lists for every clique
// instead, a warp each.
#include <algorithm>

#include "acc.cuh"
#include "bits.cuh"
#include "engine.h"

namespace gp {

namespace {

// A warp takes a root of fewer than kWarpRows smaller neighbours and at most
// kWarpCols neighbours: its matrix is at most 512 words.
constexpr int kWarpRows = 32;
constexpr int kWarpCols = 512;
constexpr int kOwnWords = 1024;     // a warp's matrices (two of 512 words, or one compacted one)
constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kListWords = kWarpCols / 2;   // a warp's member list (16-bit positions)
constexpr int kListPositions = 1 << 16;     // columns such a position can name
// Root matrices up to this many words stay in shared memory: with the warps'
// areas 108 KB a block, two blocks an SM.
constexpr int kBlockWords = 7168;

struct JoinArgs {
    DeviceGraph g;
    int64_t task_begin, task_end;
    int kk;
    int64_t n_hubs;           // vertices 0 .. n_hubs - 1 have more than kWarpCols neighbours
    int64_t n_block;          // leading roots with at least kWarpRows smaller neighbours
    int64_t n_roots;          // roots worth visiting
    int warp_chunk;
    uint32_t* big;            // per block: F, the compacted matrix, a member list (global)
    int64_t big_words, list_words;
    ResultWords* words;       // cursors: block items, warp roots
};

__device__ __forceinline__ int stride_of(int cols) { return cols <= 32 ? 1 : 4 * ((cols + 127) >> 7); }

// c (c - 1) ... (c - kk + 1)
__device__ __forceinline__ void add_falling(Acc& acc, unsigned c, int kk) {
    if (c < (unsigned)kk) return;
    if (kk == 2) { acc.add((unsigned long long)c * (c - 1)); return; }
    unsigned __int128 p = c;
    for (int t = 1; t < kk; ++t) p *= c - t;
    acc.add128((unsigned long long)p, (unsigned long long)(p >> 64));
}

// Which of four vertices x (uniform, ascending) are neighbours of the lane's
// y? Core pairs by one bit, the others by four searches side by side.
struct Four {
    int x[4];
    const int32_t* p[4];
    int n[4];
};

__device__ __forceinline__ Four four_rows(const DeviceGraph& g, const int32_t* U, int i0, int rows) {
    Four f;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        f.x[t] = __ldg(U + min(i0 + t, rows - 1));
        const int64_t b = __ldg(g.row_ptr + f.x[t]);
        f.p[t] = g.col + b;
        f.n[t] = (int)(__ldg(g.row_ptr + f.x[t] + 1) - b);
    }
    return f;
}

__device__ __forceinline__ unsigned probe_four(const DeviceGraph& g, const Four& f, int y, bool valid) {
    unsigned hits = 0;
    int b[4], n[4];
    bool search = false;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        b[t] = 0;
        n[t] = 0;
        if (!valid) continue;
        if (f.x[t] < g.core_n && y < g.core_n) {
            hits |= ((__ldg(g.core_bits + (size_t)f.x[t] * g.core_words + (y >> 5)) >> (y & 31)) & 1u) << t;
        } else {
            n[t] = f.n[t];
            search = true;
        }
    }
    if (search) {
        bool want[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) want[t] = n[t] > 0;
        while (n[0] | n[1] | n[2] | n[3]) {
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (n[t] > 0) {
                    const int half = n[t] >> 1;
                    if (__ldg(f.p[t] + b[t] + half) < y) { b[t] += half + 1; n[t] -= half + 1; } else n[t] = half;
                }
        }
#pragma unroll
        for (int t = 0; t < 4; ++t)
            if (want[t] && b[t] < f.n[t] && __ldg(f.p[t] + b[t]) == y) hits |= 1u << t;
    }
    return hits;
}

// Rows i0 .. i0 + 3 (below `rows`) of F, column words [w0, w1), one warp.
__device__ __forceinline__ void build_words(const DeviceGraph& g, const int32_t* U, int cols, int i0, int rows,
                                            int w0, int w1, uint32_t* F, int stride, int lane) {
    const Four f = four_rows(g, U, i0, rows);
    for (int w = w0; w < w1; ++w) {
        const int j = 32 * w + lane;
        const bool valid = j < cols;
        const unsigned hits = probe_four(g, f, valid ? __ldg(U + j) : 0, valid);
        uint32_t mine = 0;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const uint32_t b = __ballot_sync(kAllLanes, hits >> t & 1u);
            if (lane == t) mine = b;
        }
        if (lane < 4 && i0 + lane < rows) F[(size_t)(i0 + lane) * stride + w] = mine;
    }
}

// m = 2: the rows' sizes alone, rows [lo, hi) in fours from `first`.
__device__ __forceinline__ void count_rows(const DeviceGraph& g, const int32_t* U, int cols, int lo, int hi,
                                           int first, int step, int kk, int lane, Acc& acc) {
    for (int i0 = lo + 4 * first; i0 < hi; i0 += 4 * step) {
        const Four f = four_rows(g, U, i0, hi);
        unsigned c[4] = {0, 0, 0, 0};
        for (int j0 = 0; j0 < cols; j0 += 32) {
            const int j = j0 + lane;
            const bool valid = j < cols;
            const unsigned hits = probe_four(g, f, valid ? __ldg(U + j) : 0, valid);
#pragma unroll
            for (int t = 0; t < 4; ++t) c[t] += __popc(__ballot_sync(kAllLanes, hits >> t & 1u));
        }
#pragma unroll
        for (int t = 0; t < 4; ++t)
            if (lane == t && i0 + t < hi) add_falling(acc, c[t], kk);
    }
}

// Pairs k < j of adjacent rows of M (row j's bit k), j in [lo, hi): the
// falling factorial of the two rows' common bits. Lane k holds row k, four
// rows j are read at a time; units (word of rows k, four rows j) from `first`.
__device__ __forceinline__ void count_pairs(const uint32_t* M, int stride, int cols, int lo, int hi, int first,
                                            int step, int kk, int lane, Acc& acc) {
    const int nk = (hi + 31) >> 5, j00 = lo & ~3, quads = (hi - j00 + 3) >> 2;
    for (int u = first; u < nk * quads; u += step) {
        const int kb = u % nk, j0 = j00 + 4 * (u / nk);
        if (min(j0 + 3, hi - 1) <= 32 * kb) continue;
        const int k = 32 * kb + lane;
        const uint32_t* own = M + (size_t)min(k, hi - 1) * stride;
        unsigned c[4] = {0, 0, 0, 0};
        if (stride == 1) {
            const uint32_t a = own[0];
#pragma unroll
            for (int t = 0; t < 4; ++t) c[t] = __popc(a & M[min(j0 + t, hi - 1)]);
        } else {
            for (int q = 0; 128 * q < cols; ++q) {
                const uint4 a = *reinterpret_cast<const uint4*>(own + 4 * q);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const uint4 r = *reinterpret_cast<const uint4*>(M + (size_t)min(j0 + t, hi - 1) * stride + 4 * q);
                    c[t] += __popc(a.x & r.x) + __popc(a.y & r.y) + __popc(a.z & r.z) + __popc(a.w & r.w);
                }
            }
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int j = j0 + t;
            if (j >= lo && j < hi && k < j && (M[(size_t)j * stride + kb] >> lane & 1u)) add_falling(acc, c[t], kk);
        }
    }
}

// Number of set bits of the row, and of those below bit i.
__device__ __forceinline__ int2 row_sizes(const uint32_t* row, int nw, int i, int lane) {
    int all = 0, below = 0;
    for (int w = lane; w < nw; w += 32) {
        const uint32_t x = row[w];
        all += __popc(x);
        below += w < (i >> 5) ? __popc(x) : w == (i >> 5) ? __popc(x & ((1u << (i & 31)) - 1u)) : 0;
    }
    return make_int2(__reduce_add_sync(kAllLanes, all), __reduce_add_sync(kAllLanes, below));
}

// Positions of the set bits of words [w0, w1) of a row, from list[n] on.
template <class T>
__device__ __forceinline__ void expand(const uint32_t* row, int w0, int w1, int n, T* list, int lane) {
    for (int w = w0; w < w1; ++w) {
        const uint32_t x = row[w];
        if (x >> lane & 1u) list[n + __popc(x & lanes_below())] = (T)(32 * w + lane);
        n += __popc(x);
    }
}

// The matrix of the first `rows` members against all `cols` members of a
// list of positions in F: word by word of columns, rows in fours from
// `first`. A ballot gives one row's word.
template <class T>
__device__ __forceinline__ void compact(const uint32_t* F, int stride, const T* list, int rows, int cols,
                                        uint32_t* out, int out_stride, int lane, int first, int step) {
    for (int g = 0; 32 * g < cols; ++g) {
        const int c = 32 * g + lane;
        const int p = (c < cols) ? (int)list[c] : 0;
        const uint32_t* base = F + (p >> 5);
        const uint32_t bit = (c < cols) ? (1u << (p & 31)) : 0u;
        for (int m = 4 * first; m < rows; m += 4 * step) {
            uint32_t b[4];
#pragma unroll
            for (int t = 0; t < 4; ++t)
                b[t] = __ballot_sync(kAllLanes, base[(size_t)list[min(m + t, rows - 1)] * stride] & bit);
            if (lane == 0) {
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (m + t < rows) out[(size_t)(m + t) * out_stride + g] = b[t];
            }
        }
    }
    const int nw = (cols + 31) >> 5;               // whole 16-byte groups are read: at most three words more
    if (lane < out_stride - nw)
        for (int m = 4 * first; m < rows; m += 4 * step)
            for (int t = 0; t < 4 && m + t < rows; ++t) out[(size_t)(m + t) * out_stride + nw + lane] = 0u;
}

constexpr int kMostLarge = 1024;    // large rows a block notes; with more it looks through all rows again

struct BlockState {
    int next, n_large;
    int sums[kWarps];
    int large[kMostLarge];
};

// m = 4, one row i of F whose compacted matrix a warp cannot hold: the block
// compacts it into C and counts its pairs.
__device__ __forceinline__ void block_row(const uint32_t* F, int stride, int W, int i, int2 size, uint32_t* C,
                                          uint32_t* list, int kk, BlockState* bs, Acc& acc) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t* row = F + (size_t)i * stride;
    const int per = (W + kWarps - 1) / kWarps, w0 = min(W, warp * per), w1 = min(W, w0 + per);
    int n = 0;
    for (int w = w0 + lane; w < w1; w += 32) n += __popc(row[w]);
    n = __reduce_add_sync(kAllLanes, n);
    __syncthreads();                               // C, list and sums are free
    if (lane == 0) bs->sums[warp] = n;
    __syncthreads();
    int at = 0;
    for (int q = 0; q < warp; ++q) at += bs->sums[q];
    expand(row, w0, w1, at, list, lane);
    __syncthreads();
    const int cs = stride_of(size.x);
    compact(F, stride, list, size.y, size.x, C, cs, lane, warp, kWarps);
    __syncthreads();
    count_pairs(C, cs, size.x, 0, size.y, warp, kWarps, kk, lane, acc);
}

template <int M>
__global__ void __launch_bounds__(kThreads, 2)
k_join(const __grid_constant__ JoinArgs a) {
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ BlockState bs;
    __shared__ unsigned long long s_item;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long t_start = clock64();
    uint16_t* const list = reinterpret_cast<uint16_t*>(smem + warp * (kListWords + kOwnWords));
    uint32_t* const own = smem + warp * (kListWords + kOwnWords) + kListWords;
    uint32_t* const shared_F = smem + kWarps * (kListWords + kOwnWords);
    uint32_t* const big_F = a.big + (size_t)blockIdx.x * (2 * a.big_words + a.list_words);
    Acc acc;
    // hubs and roots with many smaller neighbours: a block each
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) { s_item = atomicAdd(&a.words->cursor[0], 1ull); bs.next = 0; bs.n_large = 0; }
        __syncthreads();
        const unsigned long long item = s_item;
        if (item >= (unsigned long long)(a.n_hubs + a.n_block)) break;
        const bool hub = item < (unsigned long long)a.n_hubs;
        const int v0 = hub ? (int)item : __ldg(a.g.roots + (item - a.n_hubs));
        if (!hub && v0 < a.n_hubs) continue;           // taken as a hub
        const int64_t rb = __ldg(a.g.row_ptr + v0);
        const int cols = (int)(__ldg(a.g.row_ptr + v0 + 1) - rb), n = __ldg(a.g.dplus + v0);
        const int lo = (int)max((int64_t)0, min((int64_t)n, a.task_begin - rb));
        const int hi = (int)max((int64_t)0, min((int64_t)n, a.task_end - rb));
        if (lo >= hi || hi < M - 1) continue;
        const int32_t* U = a.g.col + rb;
        if constexpr (M == 2) {
            count_rows(a.g, U, cols, lo, hi, warp, kWarps, a.kk, lane, acc);
        } else {
            const int stride = stride_of(cols), W = (cols + 31) >> 5;
            uint32_t* F = (size_t)hi * stride <= kBlockWords ? shared_F : big_F;
            // units of four rows and 32 column words, padded to the stride
            const int quads = (hi + 3) >> 2, chunks = (stride + 31) >> 5;
            for (int u = warp; u < quads * chunks; u += kWarps) {
                const int q = u / chunks, w0 = 32 * (u % chunks);
                build_words(a.g, U, cols, 4 * q, hi, w0, min(stride, w0 + 32), F, stride, lane);
            }
            __syncthreads();
            if constexpr (M == 3) {
                count_pairs(F, stride, cols, lo, hi, warp, kWarps, a.kk, lane, acc);
            } else {
                // rows whose compacted matrix fits a warp's area (and whose
                // members a warp's list can name)
                const auto warp_holds = [cols](int2 size) {
                    return cols <= kListPositions && size.x <= kWarpCols && size.y * stride_of(size.x) <= kOwnWords;
                };
                for (;;) {
                    int q = 0;
                    if (lane == 0) q = atomicAdd(&bs.next, 1);
                    q = __shfl_sync(kAllLanes, q, 0);
                    const int i = hi - 1 - q;
                    if (i < lo) break;
                    const uint32_t* row = F + (size_t)i * stride;
                    const int2 size = row_sizes(row, W, i, lane);
                    const int cs = stride_of(size.x);
                    if (size.y < 2) continue;
                    if (!warp_holds(size)) {
                        if (lane == 0) {
                            const int at = atomicAdd(&bs.n_large, 1);
                            if (at < kMostLarge) bs.large[at] = i;
                        }
                        continue;
                    }
                    expand(row, 0, W, 0, list, lane);
                    __syncwarp();
                    compact(F, stride, list, size.y, size.x, own, cs, lane, 0, 1);
                    __syncwarp();
                    count_pairs(own, cs, size.x, 0, size.y, 0, 1, a.kk, lane, acc);
                    __syncwarp();
                }
                __syncthreads();
                // the others, by the block
                const int n_large = bs.n_large;
                const bool noted = n_large <= kMostLarge;
                for (int q = 0; q < (noted ? n_large : hi - lo); ++q) {
                    const int i = noted ? bs.large[q] : lo + q;
                    const int2 size = row_sizes(F + (size_t)i * stride, W, i, lane);
                    if (size.y < 2 || warp_holds(size)) continue;
                    block_row(F, stride, W, i, size, big_F + a.big_words, big_F + 2 * a.big_words, a.kk, &bs, acc);
                }
            }
        }
    }
    __syncthreads();
    // the others: a warp each
    const unsigned long long n_warp = (unsigned long long)(a.n_roots - a.n_block);
    for (;;) {
        unsigned long long t0 = 0;
        if (lane == 0) t0 = atomicAdd(&a.words->cursor[1], (unsigned long long)a.warp_chunk);
        t0 = __shfl_sync(kAllLanes, t0, 0);
        if (t0 >= n_warp) break;
        const bool have = lane < a.warp_chunk && t0 + lane < n_warp;
        const int lv = have ? __ldg(a.g.roots + a.n_block + t0 + lane) : 0;
        const int64_t lrb = have ? __ldg(a.g.row_ptr + lv) : 0;
        const int lcols = have ? (int)(__ldg(a.g.row_ptr + lv + 1) - lrb) : 0;
        const int ln = have && lv >= a.n_hubs ? __ldg(a.g.dplus + lv) : 0;
        for (int q = 0; q < a.warp_chunk; ++q) {
            const int64_t rb = __shfl_sync(kAllLanes, lrb, q);
            const int cols = __shfl_sync(kAllLanes, lcols, q), n = __shfl_sync(kAllLanes, ln, q);
            const int lo = (int)max((int64_t)0, min((int64_t)n, a.task_begin - rb));
            const int hi = (int)max((int64_t)0, min((int64_t)n, a.task_end - rb));
            if (lo >= hi || hi < M - 1) continue;
            const int32_t* U = a.g.col + rb;
            if constexpr (M == 2) {
                count_rows(a.g, U, cols, lo, hi, 0, 1, a.kk, lane, acc);
            } else {
                const int stride = stride_of(cols), W = (cols + 31) >> 5;
                for (int i = 0; i < hi; i += 4) build_words(a.g, U, cols, i, hi, 0, stride, own, stride, lane);
                __syncwarp();
                if constexpr (M == 3) {
                    count_pairs(own, stride, cols, lo, hi, 0, 1, a.kk, lane, acc);
                } else {
                    uint32_t* next = own + kOwnWords / 2;
                    for (int i = max(lo, 2); i < hi; ++i) {
                        const uint32_t* row = own + i * stride;
                        const int2 size = row_sizes(row, W, i, lane);
                        if (size.y < 2) continue;
                        const int cs = stride_of(size.x);
                        expand(row, 0, W, 0, list, lane);
                        __syncwarp();
                        compact(own, stride, list, size.y, size.x, next, cs, lane, 0, 1);
                        __syncwarp();
                        count_pairs(next, cs, size.x, 0, size.y, 0, 1, a.kk, lane, acc);
                        __syncwarp();
                    }
                }
                __syncwarp();
            }
        }
    }
    flush(acc, a.words->total);
    if (lane == 0) atomicAdd(&a.words->busy, (unsigned long long)(clock64() - t_start));
}

// m of the plan, or 0: its outer vertices are mutually adjacent and totally
// ordered by the restrictions (*descending: the earlier the larger), its
// inner ones unrestricted and adjacent to all outer ones.
int join_outer(const GpPlan& P, bool* descending) {
    const int m = P.k - P.iep;
    if (P.labeled || P.iep < 2 || m < 2 || m > 4) return 0;
    *descending = true;
    for (int d = 1; d < P.k; ++d) {
        const GpLevel& L = P.lvl[d];
        const uint8_t all = (uint8_t)((1u << std::min(d, m)) - 1u);
        if (L.op_mask != all) return 0;
        if (d < m) {
            if ((uint8_t)(L.lo_mask | L.hi_mask) != all) return 0;
            if (L.hi_mask != all) *descending = false;
        } else if (L.lo_mask || L.hi_mask) {
            return 0;
        }
    }
    return m;
}

}  // namespace

bool join_applies(const CountJob& job, const gp_graph* g, const LaunchOpts& opt) {
    bool descending = false;
    if (opt.stats || opt.no_core || opt.bitmap_mode != 2 || opt.budget_cycles > 0 || opt.task_cycles > 0) return false;
    if (!g->perm || !g->roots || join_outer(job.plan, &descending) == 0) return false;
    if (g->max_root_words > kMostRootWords) return false;
    return descending || (job.task_begin == 0 && job.ntasks == g->nnz);
}

gp_status launch_join(const CountJob& job, const gp_graph* g, cudaStream_t st, ResultWords* words, int64_t* warps) {
    bool descending = false;
    const int m = join_outer(job.plan, &descending);
    int dev = 0, nsm = 0;
    GP_CUDA_TRY(cudaGetDevice(&dev));
    GP_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    JoinArgs a = {};
    a.g = device_graph(g);
    a.task_begin = job.task_begin;
    a.task_end = job.task_begin + job.ntasks;
    a.kk = job.plan.iep;
    a.n_hubs = g->n_hubs;
    static_assert(kWarpRows == 1 << 5 && kWarpCols == kHubDegree, "classes kept with the graph");
    a.n_block = g->roots_ge[5];
    a.n_roots = g->roots_ge[m <= 3 ? m - 2 : 1];   // at least m - 1 smaller neighbours
    a.n_roots = std::max(a.n_roots, a.n_block);
    auto fn = m == 2 ? k_join<2> : m == 3 ? k_join<3> : k_join<4>;
    const size_t smem = m == 2 ? 0 : sizeof(uint32_t) * (size_t)(kWarps * (kListWords + kOwnWords) + kBlockWords);
    if (smem) {
        const gp_status rc = raise_shared_limit((const void*)fn, smem);
        if (rc != GP_OK) return rc;
    }
    int occ = 0;
    GP_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kThreads, smem));
    int64_t blocks = (int64_t)nsm * std::max(occ, 1);
    const int64_t n_warp = a.n_roots - a.n_block;
    a.warp_chunk = (int)std::max<int64_t>(1, std::min<int64_t>(32, n_warp / (blocks * kWarps * 8)));
    // matrices that do not fit shared memory: per block, if any can occur
    if (m >= 3 && (g->max_root_words > kBlockWords || m == 4)) {
        a.big_words = (g->max_root_words + 3) & ~(int64_t)3;
        a.list_words = ((int64_t)g->max_deg + 4) & ~(int64_t)3;
    }
    const size_t per_block = sizeof(uint32_t) * (size_t)(2 * a.big_words + a.list_words);
    gp_status rc = fit_blocks(nsm, per_block, &blocks);
    if (rc != GP_OK) return rc;
    LaunchScratch mem(st);
    rc = mem.alloc(per_block * (size_t)blocks);
    if (rc != GP_OK) return rc;
    a.words = words;
    a.big = reinterpret_cast<uint32_t*>(mem.p);
    fn<<<(unsigned)blocks, kThreads, smem, st>>>(a);
    count_launch();
    GP_CUDA_TRY(cudaGetLastError());
    *warps = blocks * kWarps;
    return GP_OK;
}

}  // namespace gp
