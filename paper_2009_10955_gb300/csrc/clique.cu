// clique.cu -- k-clique counts (k = 3..7) on local bit matrices.
//
// A clique's plan searches v0 > v1 > ... > v(k-1) (ids; with the degree
// order, v0 has the lowest degree), every vertex in the neighbourhood of all
// earlier ones. Everything after v0 therefore happens inside
// U = N(v0) ∩ [0, v0), which is short on a degree-ordered graph (at most 600
// vertices on a skewed graph of a million) and sorted, so positions in U keep
// the id order. For a root v0 the kernel builds the strictly lower triangular
// bit matrix L of the graph induced on U (row i: neighbours of U[i] among
// U[0..i)), and the count is the number of (k-1)-cliques of L. The last three
// vertices are counted by a dense pass over a bit matrix: for rows k < j with
// bit (j, k) set, popc(row j & row k). Each vertex before those compacts the
// matrix to the neighbours of one row, so that the dense pass runs on words
// that hold little but members.
//
// What bounds it: the 32-bit logic and population-count pipes; the graph is
// read once to build the matrices (one bit probe of the core matrix, or a
// binary search, per pair of U).
#include <algorithm>
#include <vector>

#include "acc.cuh"
#include "bits.cuh"
#include "engine.h"

namespace gp {

namespace {

constexpr unsigned kFull = kAllLanes;
// Largest matrix a single warp works on, in rows: 128 rows of 4 words are
// 2 KB of shared memory per level, and the pass over it takes a few
// microseconds.
constexpr int kWarpRows = 128;
constexpr int kWarpWords = kWarpRows / 32;
// Largest matrix a block keeps in shared memory, in rows (20-word rows:
// 51 KB, twice: the root's and the compacted one).
constexpr int kBlockRows = 640;
// Largest root matrix at all; beyond it the general kernel counts.
constexpr int kMostRows = 4096;

struct CliqueArgs {
    DeviceGraph g;            // dplus is |U|, roots are the vertices by |U|
    int64_t task_begin, task_end;
    int64_t n_block;          // leading roots handled by a whole block each ...
    int parts;                // ... in this many parts (the rows modulo parts)
    int64_t n_roots;          // roots worth visiting (|U| >= k - 1)
    int warp_chunk;           // roots a warp takes per grab
    int block_rows;           // rows of the root's matrix in shared memory
    uint32_t* big;            // two matrices and a member list per block for larger ones (global)
    int64_t big_words;        // words of one of the matrices there
    int big_stride;
    uint32_t* sets;           // 4 sets per warp for masked_cliques (global)
    ResultWords* words;       // cursors: block items, warp roots
};

// Is y (below x) a neighbour of x? Core rows answer with one bit; other
// lists are searched below their own vertex.
__device__ __forceinline__ bool adjacent(const CliqueArgs& a, int x, int y) {
    if (x < a.g.core_n)
        return (__ldg(a.g.core_bits + (size_t)x * a.g.core_words + (y >> 5)) >> (y & 31)) & 1u;
    const int32_t* p = a.g.col + __ldg(a.g.row_ptr + x);
    int n = __ldg(a.g.dplus + x), base = 0;
    while (n > 0) {
        const int half = n >> 1;
        if (__ldg(p + base + half) < y) { base += half + 1; n -= half + 1; } else n = half;
    }
    return base < __ldg(a.g.dplus + x) && __ldg(p + base) == y;
}

// A row of a graph without the degree order by the list of its own vertex x,
// one warp: a hub of the larger ids has many smaller neighbours with lists
// shorter than the row, and such a list is looked up in U (5-cliques of R-MAT 14
// with the ids reversed: 14.9 -> 7.3 ms); short rows cost no more by their
// pairs. False, nothing written, for the others.
__device__ __forceinline__ bool walk_row(const CliqueArgs& a, const int32_t* U, int i, int x, uint32_t* row, int stride,
                                      int lane) {
    const int len = __ldg(a.g.dplus + x);
    if (i < 256 || 4 * len >= i) return false;
    for (int w = lane; w < stride; w += 32) row[w] = 0u;
    __syncwarp();
    const int32_t* list = a.g.col + __ldg(a.g.row_ptr + x);
    for (int e = lane; e < len; e += 32) {
        const int y = __ldg(list + e);
        int base = 0, n = i;
        while (n > 0) {
            const int half = n >> 1;
            if (__ldg(U + base + half) < y) { base += half + 1; n -= half + 1; } else n = half;
        }
        if (base < i && __ldg(U + base) == y) atomicOr(row + (base >> 5), 1u << (base & 31));
    }
    return true;
}

// Row i of the root's matrix, one warp: a ballot per 32 columns. The words
// above the diagonal are zero: a compaction reads them. kWalk: 5-cliques and
// larger ones only, as 4-cliques of such graphs are the general kernel's.
template <bool kWalk>
__device__ __forceinline__ void build_row(const CliqueArgs& a, const int32_t* U, int i, uint32_t* row, int stride,
                                          int lane) {
    const int x = __ldg(U + i);
    if (kWalk && a.g.core_n == 0 && walk_row(a, U, i, x, row, stride, lane)) return;
    const int nw = (i >> 5) + 1;
    for (int w = 0; w < nw; ++w) {
        const int j = 32 * w + lane;
        const bool hit = j < i && adjacent(a, x, __ldg(U + j));
        const uint32_t b = __ballot_sync(kFull, hit);
        if (lane == 0) row[w] = b;
    }
    for (int w = nw + lane; w < stride; w += 32) row[w] = 0u;
}

// Four consecutive rows at once, so that their probes overlap.
template <bool kWalk>
__device__ __forceinline__ void build_rows4(const CliqueArgs& a, const int32_t* U, int i0, int n, uint32_t* M,
                                            int stride, int lane) {
    const int last = min(i0 + 3, n - 1);
    int x[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) x[t] = __ldg(U + min(i0 + t, last));
    // ids grow with the position: the last row is outside the core first
    if (x[3] >= a.g.core_n) {
        for (int i = i0; i <= last; ++i) build_row<kWalk>(a, U, i, M + (size_t)i * stride, stride, lane);
        return;
    }
    const int nw = (last >> 5) + 1;
    for (int w = 0; w < nw; ++w) {
        const int j = 32 * w + lane;
        const int y = (j < last) ? __ldg(U + j) : 0;
        const uint32_t bit = 1u << (y & 31);
        uint32_t v[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) v[t] = __ldg(a.g.core_bits + (size_t)x[t] * a.g.core_words + (y >> 5));
        uint32_t mine = 0;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const uint32_t b = __ballot_sync(kFull, j < i0 + t && (v[t] & bit));
            if (lane == t) mine = b;
        }
        if (lane < 4 && i0 + lane <= last) M[(size_t)(i0 + lane) * stride + w] = mine;
    }
    for (int w = nw + (lane >> 2); w < stride; w += 8)
        if (i0 + (lane & 3) <= last) M[(size_t)(i0 + (lane & 3)) * stride + w] = 0u;
}

// Triangles of a strictly lower triangular matrix of s <= 32 one-word rows
// (zero rows up to a multiple of four), the largest vertex in [lo, hi): lane
// k holds row k, the rows j are read four at a time (one broadcast load).
template <bool kRange>
__device__ __forceinline__ unsigned triangles32(const uint32_t* M, int s, int lo, int hi, int lane) {
    const uint32_t own = (lane < s) ? M[lane] : 0u;
    const uint32_t bit = 1u << lane;
    unsigned c = 0;
    for (int j = kRange ? (lo & ~3) : 0; j < (kRange ? hi : s); j += 4) {
        const uint4 r = *reinterpret_cast<const uint4*>(M + j);
        if ((r.x & bit) && (!kRange || j >= lo)) c += __popc(r.x & own);
        if ((r.y & bit) && (!kRange || (j + 1 >= lo && j + 1 < hi))) c += __popc(r.y & own);
        if ((r.z & bit) && (!kRange || (j + 2 >= lo && j + 2 < hi))) c += __popc(r.z & own);
        if ((r.w & bit) && (!kRange || (j + 3 >= lo && j + 3 < hi))) c += __popc(r.w & own);
    }
    return c;
}

// The same for s <= 128 rows of four words: for each word of columns, lane k
// holds row 32 wk + k and walks the rows j above it.
template <int WK>
__device__ __forceinline__ unsigned triangles_word(const uint32_t* M, int s, int lo, int hi, int lane) {
    const int k = 32 * WK + lane;
    uint4 own = make_uint4(0, 0, 0, 0);
    if (k < s) own = *reinterpret_cast<const uint4*>(M + 4 * k);
    const uint32_t bit = 1u << lane;
    unsigned c = 0;
#pragma unroll 4
    for (int j = max(lo, 32 * WK + 1); j < hi; ++j) {
        const uint4 r = *reinterpret_cast<const uint4*>(M + 4 * j);
        const uint32_t act = (WK == 0 ? r.x : WK == 1 ? r.y : WK == 2 ? r.z : r.w) & bit;
        unsigned p = __popc(r.x & own.x);
        if (WK >= 1) p += __popc(r.y & own.y);
        if (WK >= 2) p += __popc(r.z & own.z);
        if (WK >= 3) p += __popc(r.w & own.w);
        if (act) c += p;
    }
    return c;
}

template <bool kRange>
__device__ __forceinline__ unsigned triangles_warp(const uint32_t* M, int s, int lo, int hi, int lane) {
    if (s <= 32) return triangles32<kRange>(M, s, lo, hi, lane);
    unsigned c = triangles_word<0>(M, s, lo, hi, lane);
    c += triangles_word<1>(M, s, lo, hi, lane);
    if (s > 64) c += triangles_word<2>(M, s, lo, hi, lane);
    if (s > 96) c += triangles_word<3>(M, s, lo, hi, lane);
    return c;
}

// A warp's share (unit = warp, warp + nwarps, ...) of the triangles of a
// larger matrix: a unit is one word of columns and eight rows j.
__device__ __forceinline__ unsigned triangles_block(const uint32_t* M, int stride, int s, int lo, int hi, int lane,
                                                    int warp, int nwarps) {
    const int nw = (s + 31) >> 5, j0 = lo & ~7, chunks = (hi - j0 + 7) >> 3;
    unsigned total = 0;
    for (int u = warp; u < nw * chunks; u += nwarps) {
        const int wk = u % nw, j = j0 + 8 * (u / nw);
        if (min(j + 7, hi - 1) <= 32 * wk) continue;         // no row of the unit is above a column
        const int k = min(32 * wk + lane, s - 1);
        unsigned c[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int q = 0; q <= (wk >> 2); ++q) {
            const uint4 own = *reinterpret_cast<const uint4*>(M + (size_t)k * stride + 4 * q);
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int jt = min(max(j + t, 32 * wk), hi - 1);
                const uint4 r = *reinterpret_cast<const uint4*>(M + (size_t)jt * stride + 4 * q);
                c[t] += __popc(r.x & own.x) + __popc(r.y & own.y) + __popc(r.z & own.z) + __popc(r.w & own.w);
            }
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int jt = j + t;
            if (jt < lo || jt >= hi || jt <= 32 * wk) continue;
            if (M[(size_t)jt * stride + wk] >> lane & 1u) total += c[t];
        }
    }
    return total;
}

// The members of a set as a warp (or block) uses them to compact a matrix:
// their positions and their rows' offsets, the offsets padded to a multiple
// of four with row 0 (which is all zero).
struct Members {
    uint32_t* off;
    uint16_t* pos;
};

__device__ __forceinline__ int expand(const uint32_t* S, int nw, int stride, Members mem, int lane) {
    int n = 0;
    for (int w = 0; w < nw; ++w) {
        const uint32_t x = S[w];
        if (x >> lane & 1u) {
            const int at = n + __popc(x & lanes_below()), p = 32 * w + lane;
            mem.pos[at] = (uint16_t)p;
            mem.off[at] = (uint32_t)(p * stride);
        }
        n += __popc(x);
    }
    if (lane < (-n & 3)) mem.off[n + lane] = 0u;
    __syncwarp();
    return n;
}

__device__ __forceinline__ int size_of(const uint32_t* S, int nw) {
    int n = 0;
    for (int w = 0; w < nw; ++w) n += __popc(S[w]);
    return n;
}

// The matrix induced by M on s <= 32 members (one-word rows): which members
// below m are neighbours of member m. A ballot gives a row.
__device__ __forceinline__ void compact32(const uint32_t* M, Members mem, int s, uint32_t* out, int lane) {
    const int p = (lane < s) ? mem.pos[lane] : 0;
    const uint32_t* base = M + (p >> 5);
    const uint32_t bit = (lane < s) ? (1u << (p & 31)) : 0u;
    for (int m = 0; m < s; m += 4) {
        const uint4 o = *reinterpret_cast<const uint4*>(mem.off + m);
        uint4 b;
        b.x = __ballot_sync(kFull, base[o.x] & bit);
        b.y = __ballot_sync(kFull, base[o.y] & bit);
        b.z = __ballot_sync(kFull, base[o.z] & bit);
        b.w = __ballot_sync(kFull, base[o.w] & bit);
        if (lane == 0) *reinterpret_cast<uint4*>(out + m) = b;
    }
}

// The same for any s: word by word of columns, rows in fours, the fours
// `first`, first + step, ... by this warp. Words above the diagonal are zero.
__device__ __forceinline__ void compact(const uint32_t* M, Members mem, int s, uint32_t* out, int out_stride,
                                        int lane, int first, int step) {
    for (int g = 0; 32 * g < s; ++g) {
        const int c = 32 * g + lane;
        const int p = (c < s) ? mem.pos[c] : 0;
        const uint32_t* base = M + (p >> 5);
        const uint32_t bit = (c < s) ? (1u << (p & 31)) : 0u;
        for (int m = 4 * (8 * g + first); m < s; m += 4 * step) {
            const uint4 o = *reinterpret_cast<const uint4*>(mem.off + m);
            uint32_t b[4];
            b[0] = __ballot_sync(kFull, base[o.x] & bit);
            b[1] = __ballot_sync(kFull, base[o.y] & bit);
            b[2] = __ballot_sync(kFull, base[o.z] & bit);
            b[3] = __ballot_sync(kFull, base[o.w] & bit);
            if (lane == 0) {
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (m + t < s) out[(m + t) * out_stride + g] = b[t];
            }
        }
    }
}

// The members' matrix (s <= kWarpRows) in a warp's own buffer.
__device__ __forceinline__ void compact_own(const uint32_t* M, Members mem, int s, uint32_t* out, int lane) {
    if (s <= 32) {
        compact32(M, mem, s, out, lane);
    } else {
        clear_words(out, s * kWarpWords, lane, 32);
        __syncwarp();
        compact(M, mem, s, out, kWarpWords, lane, 0, 1);
    }
    __syncwarp();
}

// R-cliques of a warp's matrix (s rows), R >= 3, largest vertex in [lo, hi)
// (kRange; all of them otherwise). Deeper levels use the following
// kWarpRows x kWarpWords buffers.
template <int R, bool kRange>
__device__ __forceinline__ void warp_cliques(uint32_t* M, Members mem, int s, int lo, int hi, int lane, Acc& acc) {
    if constexpr (R == 3) {
        acc.add(triangles_warp<kRange>(M, s, lo, hi, lane));
    } else {
        const int stride = (s <= 32) ? 1 : kWarpWords;
        uint32_t* next = M + kWarpRows * kWarpWords;
        for (int i = max(lo, R - 1); i < hi; ++i) {
            const int t = expand(M + i * stride, (i >> 5) + 1, stride, mem, lane);
            if (t >= R - 1) {
                compact_own(M, mem, t, next, lane);
                warp_cliques<R - 1, false>(next, mem, t, 0, t, lane, acc);
            }
            __syncwarp();
        }
    }
}

// R-cliques inside the set S (nw words) of a matrix, one warp, for sets too
// large for the warp's own matrices: sets of deeper levels go to `sets`.
template <int R>
__device__ void masked_cliques(const uint32_t* M, int stride, const uint32_t* S, int nw, uint32_t* sets, int lane,
                               Acc& acc) {
    if constexpr (R == 2) {
        unsigned long long c = 0;
        for (int w = 0; w < nw; ++w) {
            if (!(S[w] >> lane & 1u)) continue;
            const uint32_t* row = M + (size_t)(32 * w + lane) * stride;
            for (int q = 0; q <= w; ++q) c += __popc(S[q] & row[q]);
        }
        acc.add(c);
        __syncwarp();
    } else {
        for (int w = 0; w < nw; ++w)
            for (uint32_t x = S[w]; x; x &= x - 1) {
                const int j = 32 * w + __ffs(x) - 1;
                for (int q = lane; q <= w; q += 32) sets[q] = S[q] & M[(size_t)j * stride + q];
                __syncwarp();
                masked_cliques<R - 1>(M, stride, sets, w + 1, sets + kMostRows / 32, lane, acc);
                __syncwarp();
            }
    }
}

// Shared state of a block working on one root.
struct BlockState {
    int next;                 // next row (or row of the compacted matrix) to hand to a warp
    int n_large;              // rows with more neighbours than a warp's matrix holds ...
    uint16_t large[kMostRows];// ... and which
};

// (K-2)-cliques inside one row's neighbours when they are more than a warp's
// matrix holds: the block compacts the root's matrix to them (into C) and
// shares out the rows of the result.
template <int K>
__device__ __forceinline__ void block_row(const uint32_t* L, int stride, int i, uint32_t* C, Members bmem,
                                          uint32_t* own, Members mem, BlockState* bs, uint32_t* sets, Acc& acc) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const uint32_t* S = L + (size_t)i * stride;
    const int nw = (i >> 5) + 1, t = size_of(S, nw), cs = row_stride(t);
    __syncthreads();                                 // C, bmem and the warps' buffers are free
    if (warp == 0) expand(S, nw, stride, bmem, lane);
    clear_words(C, t * cs, threadIdx.x, blockDim.x);
    if (threadIdx.x == 0) bs->next = 0;
    __syncthreads();
    compact(L, bmem, t, C, cs, lane, warp, nwarps);
    __syncthreads();
    if constexpr (K == 5) {
        acc.add(triangles_block(C, cs, t, 0, t, lane, warp, nwarps));
    } else {
        for (;;) {
            int q = 0;
            if (lane == 0) q = atomicAdd(&bs->next, 1);
            q = __shfl_sync(kFull, q, 0);
            const int j = t - 1 - q;
            if (j < 0) break;
            const uint32_t* T = C + (size_t)j * cs;
            const int jw = (j >> 5) + 1, size = size_of(T, jw);
            if (size < K - 3) continue;
            if (size <= kWarpRows) {
                const int u = expand(T, jw, cs, mem, lane);
                compact_own(C, mem, u, own, lane);
                warp_cliques<K - 3, false>(own, mem, u, 0, u, lane, acc);
                __syncwarp();
            } else {
                masked_cliques<K - 3>(C, cs, T, jw, sets, lane, acc);
            }
        }
    }
}

// Everything under one root for a whole block: the rows [lo, hi) of its
// matrix L with (hi - 1 - i) mod parts == part. `spare` (spare_words of
// shared memory) and G (global) hold the compacted matrix of large rows.
template <int K>
__device__ __forceinline__ void block_root(const CliqueArgs& a, const int32_t* U, int lo, int hi, int part, int parts,
                                           uint32_t* L, int stride, uint32_t* spare, int spare_words, uint32_t* G,
                                           Members bmem, uint32_t* own, Members mem, BlockState* bs, uint32_t* sets,
                                           Acc& acc) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int i = 4 * warp; i < hi; i += 4 * nwarps) build_rows4<(K > 4)>(a, U, i, hi, L, stride, lane);
    if (threadIdx.x == 0) { bs->next = 0; bs->n_large = 0; }
    __syncthreads();
    if constexpr (K == 4) {
        acc.add(triangles_block(L, stride, hi, lo, hi, lane, warp, nwarps));
    } else {
        // rows whose neighbours fit a warp's matrix, one warp each
        for (;;) {
            int q = 0;
            if (lane == 0) q = atomicAdd(&bs->next, 1);
            q = __shfl_sync(kFull, q, 0);
            const int i = hi - 1 - part - q * parts;
            if (i < lo) break;
            const uint32_t* S = L + (size_t)i * stride;
            const int nw = (i >> 5) + 1, size = size_of(S, nw);
            if (size < K - 2) continue;
            if (size > kWarpRows) {
                if (lane == 0) bs->large[atomicAdd(&bs->n_large, 1)] = (uint16_t)i;
                continue;
            }
            expand(S, nw, stride, mem, lane);
            compact_own(L, mem, size, own, lane);
            warp_cliques<K - 2, false>(own, mem, size, 0, size, lane, acc);
            __syncwarp();
        }
        __syncthreads();
        // the others, one at a time by the block
        const int n_large = bs->n_large;
        for (int q = 0; q < n_large; ++q) {
            const int i = bs->large[q];
            const int t = size_of(L + (size_t)i * stride, (i >> 5) + 1);
            if (t * row_stride(t) <= spare_words)
                block_row<K>(L, stride, i, spare, bmem, own, mem, bs, sets, acc);
            else
                block_row<K>(L, stride, i, G, bmem, own, mem, bs, sets, acc);
        }
    }
    __syncthreads();                                   // the matrices are free again
}

// Pairs of U joined by an edge, rows [lo, hi) shared out over nwarps warps
// (the triangles of one root): no matrix is stored.
__device__ __forceinline__ unsigned edges_of(const CliqueArgs& a, const int32_t* U, int lo, int hi, int first,
                                             int step, int lane) {
    unsigned c = 0;
    for (int i0 = lo + 4 * first; i0 < hi; i0 += 4 * step) {
        const int last = min(i0 + 3, hi - 1);
        int x[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) x[t] = __ldg(U + min(i0 + t, last));
        if (x[3] >= a.g.core_n) {
            for (int i = i0; i <= last; ++i)
                for (int j = lane; j < i; j += 32) c += adjacent(a, __ldg(U + i), __ldg(U + j));
            continue;
        }
        for (int j = lane; j < last; j += 32) {
            const int y = __ldg(U + j);
            uint32_t v[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) v[t] = __ldg(a.g.core_bits + (size_t)x[t] * a.g.core_words + (y >> 5));
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (j < i0 + t && i0 + t <= last) c += (v[t] >> (y & 31)) & 1u;
        }
    }
    return c;
}

// Shared memory, in words. Block phase: the root's matrix L, a member list,
// then per warp its member list and its matrices (one per level below the
// row); for K = 5 the compacted matrix of a large row overlays the warps'
// matrices, which are idle meanwhile. Warp phase: per warp its member list and
// one matrix more (the root's own).
template <int K>
struct Layout {
    static constexpr int kThreads = K == 3 ? 256 : K <= 5 ? 512 : 256;
    static constexpr int kWarps = kThreads / 32;
    static constexpr int kMatrix = kWarpRows * kWarpWords;
    static constexpr int kList = kWarpRows + kWarpRows / 2;       // offsets, positions
    static constexpr int kBlockLevels = K <= 4 ? 0 : K - 4;
    static constexpr int kWarpLevels = K == 3 ? 0 : K - 3;
    static constexpr int kWarpPhase = kWarps * (kList + kWarpLevels * kMatrix);
    __host__ __device__ static int matrix_words(int rows) { return rows * row_stride(rows); }
    __host__ __device__ static int list_words(int rows) { return K <= 4 ? 0 : (rows + (rows + 1) / 2 + 7) & ~3; }
    __host__ __device__ static int block_phase(int rows) {
        return matrix_words(rows) + list_words(rows) + kWarps * ((K <= 4 ? 0 : kList) + kBlockLevels * kMatrix);
    }
    __host__ __device__ static int words(int rows) { const int b = block_phase(rows); return b > kWarpPhase ? b : kWarpPhase; }
};

template <int K>
__global__ void __launch_bounds__(Layout<K>::kThreads, K == 3 ? 5 : K <= 5 ? 2 : 3)
k_clique(const __grid_constant__ CliqueArgs a) {
    using Y = Layout<K>;
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ BlockState bs;
    __shared__ unsigned long long s_item;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const long long t_start = clock64();
    Acc acc;
    // large roots: one block each, largest first
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(&a.words->cursor[0], 1ull);
        __syncthreads();
        const unsigned long long item = s_item;
        if (item >= (unsigned long long)a.n_block * a.parts) break;
        const int v0 = __ldg(a.g.roots + item / a.parts), part = (int)(item % a.parts);
        const int64_t rb = __ldg(a.g.row_ptr + v0);
        const int n = __ldg(a.g.dplus + v0);
        const int lo = (int)max((int64_t)0, min((int64_t)n, a.task_begin - rb));
        const int hi = (int)max((int64_t)0, min((int64_t)n, a.task_end - rb));
        if (lo >= hi) continue;
        const int32_t* U = a.g.col + rb;
        if constexpr (K == 3) {
            acc.add(edges_of(a, U, lo, hi, warp, nwarps, lane));
        } else {
            // lists and matrices behind L
            uint32_t* at = smem + Y::matrix_words(a.block_rows);
            Members bmem{at, reinterpret_cast<uint16_t*>(at + ((a.block_rows + 3) & ~3))};
            at += Y::list_words(a.block_rows);
            Members mem{at + warp * Y::kList, reinterpret_cast<uint16_t*>(at + warp * Y::kList + kWarpRows)};
            at += Y::kWarps * Y::kList;
            uint32_t* own = at + warp * Y::kBlockLevels * Y::kMatrix;
            const int spare = K == 5 ? Y::kWarps * Y::kMatrix : 0;
            uint32_t* G = a.big + (size_t)blockIdx.x * (2 * a.big_words + 2 * kMostRows);
            uint32_t* sets = a.sets + ((size_t)blockIdx.x * nwarps + warp) * 4 * (kMostRows / 32);
            if (n <= a.block_rows) {
                block_root<K>(a, U, lo, hi, part, a.parts, smem, row_stride(a.block_rows), at, spare, G, bmem, own, mem,
                              &bs, sets, acc);
            } else {
                uint32_t* list = G + 2 * a.big_words;
                Members gmem{list, reinterpret_cast<uint16_t*>(list + kMostRows)};
                block_root<K>(a, U, lo, hi, part, a.parts, G + a.big_words, a.big_stride, at, spare, G, gmem, own, mem,
                              &bs, sets, acc);
            }
        }
    }
    __syncthreads();
    // the others: a warp each
    const unsigned long long n_warp = (unsigned long long)(a.n_roots - a.n_block);
    uint32_t* const area = smem + warp * (Y::kList + Y::kWarpLevels * Y::kMatrix);
    const Members mem{area, reinterpret_cast<uint16_t*>(area + kWarpRows)};
    uint32_t* const own = area + Y::kList;
    for (;;) {
        unsigned long long t0 = 0;
        if (lane == 0) t0 = atomicAdd(&a.words->cursor[1], (unsigned long long)a.warp_chunk);
        t0 = __shfl_sync(kFull, t0, 0);
        if (t0 >= n_warp) break;
        // lane l fetches root l of the chunk
        const bool have = lane < a.warp_chunk && t0 + lane < n_warp;
        const int lv = have ? __ldg(a.g.roots + a.n_block + t0 + lane) : 0;
        const int64_t lrb = have ? __ldg(a.g.row_ptr + lv) : 0;
        const int ln = have ? __ldg(a.g.dplus + lv) : 0;
        for (int q = 0; q < a.warp_chunk; ++q) {
            const int64_t rb = __shfl_sync(kFull, lrb, q);
            const int n = __shfl_sync(kFull, ln, q);
            const int lo = (int)max((int64_t)0, min((int64_t)n, a.task_begin - rb));
            const int hi = (int)max((int64_t)0, min((int64_t)n, a.task_end - rb));
            if (lo >= hi || hi < K - 1) continue;
            const int32_t* U = a.g.col + rb;
            if constexpr (K == 3) {
                acc.add(edges_of(a, U, lo, hi, 0, 1, lane));
            } else {
                const int stride = (hi <= 32) ? 1 : kWarpWords;
                if (hi <= 32 && lane < (-hi & 3)) own[hi + lane] = 0u;             // one-word rows: zero up to a multiple of four
                for (int i = 0; i < hi; i += 4) build_rows4<(K > 4)>(a, U, i, hi, own, stride, lane);
                __syncwarp();
                if (lo == 0) warp_cliques<K - 1, false>(own, mem, hi, 0, hi, lane, acc);
                else warp_cliques<K - 1, true>(own, mem, hi, lo, hi, lane, acc);
                __syncwarp();
            }
        }
    }
    flush(acc, a.words->total);
    if (lane == 0) atomicAdd(&a.words->busy, (unsigned long long)(clock64() - t_start));
}

struct Variant {
    void (*fn)(const CliqueArgs);
    int threads;
    int (*words)(int);
};

template <int K>
Variant variant() { return {k_clique<K>, Layout<K>::kThreads, Layout<K>::words}; }

Variant variant_for(int k) {
    switch (k) {
        case 3: return variant<3>();
        case 4: return variant<4>();
        case 5: return variant<5>();
        case 6: return variant<6>();
        default: return variant<7>();
    }
}

bool is_clique_plan(const GpPlan& P, bool* descending) {
    if (P.labeled || P.iep || P.k < 3) return false;
    *descending = true;
    for (int d = 1; d < P.k; ++d) {
        const uint8_t all = (uint8_t)((1u << d) - 1u);
        if (P.lvl[d].op_mask != all) return false;
        if (P.lvl[d].hi_mask != all) *descending = false;
    }
    return true;
}

}  // namespace

bool clique_applies(const CountJob& job, const gp_graph* g, const LaunchOpts& opt) {
    bool descending = false;
    if (opt.stats || opt.no_core || opt.bitmap_mode != 2 || opt.budget_cycles > 0 || opt.task_cycles > 0) return false;
    if (!g->roots || g->max_dplus > kMostRows || !is_clique_plan(job.plan, &descending)) return false;
    // without the degree order a hub's list below it is long and all its pairs
    // are probed, where the general kernel walks the shorter list of each
    // (triangles of an unordered R-MAT 14: 1.58 against 1.44 ms; 5-cliques 1.8
    // against 35 ms). Hubs over a sparse rest hold few cliques: with pairs of
    // smaller neighbours beyond 200 an entry the matrices cost more than the
    // lists (500 hubs of 3000 neighbours among the largest ids, 658 an entry:
    // 5-cliques 6.8 against 2.7 ms, 6-cliques 40 against 2.7; R-MAT 14 with the
    // ids reversed, 109: 7.3 against 232)
    if (!g->perm && (job.plan.k <= 4 ? (int64_t)g->max_deg * g->n > 8 * g->nnz : g->dplus_pairs > 200.0 * (double)g->nnz))
        return false;
    // a clique's count over all tasks is the same under every plan; over some
    // of them it is the plan's own
    return descending || (job.task_begin == 0 && job.ntasks == g->nnz);
}

gp_status launch_clique(const CountJob& job, const gp_graph* g, cudaStream_t st, ResultWords* words, int64_t* warps) {
    const int k = job.plan.k;
    int dev = 0, nsm = 0;
    GP_CUDA_TRY(cudaGetDevice(&dev));
    GP_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    CliqueArgs a = {};
    a.g = device_graph(g);
    a.task_begin = job.task_begin;
    a.task_end = job.task_begin + job.ntasks;
    // a root goes to a whole block from |U| = 128 (the largest warp matrix);
    // from fewer for 6- and 7-cliques, whose work grows with a higher power
    // of |U|, and where the smaller roots are no more than the SMs
    int block_class = k <= 5 ? 7 : k == 6 ? 6 : 5;
    while (k >= 5 && block_class > 4 && g->roots_ge[block_class - 1] <= 2 * (int64_t)nsm) --block_class;
    a.n_block = g->roots_ge[block_class];
    a.n_roots = g->roots_ge[k <= 4 ? 1 : 2];
    const Variant var = variant_for(k);
    const int threads = var.threads;
    a.block_rows = a.n_block > 0 ? std::min(g->max_dplus, kBlockRows) : 0;
    const size_t smem = k == 3 ? 0 : sizeof(uint32_t) * (size_t)var.words(a.block_rows);
    auto fn = var.fn;
    if (smem > kDefaultShared) {
        const gp_status rc = raise_shared_limit((const void*)fn, sizeof(uint32_t) * (size_t)var.words(kBlockRows));
        if (rc != GP_OK) return rc;
    }
    int occ = 0;
    GP_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem));
    int64_t blocks = (int64_t)nsm * std::max(occ, 1);
    const bool big = (k > 3 && g->max_dplus > kBlockRows) || (k > 4 && g->max_dplus > kWarpRows);
    if (big) {
        a.big_stride = row_stride(g->max_dplus);
        a.big_words = ((int64_t)g->max_dplus * a.big_stride + 3) & ~(int64_t)3;
    }
    const size_t big_b = big ? sizeof(uint32_t) * (2 * (size_t)a.big_words + 2 * kMostRows) : 0;
    const size_t sets_b = k >= 6 && a.n_block > 0 ? sizeof(uint32_t) * (size_t)(threads / 32) * 4 * (kMostRows / 32) : 0;
    // asking for the free memory takes 12 us, a quarter of a small count: scratch
    // of up to 64 MB is simply asked for (without it the general kernel counts)
    gp_status rc = (big_b + sets_b) * (size_t)blocks > ((size_t)64 << 20) ? fit_blocks(nsm, big_b + sets_b, &blocks) : GP_OK;
    if (rc != GP_OK) return rc;
    // roots are cut into parts where they are too few to fill the grid evenly.
    // Each part builds the root's matrix anew, which is most of the work where
    // it is large and sparse, as under hubs of a graph without the degree order:
    // 6-cliques of 500 hubs of 600 neighbours 5.4 ms in 58 parts, 2.4 in 16
    a.parts = k <= 4 || a.n_block == 0 ? 1
              : (int)std::max<int64_t>(1, std::min<int64_t>(k == 5 ? 8 : g->perm ? 64 : 16, (k == 5 ? 16 : 64) * blocks / a.n_block));
    const int64_t n_warp = a.n_roots - a.n_block;
    a.warp_chunk = (int)std::max<int64_t>(1, std::min<int64_t>(32, n_warp / (blocks * (threads / 32) * 8)));
    LaunchScratch mem(st);
    rc = mem.alloc((big_b + sets_b) * (size_t)blocks);
    if (rc != GP_OK) return rc;
    a.words = words;
    a.big = reinterpret_cast<uint32_t*>(mem.p);
    a.sets = reinterpret_cast<uint32_t*>(mem.p + big_b * (size_t)blocks);
    fn<<<(unsigned)blocks, threads, smem, st>>>(a);
    count_launch();
    GP_CUDA_TRY(cudaGetLastError());
    *warps = blocks * (threads / 32);
    return GP_OK;
}

}  // namespace gp
