// bits.cuh -- what the kernels on local bit matrices share: adjacency tests
// against the graph, row strides, and the launch of a counting kernel with
// its few result words.
#pragma once
#include <cuda_runtime.h>

#include "engine.h"

namespace gp {

constexpr unsigned kAllLanes = 0xffffffffu;

// The data graph as the device sees it.
struct DeviceGraph {
    const int64_t* row_ptr;
    const int32_t* col;
    const int32_t* dplus;     // neighbours with a smaller id, per vertex
    const int32_t* roots;     // vertices by dplus, largest first
    const uint32_t* core_bits;
    int core_n, core_words;
};

inline DeviceGraph device_graph(const gp_graph* g) {
    return {g->row_ptr, g->col, g->dplus, g->roots, g->core_bits, g->core_bits ? g->core_n : 0, g->core_words};
}

static __device__ __forceinline__ unsigned lanes_below() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Row stride in words for n columns: whole 16-byte groups, an odd number of
// them, so that eight lanes reading 16 bytes of eight consecutive rows hit
// all 32 banks once.
__host__ __device__ constexpr int row_stride(int n) { return 4 * (((n + 127) / 128) | 1); }

static __device__ __forceinline__ void clear_words(uint32_t* M, int words, int first, int step) {
    for (int q = 4 * first; q < words; q += 4 * step) *reinterpret_cast<uint4*>(M + q) = make_uint4(0, 0, 0, 0);
}

// Result words of one counting launch, zero before it: the 128-bit total,
// work cursors, the busy-cycle sum, the error word.
struct ResultWords {
    unsigned long long total[2], cursor[3], busy;
    int err;
};

// The totals of n launches from their words as read back (res: two words
// each) and the sum of their busy cycles; an error word fails the call.
inline gp_status read_results(const ResultWords* words, int n, uint64_t* const* res, uint64_t* busy) {
    *busy = 0;
    for (int j = 0; j < n; ++j) {
        if (words[j].err) {
            set_error("count kernel reported internal error %d", words[j].err);
            return GP_ERR_INTERNAL;
        }
        res[j][0] = words[j].total[0];
        res[j][1] = words[j].total[1];
        *busy += words[j].busy;
    }
    return GP_OK;
}

// Stream-ordered scratch of one launch, released behind it.
struct LaunchScratch {
    cudaStream_t st;
    char* p = nullptr;
    explicit LaunchScratch(cudaStream_t s) : st(s) {}
    ~LaunchScratch() { if (p) cudaFreeAsync(p, st); }
    // GP_ERR_SCRATCH when the device has no room: the general kernel counts then.
    gp_status alloc(size_t bytes) {
        if (bytes == 0) return GP_OK;
        const cudaError_t e = cudaMallocAsync((void**)&p, bytes, st);
        if (e == cudaSuccess) return GP_OK;
        p = nullptr;
        cudaGetLastError();
        set_error("cannot allocate %zu bytes of scratch: %s", bytes, cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? GP_ERR_SCRATCH : GP_ERR_CUDA;
    }
};

// Reduce the *blocks of a launch that takes per_block bytes of scratch for each,
// in whole waves of SMs, until they take a quarter of the free device memory;
// GP_ERR_SCRATCH where one block an SM takes more than half of it (capi.cu).
gp_status fit_blocks(int64_t nsm, size_t per_block, int64_t* blocks);

// Launches that ask for more dynamic shared memory than this raise their
// kernel's limit first: the default is 48 KB with the static part, at most
// 8 KB in the kernels that ever ask for less than this.
constexpr size_t kDefaultShared = 40 * 1024;

// Raise the dynamic shared memory limit of a kernel, once per device, to
// `most`: the largest size any launch of it can ask for. The limit belongs to
// the function, not to a launch, so one set to a launch's own size would be
// lowered by another thread's smaller launch before this one starts (capi.cu).
gp_status raise_shared_limit(const void* kernel, size_t most);

}  // namespace gp
