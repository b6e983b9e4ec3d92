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

// Run a counting kernel: 64 zeroed bytes of result words (two of the 128-bit
// total, three cursors, the busy-cycle sum) and `extra` bytes behind them,
// launch(mem), read the words back, synchronise.
struct ResultWords {
    unsigned long long total[2], cursor[3], busy;
};

template <class Launch>
gp_status run_with_words(cudaStream_t st, size_t extra, float* kernel_ms, uint64_t* results, uint64_t* busy,
                         const char* what, Launch launch) {
    static_assert(sizeof(ResultWords) <= 64, "result words");
    char* mem = nullptr;
    GP_CUDA_TRY(cudaMallocAsync((void**)&mem, 64 + extra, st));
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    ResultWords h = {};
    cudaError_t e = cudaSuccess;
    if (kernel_ms) {
        e = cudaEventCreate(&ev0);
        if (e == cudaSuccess) e = cudaEventCreate(&ev1);
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(mem, 0, 64, st);
    if (e == cudaSuccess && ev0) e = cudaEventRecord(ev0, st);
    if (e == cudaSuccess) {
        launch(reinterpret_cast<ResultWords*>(mem), mem + 64);
        count_launch();
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && ev1) e = cudaEventRecord(ev1, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, mem, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess && ev1) e = cudaEventElapsedTime(kernel_ms, ev0, ev1);
    if (ev0) cudaEventDestroy(ev0);
    if (ev1) cudaEventDestroy(ev1);
    cudaFreeAsync(mem, st);
    if (e != cudaSuccess) {
        set_error("%s kernel failed: %s", what, cudaGetErrorString(e));
        return GP_ERR_CUDA;
    }
    results[0] = h.total[0];
    results[1] = h.total[1];
    if (busy) *busy = h.busy;
    return GP_OK;
}

}  // namespace gp
