// acc.cuh -- the per-lane 128-bit counter of the counting kernels and its
// warp reduction.
#pragma once
#include <cuda_runtime.h>

namespace gp {

struct Acc {   // per-lane 128-bit counter
    unsigned long long lo = 0, hi = 0;
    __device__ __forceinline__ void add(unsigned long long x) { lo += x; hi += (lo < x); }
    __device__ __forceinline__ void sub(unsigned long long x) { hi -= (lo < x); lo -= x; }
    __device__ __forceinline__ void add128(unsigned long long xl, unsigned long long xh) {
        lo += xl;
        hi += xh + (lo < xl);
    }
};

// Sum of the warp's counters, published with one atomic pair (low word,
// carry into the high word); the counters start over at zero.
static __device__ void flush(Acc& acc, unsigned long long* res) {
    unsigned long long lo = acc.lo, hi = acc.hi;
    for (int o = 16; o; o >>= 1) {
        unsigned long long l2 = __shfl_down_sync(0xffffffffu, lo, o);
        unsigned long long h2 = __shfl_down_sync(0xffffffffu, hi, o);
        lo += l2;
        hi += h2 + (lo < l2);
    }
    if ((threadIdx.x & 31) == 0 && (lo | hi)) {
        unsigned long long old = atomicAdd(res, lo);
        unsigned long long carry = (old + lo < old) ? 1ull : 0ull;
        if (hi + carry) atomicAdd(res + 1, hi + carry);
    }
    acc.lo = acc.hi = 0;
}

}  // namespace gp
