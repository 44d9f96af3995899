// grid_stride.cuh -- a thread's cells in a grid-stride loop.  Also compiles as host C++, so
// that the index range can be replayed without a GPU (tests/test_grid_stride.py).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define CGK_HD __host__ __device__ __forceinline__
#else
#define CGK_HD inline
#endif

namespace cgk {

// Calls many(k, step) for W cells k, k + step, .., k + (W - 1) step at a time, then one(k) for
// the rest: every cell first, first + step, first + 2 step, .. below n, once and in order.
// The counter is 64-bit: a mesh may have up to 2^31 - 1 cells, and the counter passes n by up
// to W steps (a grid of 1216 blocks of 256 steps by 311,296).
template <int W, class Many, class One>
CGK_HD void grid_stride(int64_t n, int64_t first, int64_t step, Many many, One one) {
    int64_t k = first;
    for (; k + (W - 1) * step < n; k += W * step) many(k, step);
    for (; k < n; k += step) one(k);
}

}  // namespace cgk
