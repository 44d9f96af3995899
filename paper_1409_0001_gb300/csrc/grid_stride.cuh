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
// A mesh may have up to 2^31 - 1 cells and the counter passes n by up to W steps (a grid of 1216
// blocks of 256 steps by 311,296): beyond an int, within an unsigned up to steps of 2^31 / W.
// (With a 64-bit counter the FP64 update needs 108 registers and an iteration of 128^3 cells
// takes 6 % longer.)
template <int W, class Many, class One>
CGK_HD void grid_stride(uint32_t n, uint32_t first, uint32_t step, Many many, One one) {
    uint32_t k = first;
    for (; k + (W - 1) * step < n; k += W * step) many(k, step);
    for (; k < n; k += step) one(k);
}

}  // namespace cgk
