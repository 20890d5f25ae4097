// pt_rules.h -- index and scheduling arithmetic of the kernels and their launchers, free of CUDA so that a host compiler
// takes it too (tests/test_rules_host.py runs it at sizes no GPU test reaches).
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define PT_HD __host__ __device__
#else
#define PT_HD
#endif

namespace ptgb {

// Warp of a thread counted over the grid.  64 bits: a block index times the block size passes 2^32 from 2^27 warps on, and
// a context may hold 2^28 chains.
PT_HD inline int64_t grid_warp(unsigned block, unsigned block_threads, unsigned thread) {
    return (int64_t)block * (block_threads / 32u) + thread / 32u;
}

}  // namespace ptgb
