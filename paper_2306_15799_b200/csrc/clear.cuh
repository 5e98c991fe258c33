// Zeroes the accumulators of a call (status words, arrival counters, K', V'; da, db of the backward pass; E X, F X of
// the call with linear maps) as the first kernel of a chain of programmatically dependent launches.
//
// A memset node costs the host more than a kernel launch (4.4 against 1.8 us) and the next kernel can only start once
// it is complete.  This kernel waits for what came before the call in the stream, then at once lets the next kernel
// start: stage 1 sets up, loads and multiplies while the zeros are written, and waits for them only before its first
// reduction into K', V'.  B = 1, H = 2, N = 1024: memset + gap 3.8 us before stage 1;
// this kernel takes 1.3 us, and stage 1 is under way before it ends.
#pragma once

#include <cuda_runtime.h>

#include "tc_common.cuh"

namespace flurka {

struct ClearRanges {
  uint4* ptr[2];           // 16-byte aligned
  size_t count[2];         // 16-byte words
};

__global__ void __launch_bounds__(256)
clear_ranges(const ClearRanges r) {
  tc::grid_dependency_wait();
  tc::grid_launch_dependents();
  const size_t first = (size_t)blockIdx.x * 256 + threadIdx.x, step = (size_t)gridDim.x * 256;
#pragma unroll
  for (int i = 0; i < 2; ++i)
    for (size_t w = first; w < r.count[i]; w += step) r.ptr[i][w] = make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace flurka
