// Copies of E, F (and of dE, dF back) between their dense [rows][N] form and rows whose pitch is a multiple of
// 16 bytes, for sequence lengths that are no multiple of 8.
//
// TMA wants row pitches that are multiples of 16 bytes; of the operands only E, F ([k][N], the contraction
// E K of arxiv 2306.15799, Section 2.1 / Eq. (2), runs along their rows) have a pitch of N elements.  They
// are shared by all heads, so a copy moves 2 k N elements against the 2 B H d N of K and V; the tensor maps
// keep the true extent N, so the padding is never read.  Bound by memory traffic; measured at B H = 16, N = 6001,
// d = 64, k = m = 256: the forward 449 us on the CUDA-core kernels, 60 on tensor cores, of which the copy is 4.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "tc_common.cuh"

namespace flurka {

// Eight bf16 from src[at .. at + 7], `at` not aligned: the two 16-byte pieces they lie in, shifted into place.
// `total`: elements of src; a piece that would reach past it is read element by element.
__device__ __forceinline__ uint4 load8_unaligned(const uint16_t* __restrict__ src, long long at, long long total, int live) {
  const long long a0 = at & ~7ll;
  if (a0 + 16 <= total) {
    const uint4 lo = *reinterpret_cast<const uint4*>(src + a0), hi = *reinterpret_cast<const uint4*>(src + a0 + 8);
    uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    const int s = (int)(at - a0);
    if (s & 4) {
#pragma unroll
      for (int i = 0; i < 6; ++i) w[i] = w[i + 2];
    }
    if (s & 2) {
#pragma unroll
      for (int i = 0; i < 5; ++i) w[i] = w[i + 1];
    }
    if (s & 1) {
#pragma unroll
      for (int i = 0; i < 4; ++i) w[i] = __byte_perm(w[i], w[i + 1], 0x5432);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
  uint32_t v[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) v[e] = e < live ? src[at + e] : 0;
  return make_uint4(v[0] | (v[1] << 16), v[2] | (v[3] << 16), v[4] | (v[5] << 16), v[6] | (v[7] << 16));
}

// dst0 / dst1 [rows][pitch] <- src0 / src1 [rows][N]; one thread per 16 bytes of a padded row.
__global__ void __launch_bounds__(256)
pad_rows(const uint16_t* __restrict__ src0, const uint16_t* __restrict__ src1, uint16_t* __restrict__ dst0,
         uint16_t* __restrict__ dst1, int rows, int N, int pitch) {
  tc::grid_launch_dependents();
  tc::grid_dependency_wait();       // (so that its own completion says that everything before it is complete)
  const uint16_t* __restrict__ src = blockIdx.z ? src1 : src0;
  uint16_t* __restrict__ dst = blockIdx.z ? dst1 : dst0;
  const int c = (blockIdx.x * 256 + threadIdx.x) * 8;
  if (c >= N) return;
  const long long total = (long long)rows * N;
  for (int r = blockIdx.y; r < rows; r += gridDim.y)
    *reinterpret_cast<uint4*>(dst + (size_t)r * pitch + c) = load8_unaligned(src, (long long)r * N + c, total, N - c);
}

// dst0 / dst1 [rows][N] <- src0 / src1 [rows][pitch]; one thread per 16 bytes of the dense result, which lie in
// one row or run over into the next (N >= 8).
__global__ void __launch_bounds__(256)
unpad_rows(const uint16_t* __restrict__ src0, const uint16_t* __restrict__ src1, uint16_t* __restrict__ dst0,
           uint16_t* __restrict__ dst1, int rows, int N, int pitch) {
  const uint16_t* __restrict__ src = blockIdx.z ? src1 : src0;
  uint16_t* __restrict__ dst = blockIdx.z ? dst1 : dst0;
  const long long total = (long long)rows * N;
  for (long long at = ((long long)blockIdx.x * 256 + threadIdx.x) * 8; at < total; at += (long long)gridDim.x * 2048) {
    long long r = at / N;
    int c = (int)(at - r * N);
    uint32_t v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      v[e] = at + e < total ? src[(size_t)r * pitch + c] : 0;
      if (++c == N) { c = 0; ++r; }
    }
    if (at + 8 <= total) {
      *reinterpret_cast<uint4*>(dst + at) =
          make_uint4(v[0] | (v[1] << 16), v[2] | (v[3] << 16), v[4] | (v[5] << 16), v[6] | (v[7] << 16));
    } else {
      for (int e = 0; at + e < total; ++e) dst[at + e] = (uint16_t)v[e];
    }
  }
}

}  // namespace flurka
