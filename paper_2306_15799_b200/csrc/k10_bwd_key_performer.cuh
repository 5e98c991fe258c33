// Backward of the key side on tensor cores for PERFORMER where its arithmetic keeps 24 bits: d = 128, and ragged lengths
// (k a multiple of 64 up to 512, p = 64 .. 256).  The formulas are those of k6_bwd_key_side.cuh, which rounds A and dL to bf16.
//
// A CTA owns 128 projected keys of a head and walks the features 64 at a time with a key per lane: L = K' W^T and T = V' da^T
// have a feature per column, so that A and dL go back into TMEM as A operands of dV' += A da and dK' += dL W, and what belongs
// to a key (d = 128: |k'|^2 / 2; the sum of its dL) stays with the two threads that share it.
// Everything but W (bf16, exact) is three bf16 terms, fp32's 24 bits, and a product of two such is the six pairs of terms down to
// 2^-24.  With d = 128 shared memory holds two terms of V' and TMEM the third (T's A operand may lie in either).
// What bounds it is the chain of a block of features: L, exponentials, two products; da is converted under L's products, T formed
// under the exponentials, dV' under what is done with T.  us per launch, the CUDA-core kernel / two terms of everything but K' / this: 16
// heads, d = 128, k = 512, m = 256 104 / 31.9 / 36.7; 8 heads, d = 64, k = m = 256 29 / 18.2 / 19.0.
#pragma once

#include <cuda_bf16.h>

#include "k2_key_side.cuh"
#include "k6_bwd_key_side.cuh"
#include "tc_common.cuh"

namespace flurka {

constexpr int kK10Threads = 256, kK10Feats = 64;
template <int kD> struct K10Shape {
  static constexpr uint32_t kBlocks = kD / 64;               // blocks of 64 columns
  static constexpr uint32_t kVTerms = kD == 64 ? 3 : 2;      // of V' in shared memory
  static constexpr uint32_t kVBlock = kVTerms * 16384, kABlock = 3 * 8192;
  // shared memory: per block of columns the terms of K' and V' ([128 x 64]), W and the terms of da ([64 x 64])
  static constexpr uint32_t k3 = 0, v = kBlocks * 49152, w = v + kBlocks * kVBlock, da = w + kBlocks * 8192,
                            be = da + kBlocks * kABlock,     // b_i, e_i of the block's features
                            nrm = be + 512,                  // |k'_j|^2 / 2: d = 64 as an operand [128 x 16] of L, and [64 x 16] of ones
                            sum = be,                        // at the end: [2][128] sums of dL
                            bars = nrm + (kD == 64 ? 6144 : 512);
  static constexpr int bytes = (int)bars + 64 + 1024;
  // TMEM columns: L, then A; T, then dL (a thread's 32 columns become 16 of each of two terms); the third terms of A and of dL;
  // d = 128: that of V'; dV'; dK'
  static constexpr uint32_t kColT = 64, kColA3 = 128, kColDL3 = 160, kColV3 = 192, kColDV = 256, kColDK = 256 + kD, kCols = 512;
};

template <int kD>
__global__ void __launch_bounds__(kK10Threads, 1)
k10_bwd_key_performer(const __grid_constant__ CUtensorMap tmW, const K6Params prm) {
  using namespace tc;
  using L = K10Shape<kD>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t bar_w = base + L::bars, bar_l = bar_w + 8, bar_t = bar_w + 16, bar_o = bar_w + 24, tmem_slot = bar_w + 32;
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_shared;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int k = prm.k, p = prm.p, nkc = (k + 127) >> 7;
  const int head = blockIdx.x / nkc, j0 = blockIdx.x % nkc * 128, keys = min(128, k - j0);     // 64 or 128 live keys
  if (tid == 0) {
    abort_flag = 0;
    mbar_init(bar_w, 1);
    mbar_init(bar_l, 1);
    mbar_init(bar_t, 1);
    mbar_init(bar_o, 1);
    fence_mbar_init();
  }
  auto load_w = [&](int i0) {
    mbar_arrive_expect_tx(bar_w, (uint32_t)(kK10Feats * kD * 2));
    for (uint32_t cb = 0; cb < L::kBlocks; ++cb) tma_load_2d(base + L::w + cb * 8192u, &tmW, bar_w, cb * 64, i0);
  };
  if (tid == 0) load_w(0);                                   // (an input: nothing to wait for)
  if (warp == 0) {
    tmem_alloc(tmem_slot, L::kCols);
    tmem_relinquish();
  }
  grid_dependency_wait();
  // ---- all of the CTA's K', V' and the first block's da are in flight before any of them is converted
  constexpr int kLpr = kD / 4, kPer = 128 * kLpr / kK10Threads, kPerA = kK10Feats * kLpr / kK10Threads;
  constexpr int kStep = kK10Threads / kLpr;                  // rows between a thread's values
  const int r0 = tid / kLpr, ccol = tid % kLpr * 4;
  const float* __restrict__ dah = prm.da + ((size_t)head * p + r0) * kD + ccol;
  float4 xd[kPerA], y[kPer];
  float xbe = 0.f;                                           // b_i (threads 0..63) or e_i (64..127)
  auto load_da = [&](int i0) {
#pragma unroll
    for (int u = 0; u < kPerA; ++u) xd[u] = __ldcg(reinterpret_cast<const float4*>(dah + (size_t)(i0 + u * kStep) * kD));
    if (tid < 128) xbe = __ldcg((tid < 64 ? prm.weight : prm.ei) + (size_t)head * p + i0 + (tid & 63));
  };
  {
    const float* Kp = prm.kpvp + ((size_t)head * k + j0 + r0) * kD + ccol;
    const float* Vp = Kp + (size_t)prm.BH * k * kD;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 x[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      x[u] = r0 + u * kStep < keys ? __ldcg(reinterpret_cast<const float4*>(Kp + (size_t)u * kStep * kD)) : zero;
      y[u] = r0 + u * kStep < keys ? __ldcg(reinterpret_cast<const float4*>(Vp + (size_t)u * kStep * kD)) : zero;
    }
    load_da(0);
    if (kD == 64 && tid < 128)                               // (element (r, c) at (r/8)*256 + (c/8)*128 + (r%8)*16 + (c%8)*2 bytes)
      reinterpret_cast<uint4*>(base_ptr + L::nrm + 4096)[tid] = (tid & 8) ? make_uint4(0u, 0u, 0u, 0u) : make_uint4(0x3f803f80u, 0x3f80u, 0u, 0u);
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int r = r0 + u * kStep;
      k6_split_store<3>(base + L::k3 + (uint32_t)(ccol >> 6) * 49152u, r, ccol & 63, x[u]);
      // as the forward's key side adds them up, rounding for rounding: its error then cancels between L_ij and b_i.  d = 64: so does
      // that of L, which is formed from the same operands in the same order (d = 128 has no room for these, and its P, c, rounded
      // to bf16, cost more)
      float sq = fmaf(x[u].x, x[u].x, fmaf(x[u].y, x[u].y, fmaf(x[u].z, x[u].z, x[u].w * x[u].w)));
#pragma unroll
      for (int o = kLpr / 2; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
      if (ccol == 0) {
        if constexpr (kD == 64) {
          const float n0 = -0.5f * sq;
          const uint32_t t0 = k6_bf16x2(n0, 0.f);
          const float n1 = n0 - __uint_as_float(t0 << 16);
          const uint32_t t1 = k6_bf16x2(n1, 0.f);
          uint4* op = reinterpret_cast<uint4*>(base_ptr + L::nrm + (r >> 3) * 256 + (r & 7) * 16);
          op[0] = make_uint4(t0 | t1 << 16, k6_bf16x2(n1 - __uint_as_float(t1 << 16), 0.f), 0u, 0u);
          op[8] = make_uint4(0u, 0u, 0u, 0u);
        } else {
          reinterpret_cast<float*>(base_ptr + L::nrm)[r] = 0.5f * sq;
        }
      }
    }
  }
  fence_proxy_async_smem();
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  if (tid == 0) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(tmem_slot));
    tmem_base_shared = v;
  }
  __syncthreads();
  const uint32_t tmem = tmem_base_shared;
  // two threads per key, 32 of a block's 64 features each
  const int q4 = warp & 3, h = warp >> 2, row = q4 * 32 + lane;
  const uint32_t lane_base = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)h * 32u;
  const bool live = row < keys;
  const float nj = kD == 64 ? 0.f : reinterpret_cast<const float*>(base_ptr + L::nrm)[row];
  const float* be = reinterpret_cast<const float*>(base_ptr + L::be) + h * 32;
  float s_j = 0.f;
  bool ok = true;
  uint32_t phase = 0;
  constexpr uint32_t idescT = make_idesc(kFmtBF16, 0, 0, 128, kK10Feats);     // L, T: both operands K-major along d
  constexpr uint32_t idescO = make_idesc(kFmtBF16, 0, 1, 128, kD);            // dV', dK'
  // the pairs of terms (a term's weight is 2^-8 of the one before); what is left out is below 2^-24
  constexpr uint32_t kTa[6] = {0, 0, 1, 1, 0, 2}, kTb[6] = {0, 1, 0, 1, 2, 0};
  // 32 values -> two terms over the 32 columns they came from, the third into 16 columns at `col3`
  auto put_terms = [&](uint32_t col, uint32_t col3, const float (&x)[32]) {
    uint32_t t0[16], t1[16], t2[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      float a = x[2 * e], b = x[2 * e + 1];
      t0[e] = k6_bf16x2(a, b);
      a -= __uint_as_float(t0[e] << 16); b -= __uint_as_float(t0[e] & 0xffff0000u);
      t1[e] = k6_bf16x2(a, b);
      a -= __uint_as_float(t1[e] << 16); b -= __uint_as_float(t1[e] & 0xffff0000u);
      t2[e] = k6_bf16x2(a, b);
    }
    tmem_st16(lane_base + col, t0);
    tmem_st16(lane_base + col + 16, t1);
    tmem_st16(lane_base + col3 - (uint32_t)h * 16u, t2);
  };
  // the columns of a term of 16 features of A or dL: (column of the values, of their third term) -> step `half` of 2
  auto term_at = [&](uint32_t col, uint32_t col3, uint32_t t, uint32_t half) {
    return tmem + (t == 2 ? col3 + half * 16u : col + half * 32u + t * 16u);
  };

  for (int i0 = 0; i0 < p; i0 += kK10Feats, phase ^= 1) {
    // (the products of the block before, which read W, da, A and dL, are complete: waited for below)
    if (warp == 0) {
      const bool landed = mbar_wait(bar_w, phase, prm.status, &abort_flag);
      ok = __all_sync(0xffffffffu, ok && landed);
      if (ok && elect_one()) {
        tcgen05_fence_after();
#pragma unroll
        for (uint32_t t = 0; t < 3; ++t)
          for (uint32_t cb = 0; cb < L::kBlocks; ++cb)
            mma_ss_x4(tmem, make_sdesc(base + L::k3 + cb * 49152u + t * 16384u, 16, 1024, kSwizzle128),
                      make_sdesc(base + L::w + cb * 8192u, 16, 1024, kSwizzle128), 2, 2, idescT, t > 0 || cb > 0 ? 1u : 0u);
        if (kD == 64)
          mma_ss(tmem, make_sdesc(base + L::nrm, 128, 256, kSwizzleNone), make_sdesc(base + L::nrm + 4096, 128, 256, kSwizzleNone), idescT, 1u);
        mma_commit(bar_l);
      }
      __syncwarp();
    }
    // ---- V' (once) and the block's da -> bf16 terms, under those products
    if (i0 == 0) {
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const float4 rest = k6_split_store<L::kVTerms>(base + L::v + (uint32_t)(ccol >> 6) * L::kVBlock, r0 + u * kStep, ccol & 63, y[u]);
        // d = 128: the third term goes to its rows' threads through the place of da
        if (L::kVTerms == 2) k6_split_store<1>(base + L::da + (uint32_t)(ccol >> 6) * 16384u, r0 + u * kStep, ccol & 63, rest);
      }
      if constexpr (L::kVTerms == 2) {
        __syncthreads();
        const uint32_t at = base + L::da + (uint32_t)h * 16384u + (uint32_t)row * 128u;
#pragma unroll
        for (uint32_t c = 0; c < 8; c += 2) {
          uint32_t low[8];
#pragma unroll
          for (uint32_t e = 0; e < 2; ++e)
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(low[4 * e]), "=r"(low[4 * e + 1]), "=r"(low[4 * e + 2]),
                         "=r"(low[4 * e + 3]) : "r"(at + (((c + e) ^ ((uint32_t)row & 7u)) << 4)) : "memory");
          tmem_st8(lane_base + L::kColV3 + c * 4, low);
        }
        tmem_wait_st();
        tcgen05_fence_before();
        __syncthreads();
      }
    }
#pragma unroll
    for (int u = 0; u < kPerA; ++u)
      k6_split_store<3, 8192>(base + L::da + (uint32_t)(ccol >> 6) * L::kABlock, r0 + u * kStep, ccol & 63, xd[u]);
    if (tid < 128) reinterpret_cast<float*>(base_ptr + L::be)[tid] = xbe;
    if (i0 + kK10Feats < p) load_da(i0 + kK10Feats);
    fence_proxy_async_smem();
    ok = __syncthreads_and(ok) != 0;
    if (!ok) break;
    if (warp == 0 && elect_one()) {
      tcgen05_fence_after();
#pragma unroll
      for (int t = 0; t < 6; ++t)
        for (uint32_t cb = 0; cb < L::kBlocks; ++cb) {
          const uint64_t bd = make_sdesc(base + L::da + cb * L::kABlock + kTb[t] * 8192u, 16, 1024, kSwizzle128);
          if (kTa[t] >= L::kVTerms)
            mma_ts_x4(tmem + L::kColT, tmem + L::kColV3 + cb * 32u, bd, 2, idescT, 1u);
          else
            mma_ss_x4(tmem + L::kColT, make_sdesc(base + L::v + cb * L::kVBlock + kTa[t] * 16384u, 16, 1024, kSwizzle128), bd, 2, 2,
                      idescT, t > 0 || cb > 0 ? 1u : 0u);
        }
      mma_commit(bar_t);
    }
    __syncwarp();
    float A[32];
    ok = mbar_wait(bar_l, phase, prm.status, &abort_flag);
    tcgen05_fence_after();
    {
      uint32_t r[32];
      tmem_ld32(lane_base, r);
      tmem_wait_ld(r);
#pragma unroll
      for (int e = 0; e < 32; ++e) A[e] = expf((kD == 64 ? __uint_as_float(r[e]) : __uint_as_float(r[e]) - nj) - be[e]);      // b_i = log sum_j exp(L_ij): A <= 1
      put_terms(0, L::kColA3, A);
    }
    tmem_wait_st();
    tcgen05_fence_before();
    ok = __syncthreads_and(ok) != 0;
    if (!ok) break;
    if (warp == 0 && elect_one()) {
      // dV' comes behind T, under what is done with T.  (The rows of da and of W are the contraction, MN-major: 16 features = 2048 B
      // per step.)
      tcgen05_fence_after();
#pragma unroll
      for (int t = 0; t < 6; ++t)
#pragma unroll
        for (uint32_t half = 0; half < 2; ++half)
          mma_ts_x2(tmem + L::kColDV, term_at(0, L::kColA3, kTa[t], half),
                    make_sdesc(base + L::da + kTb[t] * 8192u + half * 4096u, L::kABlock, 1024, kSwizzle128), 128, idescO,
                    i0 > 0 || t > 0 || half > 0 ? 1u : 0u);
    }
    __syncwarp();
    ok = mbar_wait(bar_t, phase, prm.status, &abort_flag) && ok;
    tcgen05_fence_after();
    {
      uint32_t r[32];
      tmem_ld32(lane_base + L::kColT, r);
      tmem_wait_ld(r);
#pragma unroll
      for (int e = 0; e < 32; ++e) {
        A[e] *= __uint_as_float(r[e]) + be[64 + e];
        s_j += A[e];
      }
      put_terms(L::kColT, L::kColDL3, A);
    }
    tmem_wait_st();
    tcgen05_fence_before();
    ok = __syncthreads_and(ok) != 0;
    if (!ok) break;
    if (warp == 0 && elect_one()) {
      tcgen05_fence_after();
#pragma unroll
      for (uint32_t t = 0; t < 3; ++t)
#pragma unroll
        for (uint32_t half = 0; half < 2; ++half)
          mma_ts_x2(tmem + L::kColDK, term_at(L::kColT, L::kColDL3, t, half),
                    make_sdesc(base + L::w + half * 4096u, 8192, 1024, kSwizzle128), 128, idescO,
                    i0 > 0 || t > 0 || half > 0 ? 1u : 0u);
      mma_commit(bar_o);
    }
    __syncwarp();
    ok = mbar_wait(bar_o, phase, prm.status, &abort_flag);
    if (tid == 0 && ok && i0 + kK10Feats < p) load_w(i0 + kK10Feats);
  }
  ok = __syncthreads_and(ok) != 0;

  if (tid == 0) grid_launch_dependents();
  // ---- dk'_j = (dL W)_j - k'_j s_j and dv'_j: two threads per key, half of the columns each
  float* sums = reinterpret_cast<float*>(base_ptr + L::sum);
  sums[h * 128 + row] = s_j;
  __syncthreads();
  if (ok) {
    tcgen05_fence_after();
    s_j = sums[row] + sums[128 + row];
    const int c0 = h * (kD / 2);
    const uint32_t cols = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)c0;
    const size_t hd = (size_t)prm.BH * kD, term = (size_t)k * hd;
    __nv_bfloat16* dst = prm.split + (size_t)(j0 + (live ? row : 0)) * hd + (size_t)head * kD + c0;
    const float* kr = prm.kpvp + ((size_t)head * k + j0 + (live ? row : 0)) * kD + c0;
#pragma unroll 1
    for (int c = 0; c < kD / 2; c += 32) {
      float4 kv[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) kv[e] = __ldcg(reinterpret_cast<const float4*>(kr + c) + e);
      uint32_t r1[32], r2[32];
      tmem_ld32(cols + L::kColDK + c, r1);
      tmem_ld32(cols + L::kColDV + c, r2);
      tmem_wait_ld(r1);
      tmem_wait_ld(r2);
      if (live) {
        float x[32];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          x[4 * e] = fmaf(-kv[e].x, s_j, __uint_as_float(r1[4 * e]));
          x[4 * e + 1] = fmaf(-kv[e].y, s_j, __uint_as_float(r1[4 * e + 1]));
          x[4 * e + 2] = fmaf(-kv[e].z, s_j, __uint_as_float(r1[4 * e + 2]));
          x[4 * e + 3] = fmaf(-kv[e].w, s_j, __uint_as_float(r1[4 * e + 3]));
        }
        k2_store_split(dst + c, term, x);
#pragma unroll
        for (int e = 0; e < 32; ++e) x[e] = __uint_as_float(r2[e]);
        k2_store_split(dst + 2 * term + c, term, x);
      }
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, L::kCols);
}

}  // namespace flurka
