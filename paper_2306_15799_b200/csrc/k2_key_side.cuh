// Stage 2 on tensor cores: the key-side feature map and the two key-side contractions
// (arxiv 2306.15799, Eq. (2): phi(K')^T V' and, for the normaliser of Appendix D, phi(K')^T 1),
// kept per feature in the log domain:
//
//   PERFORMER   L_ij = w_i . k'_j - |k'_j|^2 / 2          (rows i = features, columns j = projected keys)
//               b_i  = log sum_j exp(L_ij),  a_i = sum_j softmax_j(L_i.) v'_j
//   RNN         f_ij = elu(k'_ji) + 1,  z_i = sum_j f_ij,  a_i = sum_j f_ij v'_j / z_i
//
// The work is small (2 k m d + 2 k d m FLOP and k m exponentials per head); what counts is the length of one CTA's
// chain of phases.  A CTA owns 128 features of one head and walks the keys in blocks of 16384 / d (256 or 128).  K'
// and V' are fp32 in stage 1's workspace: all sixteen warps load a whole block straight into registers (all its
// loads in flight at once) and split it so that the tensor-core products are fp32-accurate: K' = hi + mid + lo
// (three bf16 terms, exact to 24 bits) against the exact bf16 W, -|k'|^2/2 as three bf16 terms in one extra 16-wide
// contraction step, V' = hi + lo in fp16; V' is converted while the tensor core works on L.  PERFORMER: four threads
// share a feature's row of L, each holds its quarter in registers between the maximum and the exponentials (one TMEM
// read), writes fp16 weights back to TMEM and sums the rounded values, so the dominant term cancels exactly in a_i; the
// second product reads the weights from TMEM.  Several blocks: running maximum, accumulator in registers.  RNN: the
// weights are the fp16 f tile as it lies ([key][feature], the MN-major A operand), and z_i comes from the same tile
// times a column of ones.
// kTerms serves sequence lengths that are no multiple of 8: weights and V' are two bf16 terms each, 16 to 17 bits (the low
// weights where L was read from; RNN: a second f tile), three products instead of two (low x low is 2^-18), and a leaves as the
// two bf16 terms that the query side reads.  PERFORMER in the backward pass: three terms and six products, 24 bits, and a as
// three terms, for with weights near 1 a gradient dL is a difference of nearly equal da.v' and da.a (one head, N = 30001,
// k = m = 64: dK 2.9e-2 off with two terms, 3.7e-3 with three, 2.8e-3 on CUDA cores; the forward does not notice, and takes 0.8 us more).
// bf16 has fp32's range, so V' may be as large as it may be on CUDA cores.
// One block of 256 keys takes about 10 k cycles; the earlier form (eight warps, a staging copy and a block barrier per
// 128 keys, one thread per row) took 17 us after stage 1's end at B H = 64, k = m = 256, d = 64, this one 9.
//
// With few heads and several blocks the blocks are divided over `nsplit` CTAs per (head, feature tile): each keeps its
// own maximum, sum and unnormalised accumulator, writes them to a scratch area, and the CTA that arrives
// last at the tile's counter merges them (log-sum-exp over the partial maxima) and writes a_i, b_i.
// Nobody waits for anybody: the last arrival finds every partial result already in memory.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "tc_common.cuh"

namespace flurka {

struct K2Params {
  int d, k, p, BH;          // p = feature dimension (m, or d for RNN)
  int ftiles;               // ceil(p / 128)
  const float* kpvp;        // [2][BH][k][d] fp32
  float* weight;            // [BH][p]      b_i (PERFORMER) or z_i (RNN)
  __half* aT16;             // [BH][d][p]   a^T, or NULL
  float* a32;               // [BH][p][d]   a in fp32 as well (the backward pass wants it), or NULL
  __nv_bfloat16* abf;       // [BH][abf_terms][p][d]  a as two bf16 terms (the backward pass; kTerms = 3: three), or NULL
  int* status;
  int nsplit;               // CTAs per (head, feature tile) along the keys (1..4; PERFORMER only)
  float* part;              // nsplit > 1: [BH * ftiles][nsplit][d + 2][128]  max, sum, accumulator columns
  int* counters;            // nsplit > 1: [BH * ftiles], zero on entry, zero again on exit
};

constexpr int kK2Threads = 512;
constexpr int kK2BlockElems = 16384;           // keys per block x d
// shared memory: W tile (<= 32 KB; kTerms = 3: 16) | ones 4 KB | -|k'|^2/2 tile 8 KB | three 32 KB terms of K' (RNN: f tile, zero
// slab) | two or three 32 KB terms of V' | barriers
template <int kTerms> struct K2Smem {
  static constexpr uint32_t ones = kTerms == 3 ? 16384 : 32768, nrm = ones + 4096, k3 = nrm + 8192, v = k3 + 3 * 32768;
  static constexpr uint32_t bars = v + (kTerms == 3 ? 3 : 2) * 32768;
  static constexpr int bytes = (int)bars + 64 + 1024;
};
// TMEM columns of the a accumulator and of z (RNN) or the third terms of the weights (kTerms = 3)
constexpr uint32_t kK2OCol = 256, kK2ZCol = 384;

// two floats -> {lo: bf16(a), hi: bf16(b)} with one rounding instruction
__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %2, %1;" : "=r"(r) : "f"(a), "f"(b));
  return r;
}

__device__ __forceinline__ float k2_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void st_shared_v2(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
// kCols consecutive values of a feature's a, as two bf16 terms `term` elements apart, or three (kInf: an infinite one has no low term)
template <int kCols, bool kInf = false>
__device__ __forceinline__ void k2_store_split(__nv_bfloat16* dst, size_t term, const float (&v)[kCols], bool third = false) {
#pragma unroll
  for (int c = 0; c < kCols; c += 8) {
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float x = v[c + 2 * e], y = v[c + 2 * e + 1];
      hi[e] = pack_bf16x2(x, y);
      float rx = x - __uint_as_float(hi[e] << 16), ry = y - __uint_as_float(hi[e] & 0xffff0000u);
      if (kInf) {
        rx = isnan(rx) ? 0.f : rx;
        ry = isnan(ry) ? 0.f : ry;
      }
      lo[e] = pack_bf16x2(rx, ry);
    }
    *reinterpret_cast<uint4*>(dst + c) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(dst + term + c) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    if (third) {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        lo[e] = pack_bf16x2((v[c + 2 * e] - __uint_as_float(hi[e] << 16)) - __uint_as_float(lo[e] << 16),
                            (v[c + 2 * e + 1] - __uint_as_float(hi[e] & 0xffff0000u)) - __uint_as_float(lo[e] & 0xffff0000u));
      *reinterpret_cast<uint4*>(dst + 2 * term + c) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
  }
}
// one bf16 term of four values into shared memory, and what it leaves.  Packed conversions: one instruction rounds two values;
// a bf16 is the top half of an fp32
__device__ __forceinline__ void k2_put_term(uint32_t addr, float4& v) {
  const uint32_t h0 = pack_bf16x2(v.x, v.y), h1 = pack_bf16x2(v.z, v.w);
  st_shared_v2(addr, h0, h1);
  v.x -= __uint_as_float(h0 << 16); v.y -= __uint_as_float(h0 & 0xffff0000u);
  v.z -= __uint_as_float(h1 << 16); v.w -= __uint_as_float(h1 & 0xffff0000u);
}
__device__ __forceinline__ uint32_t half2_bits(__half2 h) { return *reinterpret_cast<const uint32_t*>(&h); }

// kTerms: weights and V' as so many bf16 terms each (see the header); 0: fp16 weights, V' as two fp16 terms
template <bool kPerformer, int kD, int kTerms = 0>
__global__ void __launch_bounds__(kK2Threads, 1)
k2_key_side(const __grid_constant__ CUtensorMap tmW, const K2Params prm) {
  using namespace tc;
  using L = K2Smem<kTerms>;
  static_assert(kTerms < 3 || (kPerformer && kD == 64), "room for the third terms");
  constexpr bool kSplit = kTerms > 0;
  constexpr int kATerms = kTerms == 3 ? 3 : 2;
  constexpr int KB = kK2BlockElems / kD;                  // keys per block
  constexpr int kq = kD / 64;                             // 64-wide blocks of the head dimension
  constexpr uint32_t kSlab = KB * 128;                    // bytes of one 64-column slab of a term
  constexpr int kLpr = kD / 4;                            // lanes per fp32 row (float4 each): 16 or 32
  constexpr int kRpi = 32 / kLpr;                         // rows per warp instruction
  constexpr int kIters = KB / (16 * kRpi);                // 8
  constexpr int kKeysPer = KB / 4;                        // keys of a row's thread: 64 or 32
  constexpr int kColsPer = kD / 4;                        // accumulator columns of a row's thread: 16 or 32
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t bar_w = base + L::bars, bar_l = bar_w + 8, bar_o = bar_w + 16, tmem_slot = bar_w + 24;
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_shared;
  __shared__ float red_max[4][128], red_sum[4][128];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  const int k = prm.k, p = prm.p;
  const int nsplit = prm.nsplit;
  const int sp = blockIdx.x % nsplit;                         // which part of the keys
  const int unit = blockIdx.x / nsplit;                       // (head, feature tile)
  const int head = unit / prm.ftiles;
  const int i0 = (unit % prm.ftiles) * 128;                   // first feature of this CTA
  const float* __restrict__ Kp = prm.kpvp + (size_t)head * k * kD;
  const float* __restrict__ Vp = prm.kpvp + ((size_t)prm.BH + head) * (size_t)k * kD;
  const int nblocks = (k + KB - 1) / KB;
  const int b_begin = (sp * nblocks) / nsplit, b_end = ((sp + 1) * nblocks) / nsplit;

  if (tid == 0) {
    abort_flag = 0;
    mbar_init(bar_w, 1);
    mbar_init(bar_l, 1);
    mbar_init(bar_o, 1);
    fence_mbar_init();
    if (kPerformer) {
      prefetch_tmap(&tmW);
      mbar_arrive_expect_tx(bar_w, (uint32_t)(128 * kD * 2));
      for (int kb = 0; kb < kq; ++kb) tma_load_2d(base + kb * 16384, &tmW, bar_w, kb * 64, i0);
    }
  }
  if (warp == 14) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  if (kPerformer) {
    // A operand of the bias step: [128 x 16] bf16, columns 0..2 = 1, no swizzle
    // (element (r, c) at (r/8)*256 + (c/8)*128 + (r%8)*16 + (c%8)*2 bytes)
    uint32_t* ones = reinterpret_cast<uint32_t*>(base_ptr + L::ones);
    for (int e = tid; e < 1024; e += kK2Threads) {
      const int c = (e & 3) + ((e >> 5) & 1) * 4;            // which pair of columns
      ones[e] = c == 0 ? 0x3f803f80u : (c == 1 ? 0x00003f80u : 0u);
    }
  } else {
    // B operand of z: [16 x 64 keys] fp16, K-major, no swizzle: row 0 all ones, (c, n) at (c/8)*1024 + (n/8)*128 + (c%8)*16 + (n%8)*2
    uint32_t* ones = reinterpret_cast<uint32_t*>(base_ptr + L::ones);
    if (tid < 512) ones[tid] = (tid < 256 && (tid & 31) < 4) ? (kSplit ? 0x3f803f80u : 0x3c003c00u) : 0u;
    // d = 64: features 64..127 of the f tile (its second slab) do not exist (kSplit: they are whatever lies there, and not read out)
    if (kD == 64 && !kSplit) {
      uint4* z4 = reinterpret_cast<uint4*>(base_ptr + L::k3 + kSlab);
      for (int e = tid; e < (int)(kSlab / 16); e += kK2Threads) z4[e] = make_uint4(0u, 0u, 0u, 0u);
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
  // everything above (and the W tile on its way) is independent of stage 1
  grid_dependency_wait();

  // conversion geometry: a warp instruction reads whole rows (kLpr lanes x float4 per row); a lane converts four
  // consecutive columns of kIters rows, 16 kRpi apart
  const int ccol = (lane % kLpr) * 4;                         // this lane's first column
  const int crow = warp * kRpi + lane / kLpr;                 // this lane's row in iteration 0
  const uint32_t coff = (uint32_t)(ccol >> 6) * kSlab + (uint32_t)((ccol & 7) >> 2) * 8;
  const int cchunk = (ccol & 63) >> 3;                        // 16-byte chunk of the 128-byte row before the swizzle
  // row geometry: four threads per feature (TMEM lane), quarter qd of the keys and of the accumulator columns each
  const int frow = (warp & 3) * 32 + lane, qd = warp >> 2;
  const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  const float kLog2e = 1.4426950408889634f;
  float run_max = -INFINITY, zsum = 0.f;
  float acc[kColsPer];
#pragma unroll
  for (int c = 0; c < kColsPer; ++c) acc[c] = 0.f;
  bool ok = true;
  uint32_t phase = 0;

  for (int b = b_begin; b < b_end && ok; ++b, phase ^= 1) {
    const int j0 = b * KB, live = min(KB, k - j0);            // keys of the block, a multiple of 64
    // ---- the block's fp32 rows: every load of K' is in flight before the first value is used; V' follows where the
    //      registers are (PERFORMER: once K' is converted, its latency then lies under the first product)
    float4 kx[kIters], vx[kIters];
#pragma unroll
    for (int t = 0; t < kIters; ++t) {
      const int r = crow + t * 16 * kRpi;
      kx[t] = r < live ? __ldcg(reinterpret_cast<const float4*>(Kp + (size_t)(j0 + r) * kD + ccol)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    auto load_values = [&]() {
#pragma unroll
      for (int t = 0; t < kIters; ++t) {
        const int r = crow + t * 16 * kRpi;
        vx[t] = r < live ? __ldcg(reinterpret_cast<const float4*>(Vp + (size_t)(j0 + r) * kD + ccol)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    };
    if (!kPerformer) load_values();
    if (kPerformer) {
      // ---- K' -> three bf16 tiles (K-major, 128-byte swizzle) and -|k'|^2/2
      float sq[kIters];
#pragma unroll
      for (int t = 0; t < kIters; ++t) {
        const int r = crow + t * 16 * kRpi;
        const float x = kx[t].x, y = kx[t].y, z = kx[t].z, w = kx[t].w;
        sq[t] = fmaf(x, x, fmaf(y, y, fmaf(z, z, w * w)));
        const uint32_t off = base + L::k3 + coff + r * 128 + ((cchunk ^ (r & 7)) << 4);
#pragma unroll
        for (int s3 = 0; s3 < 3; ++s3) k2_put_term(off + s3 * 32768, kx[t]);
      }
      load_values();
      // |k'_r|^2 of the eight rows over the lanes that share them, halving the number of rows per lane on the way.  The
      // halves of a row of 128 meet first: with |k'|^2 / 2 in the thousands one ulp of this sum is 1e-4 of a weight,
      // so another tree gives other results (N = 131072, k = 512: 1e-4 to 4e-4 of the output's norm; seven more shuffles than joining them last)
      static_assert(kIters == 8, "eight rows per lane");
      if (kLpr == 32) {
#pragma unroll
        for (int t = 0; t < kIters; ++t) sq[t] += __shfl_xor_sync(0xffffffffu, sq[t], 16);
      }
      float s4[4], s2[2];
      const bool up8 = (lane & 8) != 0, up4 = (lane & 4) != 0, up2 = (lane & 2) != 0;
#pragma unroll
      for (int e = 0; e < 4; ++e) s4[e] = (up8 ? sq[4 + e] : sq[e]) + __shfl_xor_sync(0xffffffffu, up8 ? sq[e] : sq[4 + e], 8);
#pragma unroll
      for (int e = 0; e < 2; ++e) s2[e] = (up4 ? s4[2 + e] : s4[e]) + __shfl_xor_sync(0xffffffffu, up4 ? s4[e] : s4[2 + e], 4);
      float s1 = (up2 ? s2[1] : s2[0]) + __shfl_xor_sync(0xffffffffu, up2 ? s2[0] : s2[1], 2);
      s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
      if ((lane & 1) == 0 && (kLpr == 16 || lane < 16)) {
        // B operand of the bias step: row r, columns 0..2 = three bf16 terms of -|k'_r|^2/2
        const int r = crow + ((up8 ? 4 : 0) + (up4 ? 2 : 0) + (up2 ? 1 : 0)) * 16 * kRpi;
        float bb = -0.5f * s1;
        const __nv_bfloat16 g0 = __float2bfloat16_rn(bb);  bb -= __bfloat162float(g0);
        const __nv_bfloat16 g1 = __float2bfloat16_rn(bb);  bb -= __bfloat162float(g1);
        const __nv_bfloat16 g2 = __float2bfloat16_rn(bb);
        uint4* na = reinterpret_cast<uint4*>(base_ptr + L::nrm + (r >> 3) * 256 + (r & 7) * 16);
        na[0] = make_uint4((uint32_t)__bfloat16_as_ushort(g0) | ((uint32_t)__bfloat16_as_ushort(g1) << 16),
                           (uint32_t)__bfloat16_as_ushort(g2), 0u, 0u);
        na[8] = make_uint4(0u, 0u, 0u, 0u);
      }
      fence_proxy_async_smem();
      bool mine = true;
      if (b == b_begin && warp == 15) mine = mbar_wait(bar_w, 0, prm.status, &abort_flag);
      ok = __syncthreads_and(mine) != 0;
      if (!ok) break;
      if (warp == 15 && elect_one()) {
        tcgen05_fence_after();
        const uint32_t idesc1 = make_idesc(kFmtBF16, 0, 0, 128, (uint32_t)live);
        for (int s3 = 0; s3 < 3; ++s3)
          for (int kb = 0; kb < kq; ++kb) {
            const uint64_t ad = make_sdesc(base + kb * 16384, 16, 1024, kSwizzle128);
            const uint64_t bd = make_sdesc(base + L::k3 + s3 * 32768 + kb * kSlab, 16, 1024, kSwizzle128);
            mma_ss_x4(tmem, ad, bd, 2, 2, idesc1, (s3 > 0 || kb > 0) ? 1u : 0u);
          }
        const uint64_t ad = make_sdesc(base + L::ones, 128, 256, kSwizzleNone);
        const uint64_t bd = make_sdesc(base + L::nrm, 128, 256, kSwizzleNone);
        mma_ss(tmem, ad, bd, idesc1, 1u);
        mma_commit(bar_l);
      }
      __syncwarp();
    } else {
      // ---- RNN: f = elu(k') + 1 as one fp16 tile (kSplit: two bf16 tiles) [key][feature]; keys past the end give zero rows
#pragma unroll
      for (int t = 0; t < kIters; ++t) {
        const int r = crow + t * 16 * kRpi;
        const float keep = r < live ? 1.f : 0.f;
        const float x = kx[t].x, y = kx[t].y, z = kx[t].z, w = kx[t].w;
        const float f0 = keep * (fmaxf(x, 0.f) + __expf(fminf(x, 0.f))), f1 = keep * (fmaxf(y, 0.f) + __expf(fminf(y, 0.f)));
        const float f2 = keep * (fmaxf(z, 0.f) + __expf(fminf(z, 0.f))), f3 = keep * (fmaxf(w, 0.f) + __expf(fminf(w, 0.f)));
        const uint32_t off = base + L::k3 + coff + r * 128 + ((cchunk ^ (r & 7)) << 4);
        if constexpr (kSplit) {
          float4 f = make_float4(f0, f1, f2, f3);
#pragma unroll
          for (int s2 = 0; s2 < 2; ++s2) k2_put_term(off + s2 * 32768, f);
        } else {
          st_shared_v2(off, half2_bits(__floats2half2_rn(f0, f1)), half2_bits(__floats2half2_rn(f2, f3)));
        }
      }
    }
    // ---- V' = hi + lo in fp16 (kSplit: bf16) as the MN-major B operand of the second product, under the first product's MMAs
#pragma unroll
    for (int t = 0; t < kIters; ++t) {
      const int r = crow + t * 16 * kRpi;
      const uint32_t off = base + L::v + coff + r * 128 + ((cchunk ^ (r & 7)) << 4);
      if constexpr (kSplit) {
#pragma unroll
        for (int s3 = 0; s3 < kTerms; ++s3) k2_put_term(off + s3 * 32768, vx[t]);
      } else {
        const __half2 hi0 = __floats2half2_rn(vx[t].x, vx[t].y), hi1 = __floats2half2_rn(vx[t].z, vx[t].w);
        const float2 b0 = __half22float2(hi0), b1 = __half22float2(hi1);
        st_shared_v2(off, half2_bits(hi0), half2_bits(hi1));
        st_shared_v2(off + 32768, half2_bits(__floats2half2_rn(vx[t].x - b0.x, vx[t].y - b0.y)),
                     half2_bits(__floats2half2_rn(vx[t].z - b1.x, vx[t].w - b1.y)));
      }
    }
    fence_proxy_async_smem();

    float rescale = 1.f;
    if (kPerformer) {
      // ---- weights of this thread's quarter of the keys
      bool mine = mbar_wait(bar_l, phase, prm.status, &abort_flag);
      tcgen05_fence_after();
      const bool have = qd * kKeysPer < live;                // (the same for the whole warp)
      uint32_t ra[32], rb[32];
      float mx = -INFINITY;
      if (mine && have) {
        tmem_ld32(lane_base + qd * kKeysPer, ra);
        if (kKeysPer == 64) tmem_ld32(lane_base + qd * kKeysPer + 32, rb);
        tmem_wait_ld(ra);
        if (kKeysPer == 64) tmem_wait_ld(rb);
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
          mx = fmax3(mx, __uint_as_float(ra[e]), __uint_as_float(ra[e + 1]));
          if (kKeysPer == 64) mx = fmax3(mx, __uint_as_float(rb[e]), __uint_as_float(rb[e + 1]));
        }
      }
      red_max[qd][frow] = mx;
      tcgen05_fence_before();
      ok = __syncthreads_and(mine) != 0;                     // every quarter has been read: L may be overwritten
      if (!ok) break;
      tcgen05_fence_after();
      const float new_max = fmaxf(fmax3(red_max[0][frow], red_max[1][frow], red_max[2][frow]), fmaxf(red_max[3][frow], run_max));
      rescale = k2_ex2((run_max - new_max) * kLog2e);        // 0 on the first block
      run_max = new_max;
      const float shift = new_max * kLog2e;
      float part = 0.f;
      if (have) {
        auto weigh = [&](const uint32_t (&r)[32], uint32_t col) {
          if constexpr (kSplit) {
#pragma unroll
            for (int c = 0; c < 16; c += 8) {
              uint32_t t0[8], t1[8];
              [[maybe_unused]] uint32_t t2[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) {
                // (the difference first: the rounding of max * log2 e would go into b_i)
                float w0 = k2_ex2((__uint_as_float(r[2 * (c + e)]) - new_max) * kLog2e);
                float w1 = k2_ex2((__uint_as_float(r[2 * (c + e) + 1]) - new_max) * kLog2e);
                if (kTerms == 3) part += w0 + w1;
                t0[e] = pack_bf16x2(w0, w1);
                const float h0 = __uint_as_float(t0[e] << 16), h1 = __uint_as_float(t0[e] & 0xffff0000u);
                w0 -= h0; w1 -= h1;
                t1[e] = pack_bf16x2(w0, w1);
                const float l0 = __uint_as_float(t1[e] << 16), l1 = __uint_as_float(t1[e] & 0xffff0000u);
                if (kTerms == 2) part += (h0 + l0) + (h1 + l1);
                else t2[e] = pack_bf16x2(w0 - l0, w1 - l1);
              }
              tmem_st8(lane_base + col + c, t0);               // (L has been read by everybody: there is room for two)
              tmem_st8(lane_base + KB / 2 + col + c, t1);
              if (kTerms == 3) tmem_st8(lane_base + kK2ZCol + col + c, t2);
            }
          } else {
            uint32_t h[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const __half2 hh = __floats2half2_rn(k2_ex2(fmaf(__uint_as_float(r[2 * e]), kLog2e, -shift)),
                                                   k2_ex2(fmaf(__uint_as_float(r[2 * e + 1]), kLog2e, -shift)));
              const float2 back = __half22float2(hh);
              part += back.x + back.y;
              h[e] = half2_bits(hh);
            }
            tmem_st16(lane_base + col, h);
          }
        };
        weigh(ra, (uint32_t)(qd * kKeysPer / 2));
        if (kKeysPer == 64) weigh(rb, (uint32_t)(qd * kKeysPer / 2 + 16));
        tmem_wait_st();
      }
      red_sum[qd][frow] = part;
    }
    tcgen05_fence_before();
    __syncthreads();
    if (warp == 15 && elect_one()) {
      // ---- a (+)= weights x V': B has 64-column slabs kSlab apart, 8-key groups 1024 B apart, 2048 B per 16 keys
      tcgen05_fence_after();
      const uint32_t first = (kPerformer || b == b_begin) ? 0u : 1u;
      for (int q4 = 0; q4 < (live >> 6); ++q4) {
        if constexpr (kSplit) {
          // the pairs of terms (a term's weight is 2^-8 of the one before); what is left out is below 2^-16 or 2^-24
          constexpr int kTa[6] = {0, 1, 0, 1, 0, 2}, kTb[6] = {0, 0, 1, 1, 2, 0};
#pragma unroll
          for (int t = 0; t < (kTerms == 3 ? 6 : 3); ++t) {
            const uint64_t bd = make_sdesc(base + L::v + kTb[t] * 32768u + q4 * 8192, kSlab, 1024, kSwizzle128);
            const uint32_t add = (q4 > 0 || t > 0) ? 1u : first;
            if constexpr (kPerformer) {
              const uint32_t at = kTa[t] == 2 ? kK2ZCol : kTa[t] * (KB / 2);
              mma_ts_x4(tmem + kK2OCol, tmem + at + q4 * 32, bd, 128, make_idesc(kFmtBF16, 0, /*B MN-major*/ 1, 128, kD), add);
            } else {
              mma_ss_x4(tmem + kK2OCol, make_sdesc(base + L::k3 + kTa[t] * 32768u + q4 * 8192, kSlab, 1024, kSwizzle128), bd, 128, 128,
                        make_idesc(kFmtBF16, 1, 1, 128, kD), add);
            }
          }
        } else {
          for (int s2 = 0; s2 < 2; ++s2) {
            const uint64_t bd = make_sdesc(base + L::v + s2 * 32768u + q4 * 8192, kSlab, 1024, kSwizzle128);
            const uint32_t add = (q4 > 0 || s2 > 0) ? 1u : first;
            if (kPerformer) {
              mma_ts_x4(tmem + kK2OCol, tmem + q4 * 32, bd, 128, make_idesc(kFmtF16, 0, /*B MN-major*/ 1, 128, kD), add);
            } else {
              const uint64_t ad = make_sdesc(base + L::k3 + q4 * 8192, kSlab, 1024, kSwizzle128);
              mma_ss_x4(tmem + kK2OCol, ad, bd, 128, 128, make_idesc(kFmtF16, 1, 1, 128, kD), add);
            }
          }
        }
        if (!kPerformer) {
          const uint64_t bo = make_sdesc(base + L::ones, 128, 1024, kSwizzleNone);
          for (int t = 0; t < (kSplit ? 2 : 1); ++t)
            mma_ss_x4(tmem + kK2ZCol, make_sdesc(base + L::k3 + t * 32768u + q4 * 8192, kSlab, 1024, kSwizzle128), bo, 128, 16,
                      make_idesc(kSplit ? kFmtBF16 : kFmtF16, 1, 0, 128, 16), q4 > 0 || t > 0 ? 1u : first);
        }
      }
      mma_commit(bar_o);
    }
    __syncwarp();
    const bool mine = mbar_wait(bar_o, phase, prm.status, &abort_flag);
    tcgen05_fence_after();
    if (kPerformer && mine) {
      zsum = fmaf(zsum, rescale, (red_sum[0][frow] + red_sum[1][frow]) + (red_sum[2][frow] + red_sum[3][frow]));
      uint32_t r[32];
      tmem_ld32(lane_base + kK2OCol + qd * kColsPer, r);     // (32 columns; kColsPer of them are this thread's)
      tmem_wait_ld(r);
#pragma unroll
      for (int c = 0; c < kColsPer; ++c) acc[c] = fmaf(acc[c], rescale, __uint_as_float(r[c]));
      tcgen05_fence_before();
    }
    ok = __syncthreads_and(mine) != 0;                       // operands and accumulator are free again
  }
  if (!kPerformer && ok) {
    tcgen05_fence_after();
    uint32_t r[32];
    tmem_ld32(lane_base + kK2ZCol, r);
    tmem_wait_ld(r);
    zsum = __uint_as_float(r[0]);
    tmem_ld32(lane_base + kK2OCol + qd * kColsPer, r);
    tmem_wait_ld(r);
#pragma unroll
    for (int c = 0; c < kColsPer; ++c) acc[c] = __uint_as_float(r[c]);
    if constexpr (kSplit) {
      // an infinite V' has no low term (inf - inf), and times a low weight it may have either sign: such a sum is formed in fp32
      bool odd = false;
#pragma unroll
      for (int c = 0; c < kColsPer; ++c) odd |= isnan(acc[c]);
      if (odd && i0 + frow < p) {
        float sum[kColsPer];
#pragma unroll
        for (int c = 0; c < kColsPer; ++c) sum[c] = 0.f;
#pragma unroll 1
        for (int j = 0; j < k; ++j) {
          const float x = __ldcg(Kp + (size_t)j * kD + i0 + frow), f = fmaxf(x, 0.f) + __expf(fminf(x, 0.f));
#pragma unroll
          for (int c = 0; c < kColsPer; ++c) sum[c] = fmaf(f, __ldcg(Vp + (size_t)j * kD + qd * kColsPer + c), sum[c]);
        }
#pragma unroll
        for (int c = 0; c < kColsPer; ++c) acc[c] = isnan(acc[c]) ? sum[c] : acc[c];
      }
    }
  }

  if (tid == 0) grid_launch_dependents();   // only the write-out (and the merge) is left
  const int feat = i0 + frow;
  // ---- a_i = accumulator / z_i, stored transposed ([d][p], fp16) for stage 3
  if (nsplit == 1) {
    // through shared memory (the K' terms are free by now): a [d][128] fp16 tile, then 16 bytes at a time, so that
    // a^T leaves in whole 128- or 256-byte runs
    if (ok) {
      // (RNN: z_i = 0 where every weight has underflowed; ragged lengths then have a_i = 0, as the CUDA-core kernels do)
      const float inv = 1.f / (kSplit ? fmaxf(zsum, 1.17549435e-38f) : zsum);
      if (qd == 0 && feat < p) prm.weight[(size_t)head * p + feat] = kPerformer ? run_max + (kSplit ? logf(zsum) : __logf(zsum)) : zsum;
      __half* tile = reinterpret_cast<__half*>(base_ptr + L::k3) + (size_t)(qd * kColsPer) * 128 + frow;
#pragma unroll
      for (int c = 0; c < kColsPer; ++c) {
        acc[c] *= inv;
        tile[c * 128] = __float2half_rn(acc[c]);
      }
      if (prm.a32 && feat < p) {
        float4* arow = reinterpret_cast<float4*>(prm.a32 + ((size_t)head * p + feat) * kD + qd * kColsPer);
#pragma unroll
        for (int c = 0; c < kColsPer; c += 4) arow[c >> 2] = make_float4(acc[c], acc[c + 1], acc[c + 2], acc[c + 3]);
      }
      if (prm.abf && feat < p)
        k2_store_split<kColsPer, kSplit && !kPerformer>(prm.abf + ((size_t)head * kATerms * p + feat) * kD + qd * kColsPer,
                                                        (size_t)p * kD, acc, kTerms == 3);
    }
    __syncthreads();
    if (ok && prm.aT16) {
      const int cpr = min(128, p - i0) >> 3;                // 16-byte pieces per row
      __half* dst = prm.aT16 + (size_t)head * kD * p + i0;
      const uint4* tile = reinterpret_cast<const uint4*>(base_ptr + L::k3);
      for (int idx = tid; idx < kD * 16; idx += kK2Threads) {
        const int c = idx >> 4, ch = idx & 15;
        if (ch < cpr) *reinterpret_cast<uint4*>(dst + (size_t)c * p + ch * 8) = tile[idx];
      }
    }
  } else {
    // partial results of this part of the keys: row 0 = maxima, row 1 = sums, rows 2.. = accumulator
    // columns, each row 128 features wide (consecutive lanes write consecutive words)
    const size_t part_stride = (size_t)(kD + 2) * 128;
    float* mine = prm.part + ((size_t)unit * nsplit + sp) * part_stride;
    if (ok) {
      if (qd == 0) {
        mine[frow] = run_max;
        mine[128 + frow] = zsum;
      }
#pragma unroll
      for (int c = 0; c < kColsPer; ++c) mine[(size_t)(2 + qd * kColsPer + c) * 128 + frow] = acc[c];
    }
    __threadfence();
    __syncthreads();
    __shared__ int last_arrival;
    if (tid == 0) last_arrival = (atomicAdd(prm.counters + unit, 1) == nsplit - 1) ? 1 : 0;
    __syncthreads();
    if (last_arrival && ok) {
      __threadfence();
      // merge: feature frow, a quarter of the d columns per thread; the partial results bypass L1
      const float* all = prm.part + (size_t)unit * nsplit * part_stride;
      float m_all = -INFINITY;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < nsplit) m_all = fmaxf(m_all, __ldcg(all + q * part_stride + frow));
      float z_all = 0.f;
#pragma unroll
      for (int c = 0; c < kColsPer; ++c) acc[c] = 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (q < nsplit) {
          const float scale = __expf(__ldcg(all + q * part_stride + frow) - m_all);
          z_all = fmaf(scale, __ldcg(all + q * part_stride + 128 + frow), z_all);
#pragma unroll
          for (int c = 0; c < kColsPer; ++c)
            acc[c] = fmaf(scale, __ldcg(all + q * part_stride + (size_t)(2 + qd * kColsPer + c) * 128 + frow), acc[c]);
        }
      }
      if (qd == 0 && feat < p) prm.weight[(size_t)head * p + feat] = m_all + (kSplit ? logf(z_all) : __logf(z_all));
      const float inv = 1.f / z_all;
      __half* dst = prm.aT16 + ((size_t)head * kD + qd * kColsPer) * p + feat;
      if (feat < p) {
#pragma unroll
        for (int c = 0; c < kColsPer; ++c) {
          acc[c] *= inv;
          if (prm.aT16) dst[(size_t)c * p] = __float2half_rn(acc[c]);
          if (prm.a32) prm.a32[((size_t)head * p + feat) * kD + qd * kColsPer + c] = acc[c];
        }
        if (prm.abf)
          k2_store_split(prm.abf + ((size_t)head * kATerms * p + feat) * kD + qd * kColsPer, (size_t)p * kD, acc,
                         kSplit && kPerformer && kATerms == 3);
      }
      if (tid == 0) prm.counters[unit] = 0;
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  if (warp == 14) tmem_dealloc(tmem, 512);
}

}  // namespace flurka
