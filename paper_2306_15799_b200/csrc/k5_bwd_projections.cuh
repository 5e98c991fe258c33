// Backward of the down-projection (arxiv 2306.15799, Eq. (2): K' = E K, V' = F V) on tensor cores:
//
//   kMode 0   dK_h = E^T dK'_h,  dV_h = F^T dV'_h        all heads that share E at once: [N x k] x [k x columns]
//   kMode 1   dE = sum_h dK'_h K_h^T,  dF = sum_h dV'_h V_h^T        [k x columns] x [columns x N]
//
// dK', dV' come from the key side as two bf16 terms (hi + lo, exact to 2^-17), `split` = [2 projections][2 terms][k][BH d].
// Both terms meet the same other operand, so a stage of the ring holds 64 contraction elements of that one operand and
// of both terms: 48 KB per CTA for 1024 cycles of MMA.  A cluster of two CTAs owns 256 x kN outputs
// (tcgen05.mma.cta_group::2: each CTA its 128 rows of A, its half of B and of the columns of every stage, as in
// k1_down_project_pair.cuh) and walks its tiles persistently; the accumulators are double-buffered in TMEM, so that four
// warps store a tile (bf16 through swizzled slabs, TMA stores of whole lines) under the next tile's products.
// kN = 256, or 128 where tiles of 256 would leave half of the machine idle.
// kParts = 2 (mode 1, where even so more than half of the machine would be): a cluster of four CTAs, two pairs, has one
// tile, each pair half of the column blocks; the second pair sends its sums into the first pair's ring, which is free by
// then (st.async, 512 bytes a warp), and the first adds them as it reads its own.
// Every head its own E_i, F_i (Theorem 1): the columns of a tile are one head's over the batch.
// Measured against one 128-row tile per CTA with the products of the two terms in separate launches of their own sweep: a
// whole backward pass 706 -> 635 us (64 heads x N = 16384, d = 64, k = 256; mode 0 takes 107 us of it, mode 1 92 us) and
// 301 -> 243 us (RNN, 96 heads x N = 4096; 59 and 53 us), together with the key side on register tiles.  With the arrival on
// bar_accfree at CTA scope mode 0 takes 84 us instead of 107 and, RNN, 49 instead of 59.  The floor is the tensor
// time of both terms: 2 x 2 x 2 N k BH d operations, 82 us at 64 heads x N = 16384 (the stores of mode 0: 41 us).
#pragma once

#include <cuda_bf16.h>

#include "k1_down_project_pair.cuh"
#include "tc_common.cuh"

namespace flurka {

struct K5Params {
  int N, k, d, BH, H;        // H > 0: K, V, dK, dV are [B,N,H,d]
  int groups;                // heads with their own E, F (1: shared by all)
  int slabs;                 // 64-wide column blocks that share an E: BH / groups * d / 64
  int row_tiles, col_tiles;  // per (projection, group)
  int tiles;                 // 2 * groups * row_tiles * col_tiles
  int* status;
};

constexpr int kK5Threads = 192;
template <int kMode, int kN> struct K5Shape {
  static constexpr int kStages = 4;
  // A: 128 rows of one operand (kMode 0: E; kMode 1: both terms); B: this CTA's half of kN (kMode 0: both terms)
  static constexpr int kABytes = kMode == 0 ? 16384 : 32768;
  static constexpr int kBTerm = kN * 64;                             // bytes of one half-slab of 64 contraction elements
  static constexpr int kStageBytes = kABytes + (kMode == 0 ? 2 : 1) * kBTerm;
  static constexpr int kSlabs = kStages * kStageBytes;               // 4 warps x 2 x 4 KB of output slabs after the ring
  static constexpr int kBars = kSlabs + 32768;
  static constexpr int kSmemBytes = kBars + 128 + 1024;
};

// tmP0/tmP1: E, F ({N, k, groups}; boxes of 64 n x 64 k) or K, V (boxes of 64 c x kN/2 n); tmS: the split terms
// ({BH d, k, 4}; kMode 0: boxes of 64 x 64, kMode 1: 64 x 128); tmO0/tmO1: dK, dV (boxes of 64 c x 32 n) or dE, dF
// ({N, k, groups}; boxes of 64 n x 32 k)
template <int kMode, int kN, int kParts = 1>
__global__ void __launch_bounds__(kK5Threads, 1)
k5_bwd_projections(const __grid_constant__ CUtensorMap tmP0, const __grid_constant__ CUtensorMap tmP1,
                   const __grid_constant__ CUtensorMap tmS, const __grid_constant__ CUtensorMap tmO0,
                   const __grid_constant__ CUtensorMap tmO1, const K5Params p) {
  using namespace tc;
  using Sh = K5Shape<kMode, kN>;
  constexpr int kStages = Sh::kStages;
  static_assert(kParts == 1 || (kMode == 1 && kN * 512 <= Sh::kSlabs), "the other pair's sums fit into the ring");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bars = base + Sh::kBars;
  const uint32_t bar_full = bars;                     // [4] even CTA's: the loads of both CTAs of a stage have landed
  const uint32_t bar_empty = bars + 32;               // [4] the pair's MMAs have read the stage
  const uint32_t bar_acc = bars + 64;                 // [2] accumulator complete
  const uint32_t bar_accfree = bars + 80;             // [2] even CTA's: both CTAs' warps have read the accumulator
  const uint32_t bar_ring = bars + 96;                // kParts = 2, second pair: the first pair's ring is free
  const uint32_t bar_sums = bars + 104;               // kParts = 2, first pair: the second pair's sums are here
  const uint32_t tmem_slot = bars + 112;
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_shared;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t crank = cluster_ctarank(), rank = crank & 1u, even = crank & ~1u;     // rank: within the pair
  const int part = (int)(crank >> 1);
  const int pair = blockIdx.x / (2 * kParts), pairs = gridDim.x / (2 * kParts);       // (kParts = 2: of clusters)
  const int dblocks = p.d >> 6;
  const int all_chunks = kMode == 0 ? p.k >> 6 : p.slabs;
  const int c_begin = part * all_chunks / kParts, nchunks = (part + 1) * all_chunks / kParts - c_begin;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int i = 0; i < kStages; ++i) {
      mbar_init(bar_full + 8 * i, 1);
      mbar_init(bar_empty + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_acc + 8 * i, 1);
      mbar_init(bar_accfree + 8 * i, 8);
    }
    mbar_init(bar_ring, 4);
    mbar_init(bar_sums, 1);
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, 512);
    tmem_relinquish_pair();
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  if (threadIdx.x == 0) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(tmem_slot));
    tmem_base_shared = v;
  }
  cluster_sync_all();
  const uint32_t tmem = tmem_base_shared;

  // a tile: projection z, group g (head with its own E, or 0), row tile, column tile (the fastest: its E is reused)
  struct Tile { int z, g, rt, ct; };
  auto tile_at = [&](int t) {
    Tile r;
    r.ct = t % p.col_tiles; t /= p.col_tiles;
    r.rt = t % p.row_tiles; t /= p.row_tiles;
    r.g = t % p.groups;
    r.z = t / p.groups;
    return r;
  };
  // 64-wide column block s of a group: its head and the block within the head
  auto head_of = [&](int s, int g) { return p.groups > 1 ? (s / dblocks) * p.groups + g : s / dblocks; };

  if (warp == 0) {
    if (elect_one()) {
      // ------------------------------------------------ TMA producer (each CTA feeds its own shared memory)
      prefetch_tmap(&tmP0);
      prefetch_tmap(&tmP1);
      prefetch_tmap(&tmS);
      grid_dependency_wait_async();
      bool ok = true;
      int it = 0;
      for (int t = pair; t < p.tiles && ok; t += pairs) {
        const Tile tl = tile_at(t);
        const CUtensorMap* tmP = tl.z ? &tmP1 : &tmP0;
        for (int c = 0; c < nchunks; ++c, ++it) {
          const int st = it % kStages;
          if (it >= kStages) ok = mbar_wait(bar_empty + 8 * st, (uint32_t)(it / kStages - 1) & 1u, p.status, &abort_flag);
          if (!ok) break;
          const uint32_t a_dst = map_to_cta(base + st * Sh::kStageBytes, crank);
          const uint32_t b_dst = a_dst + Sh::kABytes;
          const uint32_t bar = map_to_cta(bar_full + 8 * st, even);
          if (rank == 0) mbar_arrive_expect_tx(bar_full + 8 * st, 2 * Sh::kStageBytes);
          if (kMode == 0) {
            // A: this CTA's 128 rows n of E^T as two 64-row slabs (n contiguous: MN-major)
            for (int s = 0; s < 2; ++s)
              tma_load_3d_pair(a_dst + s * 8192, tmP, bar, tl.rt * 256 + (int)rank * 128 + s * 64, c << 6, tl.g);
            // B: this CTA's half of the columns, both terms; column blocks past the last read as zero
            for (int s = 0; s < kN / 128; ++s) {
              const int slab = tl.ct * (kN / 64) + (int)rank * (kN / 128) + s;
              const int x = slab < p.slabs ? head_of(slab, tl.g) * p.d + (slab % dblocks) * 64 : p.BH * p.d;
              for (int tm = 0; tm < 2; ++tm)
                tma_load_3d_pair(b_dst + tm * Sh::kBTerm + s * 8192, &tmS, bar, x, c << 6, tl.z * 2 + tm);
            }
          } else {
            const int head = head_of(c_begin + c, tl.g), dc = ((c_begin + c) % dblocks) * 64;
            // A: this CTA's 128 rows of both terms (K-major); B: its half of the positions of one head's K or V (K-major)
            for (int tm = 0; tm < 2; ++tm)
              tma_load_3d_pair(a_dst + tm * 16384, &tmS, bar, head * p.d + dc, tl.rt * 256 + (int)rank * 128, tl.z * 2 + tm);
            const int n0 = tl.ct * kN + (int)rank * (kN / 2);
            if (p.H > 0) tma_load_3d_pair(b_dst, tmP, bar, (head % p.H) * p.d + dc, n0, head / p.H);
            else tma_load_3d_pair(b_dst, tmP, bar, dc, n0, head);
          }
        }
      }
      if (!ok && rank == 0) {
        // loads in flight still land in shared memory: wait for them (bounded)
        for (int e = max(0, it - kStages); e < it; ++e)
          (void)mbar_wait(bar_full + 8 * (e % kStages), (uint32_t)(e / kStages) & 1u, p.status, &abort_flag);
      }
    }
  } else if (warp == 1) {
    if (rank == 0 && elect_one()) {
      // ------------------------------------------------ even CTA: MMA issuer for the pair
      const uint32_t idesc = kMode == 0 ? make_idesc(kFmtBF16, 1, 1, 256, kN) : make_idesc(kFmtBF16, 0, 0, 256, kN);
      bool ok = true;
      int it = 0, i = 0;
      for (int t = pair; t < p.tiles && ok; t += pairs, ++i) {
        const int buf = i & 1;
        if (i >= 2) ok = mbar_wait_cluster(bar_accfree + 8 * buf, (uint32_t)(i / 2 - 1) & 1u, p.status, &abort_flag);
        if (!ok) break;
        tcgen05_fence_after();
        for (int c = 0; c < nchunks; ++c, ++it) {
          const int st = it % kStages;
          ok = mbar_wait(bar_full + 8 * st, (uint32_t)(it / kStages) & 1u, p.status, &abort_flag);
          if (!ok) break;
          tcgen05_fence_after();
          const uint32_t a = base + st * Sh::kStageBytes, b = a + Sh::kABytes;
          for (int tm = 0; tm < 2; ++tm) {
            const uint32_t add = (c > 0 || tm > 0) ? 1u : 0u;
            if (kMode == 0) {
              // MN-major operands: 64-wide slabs 8192 B apart, 8-row (contraction) groups 1024 B apart, 16 rows per step
              mma_ss_x4_pair(tmem + buf * kN, make_sdesc(a, 8192, 1024, kSwizzle128),
                             make_sdesc(b + tm * Sh::kBTerm, 8192, 1024, kSwizzle128), 128, 128, idesc, add);
            } else {
              // K-major operands: 128-byte rows, 8-row groups 1024 B apart, 32 B per step
              mma_ss_x4_pair(tmem + buf * kN, make_sdesc(a + tm * 16384, 16, 1024, kSwizzle128),
                             make_sdesc(b, 16, 1024, kSwizzle128), 2, 2, idesc, add);
            }
          }
          mma_commit_pair(bar_empty + 8 * st, even);
        }
        if (ok) mma_commit_pair(bar_acc + 8 * buf, even);
      }
    }
  } else {
    // ------------------------------------------------ epilogue: this CTA's 128 rows, bf16 slabs of [32 rows x 64 columns]
    const int q = warp & 3;
    const uint32_t slab0 = base + Sh::kSlabs + (uint32_t)(warp - 2) * 8192u;
    const int M = kMode == 0 ? p.N : p.k;
    const uint32_t free0 = map_to_cta(bar_accfree, even);
    int i = 0, stores = 0;
    bool ok = true;
    for (int t = pair; t < p.tiles && ok; t += pairs, ++i) {
      const Tile tl = tile_at(t);
      const CUtensorMap* tmO = tl.z ? &tmO1 : &tmO0;
      const int buf = i & 1;
      const int row0 = tl.rt * 256 + (int)rank * 128 + q * 32;
      ok = mbar_wait(bar_acc + 8 * buf, (uint32_t)(i / 2) & 1u, p.status, &abort_flag);
      if (!ok) break;
      if (t + pairs >= p.tiles && warp == 2 && lane == 0) grid_launch_dependents();
      tcgen05_fence_after();
      // the other pair's sums: 16-byte pieces of four columns, 128 rows of a piece side by side
      const uint32_t piece = base + (uint32_t)(q * 32 + lane) * 16u;
      if constexpr (kParts == 2) {
        if (part == 1) {
          ok = mbar_wait_cluster(bar_ring, 0, p.status, &abort_flag);
          if (!ok) break;
          const uint32_t to = map_to_cta(piece, rank), bar = map_to_cta(bar_sums, rank);
#pragma unroll 1
          for (int c = 0; c < kN; c += 32) {
            uint32_t r[32];
            tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + c, r);
            tmem_wait_ld(r);
#pragma unroll
            for (int e = 0; e < 8; ++e)
              st_async_v4(to + (uint32_t)(c / 4 + e) * 2048u, r[4 * e], r[4 * e + 1], r[4 * e + 2], r[4 * e + 3], bar);
          }
          tcgen05_fence_before();
          break;                                           // (one tile per cluster)
        }
        // every load of this CTA's ring has landed and has been read: the accumulators are complete
        if (lane == 0) {
          mbar_arrive_cluster(map_to_cta(bar_ring, 2u + rank));     // (with it the ring is the other pair's to write)
          if (warp == 2) mbar_arrive_expect_tx(bar_sums, 512u * kN);
        }
        ok = mbar_wait(bar_sums, 0, p.status, &abort_flag);
        if (!ok) break;
      }
#pragma unroll 1
      for (int cc = 0; cc < kN / 64; ++cc) {
        uint32_t ra[32], rb[32];
        const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + buf * kN + cc * 64;
        tmem_ld32(ta, ra);
        tmem_ld32(ta + 32, rb);
        tmem_wait_ld(ra);
        tmem_wait_ld(rb);
        if constexpr (kParts == 2) {
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            float x, y, z, w;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x), "=f"(y), "=f"(z), "=f"(w)
                         : "r"(piece + (uint32_t)(cc * 16 + e) * 2048u) : "memory");
            uint32_t* r = (e < 8 ? ra : rb) + 4 * (e & 7);
            r[0] = __float_as_uint(__uint_as_float(r[0]) + x);
            r[1] = __float_as_uint(__uint_as_float(r[1]) + y);
            r[2] = __float_as_uint(__uint_as_float(r[2]) + z);
            r[3] = __float_as_uint(__uint_as_float(r[3]) + w);
          }
        }
        if (cc == kN / 64 - 1) {
          tcgen05_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_remote(free0 + 8 * buf);
        }
        // which slab of the output this is, and whether it exists
        const int slab = tl.ct * (kN / 64) + cc;
        const bool live = row0 < M && (kMode == 0 ? slab < p.slabs : slab * 64 < p.N);
        if (!live) continue;
        const uint32_t slab_buf = slab0 + (uint32_t)(stores & 1) * 4096u;
        if (lane == 0) bulk_wait_group_read1();            // the store that last read this buffer is done with it
        __syncwarp();
        ++stores;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          const uint32_t* src = g < 4 ? ra : rb;
          uint32_t v[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const __nv_bfloat162 o2 = __floats2bfloat162_rn(__uint_as_float(src[(g & 3) * 8 + 2 * e]),
                                                            __uint_as_float(src[(g & 3) * 8 + 2 * e + 1]));
            v[e] = *reinterpret_cast<const uint32_t*>(&o2);
          }
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(slab_buf + lane * 128 + ((g ^ (lane & 7)) << 4)),
                       "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          if (kMode == 0) {
            const int head = head_of(slab, tl.g), c0 = (slab % dblocks) * 64;
            if (p.H > 0) tma_store_3d(tmO, slab_buf, (head % p.H) * p.d + c0, row0, head / p.H);
            else tma_store_3d(tmO, slab_buf, c0, row0, head);
          } else {
            tma_store_3d(tmO, slab_buf, slab * 64, row0, tl.g);
          }
          bulk_commit_group();
        }
      }
    }
    if (lane == 0) bulk_wait_group0();
  }
  // neither CTA gives its TMEM back while the other may still be part of an MMA or of its commits
  tcgen05_fence_before();
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) tmem_dealloc_pair(tmem, 512);
}

}  // namespace flurka
