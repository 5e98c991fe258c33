// Backward of the query side on tensor cores for d = 64 and PERFORMER (bf16, up to 256 features).
//
// The forward's query side (arxiv 2306.15799, Eq. (2) with the normalised weights of Appendix D) is
//     O_n = sum_i P_ni a_i,    P_n. = softmax_i(l_n.),    l_ni = w_i . q_n + b_i.
// The paper trains through it but prints no backward formulas; by the chain rule, given dO,
//     g_ni = dO_n . a_i,   delta_n = sum_i P_ni g_ni,   c_ni = P_ni (g_ni - delta_n),
//     dq_n = sum_i c_ni w_i,   da_i = sum_n P_ni dO_n,   db_i = sum_n c_ni = a_i . da_i - sum_n P_ni delta_n.
// A CTA owns 128 features and walks tiles of 128 query rows; with more than 128 features a cluster of two CTAs walks the
// same tiles, half of the features each.  Per tile and CTA, every product a tcgen05 MMA with fp32 accumulators:
//     S = Q W^T  and  G = dO a^T  (a as two bf16 terms, so g is exact to 2^-17),
//     dQ = C W,   da += P^T dO,   (P^T delta) += P^T [delta_hi delta_mid delta_lo].
// What a row needs from the other half of the features, its maximum, sum and weighted sum, crosses the cluster through
// shared memory (st.async), and so does the half of dQ that the other CTA stores.  da and P^T delta stay in TMEM over all
// the tiles of a head; they are added to global memory when it changes.  The key side wants e_i = db_i - a_i . da_i, which
// is -sum_n P_ni delta_n: db itself is never formed.
//
// A tile's chain (products, maximum, exponentials, exchange of the row sums, P and C, products, exchange of dQ) is about
// three times its tensor time (1790 cycles) and its exponentials (1024), so two tiles are in flight: two groups of eight
// warps, two threads per row, take every other tile, and each fills the other's waits.  What makes room for the second:
//   * S passes through 128 columns of TMEM that both groups share: a group reads it once, into 64 registers per thread
//     that hold the weights from then on.  G stays in TMEM (128 columns a group) and is read twice, a few columns at a time.
//   * C (bf16 pairs) goes over the half of G that the same thread has read already, and is the A operand of dQ from there
//     (32 cycles a step instead of 48); dQ goes over the other half.  So that every thread overwrites only columns of its
//     own, a thread takes features 32 h .. 32 h + 31 of each half of the 128.
//   * What the other CTA adds to this CTA's half of dQ arrives in the P tile, once both CTAs' da have read theirs.
// Measured at 64 heads x N = 16384, m = 256: all features in one CTA 470 us, one tile in flight 327 us, two 322 us.
//
// kSplit (sequence lengths that are no multiple of 8): P and C as two bf16 terms each (16 to 17 bits; da and P^T delta have the
// same P), a as three, for the key side subtracts what is formed from it (see k2_key_side.cuh).  The second terms take the P
// buffer and the G columns of the second group, so one tile is in flight.
#pragma once

#include <cuda_bf16.h>

#include "k1_down_project_pair.cuh"
#include "k4_bwd_query_wide.cuh"
#include "tc_common.cuh"

namespace flurka {

template <int v> struct IntC { static constexpr int value = v; };      // a compile-time index handed to a lambda

template <bool kSplit> struct K8Shape {
  static constexpr int kGroups = kSplit ? 1 : 2;
  static constexpr int kThreads = 128 + 256 * kGroups;   // loader, MMA issuer, head operands, an idle warp; the row owners
  // registers: 640 threads x 96 at launch = 128 x 32 + 512 x 112; 384 x 168 = 128 x 72 + 256 x 216
  static constexpr int kRegsFew = kSplit ? 72 : 32, kRegsMany = kSplit ? 216 : 112;
};

// Shared memory: a Q tile is free as soon as S is formed, a dO tile only after da.
template <bool kSplit> struct K8Smem {
  static constexpr int kQ = 2, kDO = 3;                                                   // stages of 16 KB
  static constexpr uint32_t kTerms = kSplit ? 3 : 2, kGroups = kSplit ? 1 : 2;
  static constexpr uint32_t a = 0, w = kTerms * 16384, p = w + 16384;                     // P: 32 KB per group (kSplit: per term)
  static constexpr uint32_t q = p + 65536, dout = q + kQ * 16384;
  static constexpr uint32_t delta = dout + kDO * 16384;                                   // [16 x 128] bf16 per group
  static constexpr uint32_t stat = delta + kGroups * 4096;                                // [4 parts][128] x (maximum, sum, weighted sum) per group
  static constexpr uint32_t bias = stat + kGroups * 8192;                                 // b_i log2 e of two heads
  static constexpr uint32_t bars = bias + 1024;
  static constexpr int bytes = (int)bars + 256 + 1024;
};
// TMEM columns: S 0..127, G of group g 128 (1 + g) .. (C over the first 64, dQ over the others; kSplit: the two terms of C in
// place of the second group's G), da 384..447, P^T delta 448..463
constexpr uint32_t kK8ColG = 128, kK8ColDA = 384, kK8ColDD = 448;

// kParts: CTAs per cluster (1 or 2), 128 features each
template <int kParts, bool kSplit>
__global__ void __launch_bounds__(K8Shape<kSplit>::kThreads, 1)
k8_bwd_query_units(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmDO,
                   const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmA,
                   const K7Params prm) {
  using namespace tc;
  using L = K8Smem<kSplit>;
  constexpr int kGroups = K8Shape<kSplit>::kGroups, kThreads = K8Shape<kSplit>::kThreads;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t bars = base + L::bars;
  const uint32_t bar_w = bars;               // W landed
  const uint32_t bar_q = bars + 8;           // [2] Q tile landed
  const uint32_t bar_qfree = bars + 24;      // [2] ... S formed
  const uint32_t bar_do = bars + 40;         // [3] dO tile landed
  const uint32_t bar_dofree = bars + 64;     // [3] ... da added to
  const uint32_t bar_req = bars + 88;        // every product with the old head's a is complete: load the next
  const uint32_t bar_head = bars + 96;       // a, b of a new head in place
  const uint32_t bar_sfree = bars + 104;     // S read out (8 warps of the tile's group)
  const uint32_t bar_flush = bars + 112;     // da, P^T delta of the old head read out (8 warps)
  // one per group:
  const uint32_t bar_s = bars + 120;         // S ready
  const uint32_t bar_g = bars + 136;         // G ready
  const uint32_t bar_gfree = bars + 152;     // dQ, which lies over G, read out (8 warps)
  const uint32_t bar_pc = bars + 168;        // P, C, delta written (8 warps)
  const uint32_t bar_dq = bars + 184;        // dQ complete
  const uint32_t bar_out = bars + 200;       // da, P^T delta complete in all CTAs of the cluster
  const uint32_t bar_x = bars + 216;         // the row sums of all parts are here (8 local warps, the others by their bytes)
  const uint32_t bar_y = bars + 232;         // the other CTA's part of this CTA's half of dQ is here
  const uint32_t tmem_slot = bars + 248;
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_shared;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int p = prm.p;
  const uint32_t rank = kParts == 2 ? cluster_ctarank() : 0u;
  const int f0 = (int)rank * 128;                             // first feature of this CTA
  const bool both = f0 + 64 < p;                              // 128 features here (else 64: m is a multiple of 64)
  const int unit = blockIdx.x / kParts, units = gridDim.x / kParts;
  const int t_begin = (int)(((long long)unit * prm.total_tiles) / units);
  const int nt = (int)(((long long)(unit + 1) * prm.total_tiles) / units) - t_begin;

  if (tid == 0) {
    abort_flag = 0;
    mbar_init(bar_w, 1);
    for (int s = 0; s < L::kQ; ++s) {
      mbar_init(bar_q + 8 * s, 1);
      mbar_init(bar_qfree + 8 * s, 1);
    }
    for (int s = 0; s < L::kDO; ++s) {
      mbar_init(bar_do + 8 * s, 1);
      mbar_init(bar_dofree + 8 * s, 1);
    }
    mbar_init(bar_req, 1);
    mbar_init(bar_head, 33);
    mbar_init(bar_sfree, 8);
    mbar_init(bar_flush, 8);
    for (int g = 0; g < 2; ++g) {
      mbar_init(bar_s + 8 * g, 1);
      mbar_init(bar_g + 8 * g, 1);
      mbar_init(bar_gfree + 8 * g, 8);
      mbar_init(bar_pc + 8 * g, 8);
      mbar_init(bar_dq + 8 * g, 1);
      mbar_init(bar_out + 8 * g, kParts);
      mbar_init(bar_x + 8 * g, 8);
      mbar_init(bar_y + 8 * g, 1);
    }
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  {
    // the delta operands [16 x 128] (K-major, no swizzle): rows 0..2 are rewritten per tile, the rest stays zero
    uint32_t* dz = reinterpret_cast<uint32_t*>(base_ptr + L::delta);
    for (int e = tid; e < 1024 * kGroups; e += kThreads) dz[e] = 0u;
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
  if (kParts == 2) cluster_sync_all();       // the other CTA's barriers exist before anything is sent to them
  else __syncthreads();
  const uint32_t tmem = tmem_base_shared;
  const float kLog2e = 1.4426950408889634f;

  if (nt > 0) {
    if (warp < 4) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(K8Shape<kSplit>::kRegsFew));
      if (warp == 0 && elect_one()) {
        // ============================================================ loader: W, then Q and dO tiles
        prefetch_tmap(&tmQ);
        prefetch_tmap(&tmDO);
        prefetch_tmap(&tmW);
        mbar_arrive_expect_tx(bar_w, 16384u);
        tma_load_2d(base + L::w, &tmW, bar_w, 0, f0);         // rows past p read as zero
        bool ok = true;
        int head = t_begin / prm.tiles_per_head, tih = t_begin % prm.tiles_per_head;
        int i = 0;
        for (; i < nt && ok; ++i) {
          const int x = prm.H > 0 ? (head % prm.H) * 64 : 0, z = prm.H > 0 ? head / prm.H : head;
          const int sq = i % L::kQ, sd = i % L::kDO;
          if (i >= L::kQ) ok = mbar_wait(bar_qfree + 8 * sq, (uint32_t)(i / L::kQ - 1) & 1u, prm.status, &abort_flag);
          if (!ok) break;
          mbar_arrive_expect_tx(bar_q + 8 * sq, 16384u);
          tma_load_3d(base + L::q + sq * 16384, &tmQ, bar_q + 8 * sq, x, tih * 128, z);
          if (i >= L::kDO) ok = mbar_wait(bar_dofree + 8 * sd, (uint32_t)(i / L::kDO - 1) & 1u, prm.status, &abort_flag);
          if (!ok) break;
          mbar_arrive_expect_tx(bar_do + 8 * sd, 16384u);
          tma_load_3d(base + L::dout + sd * 16384, &tmDO, bar_do + 8 * sd, x, tih * 128, z);
          if (++tih == prm.tiles_per_head) { tih = 0; ++head; }
        }
        if (!ok) {
          // loads in flight still land in this CTA's shared memory: wait for them (bounded)
          for (int e = max(0, i - L::kQ); e <= i && e < nt; ++e)
            (void)mbar_wait(bar_q + 8 * (e % L::kQ), (uint32_t)(e / L::kQ) & 1u, prm.status, &abort_flag);
          for (int e = max(0, i - L::kDO); e < i; ++e)
            (void)mbar_wait(bar_do + 8 * (e % L::kDO), (uint32_t)(e / L::kDO) & 1u, prm.status, &abort_flag);
        }
      } else if (warp == 1 && elect_one()) {
        // ============================================================ MMA issuer
        const uint32_t idescS = make_idesc(kFmtBF16, 0, 0, 128, both ? 128 : 64);   // S, G: both operands K-major
        const uint32_t idescQ = make_idesc(kFmtBF16, 0, 1, 128, 64);    // dQ: C from TMEM, W MN-major
        const uint32_t idescA = make_idesc(kFmtBF16, 1, 1, 128, 64);    // da: P^T (MN-major A) x dO (MN-major B)
        const uint32_t idescD = make_idesc(kFmtBF16, 1, 0, 128, 16);    // P^T delta: delta as a K-major B
        bool ok = mbar_wait(bar_w, 0, prm.status, &abort_flag);
        int head = -1, events = 0, flushes = 0;
        auto form_sg = [&](int i) {      // S, G of tile i
          const int g = i % kGroups, h = (t_begin + i) / prm.tiles_per_head, sq = i % L::kQ, sd = i % L::kDO;
          if (h != head) {
            if (i > 0) ok = mbar_wait(bar_g + 8 * ((i - 1) % kGroups), (uint32_t)((i - 1) / kGroups) & 1u, prm.status, &abort_flag);
            if (!ok) return;
            mbar_arrive(bar_req);
            ok = mbar_wait(bar_head, (uint32_t)(events++) & 1u, prm.status, &abort_flag);
            head = h;
          }
          if (ok) ok = mbar_wait(bar_q + 8 * sq, (uint32_t)(i / L::kQ) & 1u, prm.status, &abort_flag);
          if (ok && i > 0) ok = mbar_wait(bar_sfree, (uint32_t)(i - 1) & 1u, prm.status, &abort_flag);
          if (!ok) return;
          tcgen05_fence_after();
          mma_ss_x4(tmem, make_sdesc(base + L::q + sq * 16384, 16, 1024, kSwizzle128),
                    make_sdesc(base + L::w, 16, 1024, kSwizzle128), 2, 2, idescS, 0u);
          mma_commit(bar_qfree + 8 * sq);
          mma_commit(bar_s + 8 * g);
          ok = mbar_wait(bar_do + 8 * sd, (uint32_t)(i / L::kDO) & 1u, prm.status, &abort_flag);
          if (ok && i >= kGroups) ok = mbar_wait(bar_gfree + 8 * g, (uint32_t)(i / kGroups - 1) & 1u, prm.status, &abort_flag);
          if (!ok) return;
          tcgen05_fence_after();
          const uint64_t ag = make_sdesc(base + L::dout + sd * 16384, 16, 1024, kSwizzle128);
          const uint32_t dst = tmem + kK8ColG + (uint32_t)g * 128u;
          for (uint32_t t = 0; t < L::kTerms; ++t)
            mma_ss_x4(dst, ag, make_sdesc(base + L::a + t * 16384u, 16, 1024, kSwizzle128), 2, 2, idescS, t > 0 ? 1u : 0u);
          mma_commit(bar_g + 8 * g);
        };
        if (ok) form_sg(0);
        int acc_head = -1;
        for (int i = 0; i < nt && ok; ++i) {
          const int g = i % kGroups, this_head = (t_begin + i) / prm.tiles_per_head;
          // (kSplit: one tile at a time, whose dQ has to leave before the next G comes)
          if (!kSplit && i + 1 < nt) {
            form_sg(i + 1);
            if (!ok) break;
          }
          ok = mbar_wait(bar_pc + 8 * g, (uint32_t)(i / kGroups) & 1u, prm.status, &abort_flag);
          if (!ok) break;
          tcgen05_fence_after();
          // dQ: the 32 features that a thread holds of each half of the 128 are 16 columns of C, 16 features a step
          const uint32_t col_g = tmem + kK8ColG + (uint32_t)g * 128u;
          uint32_t add = 0u;
          for (int term = 0; term < (kSplit ? 2 : 1); ++term) {
            const uint32_t c = kSplit ? tmem + kK8ColG + 128u + (uint32_t)term * 64u : col_g;
            for (int fh = 0; fh < 2; ++fh)
              for (int h = 0; h < (both ? 2 : 1); ++h) {
                mma_ts_x2(col_g + 64u, c + (uint32_t)(fh * 32 + h * 16),
                          make_sdesc(base + L::w + (uint32_t)(h * 64 + fh * 32) * 128u, 8192, 1024, kSwizzle128), 128, idescQ, add);
                add = 1u;
              }
          }
          mma_commit(bar_dq + 8 * g);
          uint32_t first = 1u;
          if (this_head != acc_head) {
            // the sums of the head before have left TMEM
            if (acc_head >= 0) ok = mbar_wait(bar_flush, (uint32_t)(flushes++) & 1u, prm.status, &abort_flag);
            if (!ok) break;
            tcgen05_fence_after();
            acc_head = this_head;
            first = 0u;
          }
          const uint32_t sm_do = base + L::dout + (i % L::kDO) * 16384;
          const uint32_t sm_p = base + L::p + (uint32_t)g * 32768u, sm_d = base + L::delta + (uint32_t)g * 4096u;
          for (int term = 0; term < (kSplit ? 2 : 1); ++term)
            for (int j = 0; j < 2; ++j) {      // 64 rows: 16 rows of P and of dO, 256 B of delta per step
              const uint64_t ap = make_sdesc(sm_p + term * 32768 + j * 8192, 16384, 1024, kSwizzle128);
              mma_ss_x4(tmem + kK8ColDA, ap, make_sdesc(sm_do + j * 8192, 8192, 1024, kSwizzle128), 128, 128, idescA, first);
              mma_ss_x4(tmem + kK8ColDD, ap, make_sdesc(sm_d + j * 1024, 128, 2048, kSwizzleNone), 128, 16, idescD, first);
              first = 1u;
            }
          mma_commit(bar_dofree + 8 * (i % L::kDO));
          if (kParts == 2) mma_commit_cluster(bar_out + 8 * g, 3);
          else mma_commit(bar_out + 8 * g);
          if (kSplit && i + 1 < nt) form_sg(i + 1);
        }
      } else if (warp == 2) {
        // ============================================================ a and b of a new head, when the issuer asks
        if (lane == 0) prefetch_tmap(&tmA);
        grid_dependency_wait_async();
        const int head0 = t_begin / prm.tiles_per_head, head1 = (t_begin + nt - 1) / prm.tiles_per_head;
        bool ok = true;
        for (int head = head0; head <= head1; ++head) {
          ok = mbar_wait(bar_req, (uint32_t)(head - head0) & 1u, prm.status, &abort_flag);
          if (!ok) break;
          if (lane == 0) {
            mbar_arrive_expect_tx(bar_head, L::kTerms * 16384u);
            for (uint32_t t = 0; t < L::kTerms; ++t)
              tma_load_3d(base + L::a + t * 16384u, &tmA, bar_head, 0, f0, head * (int)L::kTerms + (int)t);
          }
          const float* wv = prm.weight + (size_t)head * p;
          float mx = -INFINITY;
          for (int f = lane; f < p; f += 32) mx = fmaxf(mx, __ldcg(wv + f));
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
          // (the head before the last one's: every thread has read its S, with which b is read, or the last G would not be formed)
          float* bs = reinterpret_cast<float*>(base_ptr + L::bias) + ((head - head0) & 1) * 128;
          for (int f = lane; f < 128; f += 32) bs[f] = f0 + f < p ? (__ldcg(wv + f0 + f) - mx) * kLog2e : 0.f;
          mbar_arrive(bar_head);
        }
      }
    } else {
      // ============================================================ row owners: two threads per row, 64 features each
      asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(K8Shape<kSplit>::kRegsMany));
      const int g = kSplit ? 0 : (warp - 4) >> 3;
      const int q4 = warp & 3, fh = ((warp - 4) >> 2) & 1;
      int row = q4 * 32 + lane;
      const uint32_t lane_base = tmem + ((uint32_t)(q4 * 32) << 16);
      const uint32_t col_g = lane_base + kK8ColG + (uint32_t)g * 128u;
      const uint32_t peer = kParts == 2 ? (rank ^ 1u) : 0u;
      bool ok = true;
      grid_dependency_wait();

      // da, P^T delta of one head leave TMEM: lane = feature, 32 of the 64 columns per thread
      auto flush = [&](int head) {
        uint32_t r[16];
        const int feat = f0 + row;
#pragma unroll 1
        for (int c = 0; c < 32; c += 16) {
          tmem_ld16(lane_base + kK8ColDA + fh * 32 + c, r);
          tmem_wait_ld16(r);
          if (feat < p) {
            float4* darow = reinterpret_cast<float4*>(prm.da + ((size_t)head * p + feat) * 64 + fh * 32 + c);
#pragma unroll
            for (int e = 0; e < 4; ++e)
              atomicAdd(darow + e, make_float4(__uint_as_float(r[4 * e]), __uint_as_float(r[4 * e + 1]),
                                               __uint_as_float(r[4 * e + 2]), __uint_as_float(r[4 * e + 3])));
          }
        }
        if (fh == 0) {
          tmem_ld16(lane_base + kK8ColDD, r);
          tmem_wait_ld16(r);
          if (feat < p)
            atomicAdd(prm.ei + (size_t)head * p + feat, -(__uint_as_float(r[0]) + __uint_as_float(r[1]) + __uint_as_float(r[2])));
        }
      };

      const int head0 = t_begin / prm.tiles_per_head;
      for (int i = g; i < nt; i += kGroups) {
        const int head = (t_begin + i) / prm.tiles_per_head, tih = (t_begin + i) - head * prm.tiles_per_head;
        const uint32_t par = (uint32_t)(i / kGroups) & 1u;
        // (addresses are formed where they are used, tile by tile: kept over the loop they would not fit beside the weights)
        asm volatile("" : "+r"(row));
        float4* stat = reinterpret_cast<float4*>(base_ptr + L::stat) + g * 512;
        const uint32_t sm_p = base + L::p + (uint32_t)g * 32768u;
        const uint32_t prow = sm_p + (uint32_t)row * 128u;
        // the dQ columns that arrive in the P tile: four 16-byte pieces a thread, 32 rows of a piece side by side
        const uint32_t dqx = sm_p + (uint32_t)(fh * 4 + (row >> 5)) * 2048u + (uint32_t)(row & 31) * 16u;
        ok = mbar_wait(bar_s + 8 * g, par, prm.status, &abort_flag);
        if (!ok) break;
        tcgen05_fence_after();
        // this thread's weights exp(l - own maximum) as pairs: features 32 fh .. + 31, then 64 + 32 fh .. + 31 (pairs 16..),
        // 32 at a time; more in flight at once does not fit
        uint64_t w2[32];
        float mx;
        {
          const float* bs = reinterpret_cast<const float*>(base_ptr + L::bias) + ((head - head0) & 1) * 128 + fh * 32;
          const uint64_t l2 = pack2(kLog2e, kLog2e);
          float m0 = -INFINITY, m1 = -INFINITY;
          auto logits = [&](auto hh) {                   // 32 features, as two chunks
            constexpr int h = decltype(hh)::value;
            uint32_t sa[32];
            tmem_ld32(lane_base + h * 64 + fh * 32, sa);
            tmem_wait_ld(sa);
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
              const ulonglong2 b4 = *reinterpret_cast<const ulonglong2*>(bs + h * 64 + 2 * e);
              w2[16 * h + e] = fma2(pack2u(sa[2 * e], sa[2 * e + 1]), l2, b4.x);
              w2[16 * h + e + 1] = fma2(pack2u(sa[2 * e + 2], sa[2 * e + 3]), l2, b4.y);
              float x0, x1, x2, x3;
              unpack2(w2[16 * h + e], x0, x1);
              unpack2(w2[16 * h + e + 1], x2, x3);
              m0 = fmax3(m0, x0, x1);
              m1 = fmax3(m1, x2, x3);
            }
          };
          logits(IntC<0>());
          if (both) logits(IntC<1>());
          mx = fmaxf(m0, m1);
          tcgen05_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_sfree);
        }
        // ---- exponentials, their sum and the sum of P g; 16 features at a time (chunk c: columns 64 (c/2) + 32 fh + 16 (c%2))
        ok = mbar_wait(bar_g + 8 * g, par, prm.status, &abort_flag);
        if (!ok) break;
        tcgen05_fence_after();
        {
          uint64_t den2 = 0ull, num2 = 0ull;
          const uint64_t nm2 = pack2(-mx, -mx);
          auto expo = [&](auto cc) {
            constexpr int c = decltype(cc)::value;
            uint32_t ga[16];
            tmem_ld16(col_g + (c >> 1) * 64 + fh * 32 + (c & 1) * 16, ga);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              float x0, x1;
              unpack2(add2(w2[8 * c + e], nm2), x0, x1);
              w2[8 * c + e] = pack2(k4_ex2(x0), k4_ex2(x1));
              den2 = add2(den2, w2[8 * c + e]);
            }
            tmem_wait_ld16(ga);
#pragma unroll
            for (int e = 0; e < 8; ++e) num2 = fma2(w2[8 * c + e], pack2u(ga[2 * e], ga[2 * e + 1]), num2);
          };
          expo(IntC<0>());
          expo(IntC<1>());
          if (both) {
            expo(IntC<2>());
            expo(IntC<3>());
          }
          // the sums to everyone who shares the row (what was read of the tile before is read: see bar_out, bar_y)
          float d0, d1, n0, n1;
          unpack2(den2, d0, d1);
          unpack2(num2, n0, n1);
          const uint32_t at = (rank * 2 + (uint32_t)fh) * 128 + (uint32_t)row;
          stat[at] = make_float4(mx, d0 + d1, n0 + n1, 0.f);
          if (kParts == 2)
            st_async_v4(map_to_cta(base + L::stat + (uint32_t)g * 8192u + at * 16u, peer), __float_as_uint(mx), __float_as_uint(d0 + d1),
                        __float_as_uint(n0 + n1), 0u, map_to_cta(bar_x + 8 * g, peer));
          __syncwarp();
          if (lane == 0) {
            if (kParts == 2 && q4 == 0 && fh == 0) mbar_arrive_expect_tx(bar_x + 8 * g, 256u * 16u);
            else mbar_arrive(bar_x + 8 * g);
          }
        }
        ok = mbar_wait(bar_x + 8 * g, par, prm.status, &abort_flag);
        if (!ok) break;
        float delta, scale;
        {
          float4 part[2 * kParts];
          float all = -INFINITY, dsum = 0.f, nsum = 0.f;
#pragma unroll
          for (int q = 0; q < 2 * kParts; ++q) {
            part[q] = stat[q * 128 + row];
            all = fmaxf(all, part[q].x);
          }
#pragma unroll
          for (int q = 0; q < 2 * kParts; ++q) {
            const float f = k4_ex2(part[q].x - all);
            dsum = fmaf(part[q].y, f, dsum);
            nsum = fmaf(part[q].z, f, nsum);
          }
          const float inv = __fdividef(1.f, dsum);
          delta = nsum * inv;
          scale = k4_ex2(mx - all) * inv;
        }
        if (fh == 0) {
          // delta_n as three bf16 terms: element (c, n) of the [16 x 128] operand at (n/8)*128 + c*16 + (n%8)*2 bytes
          __nv_bfloat16* dt = reinterpret_cast<__nv_bfloat16*>(base_ptr + L::delta) + g * 2048 + (row >> 3) * 64 + (row & 7);
          float r = delta;
          const __nv_bfloat16 d0 = __float2bfloat16_rn(r);  r -= __bfloat162float(d0);
          const __nv_bfloat16 d1 = __float2bfloat16_rn(r);  r -= __bfloat162float(d1);
          dt[0] = d0; dt[8] = d1; dt[16] = __float2bfloat16_rn(r);
        }
        // ---- P into shared memory, C into TMEM
        {
          const uint64_t sc2 = pack2(scale, scale), nd2 = pack2(-delta, -delta);
          const uint32_t swz = (uint32_t)(row & 7);
          // eight features at a time (chunk c: columns 64 (c/4) + 32 fh + 8 (c%4)), the next chunk's G on its way
          uint32_t ga[2][8];
          tmem_ld8(col_g + fh * 32, ga[0]);
          auto weights = [&](auto cc) {
            constexpr int c = decltype(cc)::value;
            uint32_t v[4];
            [[maybe_unused]] uint32_t lo[4];
            auto pack = [&](uint64_t x2, int e) {
              float x0, x1;
              unpack2(x2, x0, x1);
              v[e] = k4_bf16x2(x0, x1);
              if constexpr (kSplit)
                lo[e] = k4_bf16x2(x0 - __uint_as_float(v[e] << 16), x1 - __uint_as_float(v[e] & 0xffff0000u));
            };
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              w2[4 * c + e] = mul2(w2[4 * c + e], sc2);
              pack(w2[4 * c + e], e);
            }
            const uint32_t to = prow + (c >> 2) * 16384u + (((uint32_t)(fh * 4 + (c & 3)) ^ swz) << 4);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(to), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
            if constexpr (kSplit)
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(to + 32768u), "r"(lo[0]), "r"(lo[1]), "r"(lo[2]),
                           "r"(lo[3]) : "memory");
            tmem_wait_ld8(ga[c & 1]);
            if (c < 3 || (c < 7 && both)) tmem_ld8(col_g + ((c + 1) >> 2) * 64 + fh * 32 + ((c + 1) & 3) * 8, ga[(c + 1) & 1]);
#pragma unroll
            for (int e = 0; e < 4; ++e)
              pack(mul2(w2[4 * c + e], add2(pack2u(ga[c & 1][2 * e], ga[c & 1][2 * e + 1]), nd2)), e);
            // C: four columns a chunk; kSplit: in columns of their own, else over some that this thread has read (chunk c > 0:
            // over those of chunk c / 2)
            if constexpr (kSplit) {
              tmem_st4(col_g + 128 + fh * 32 + c * 4, v);
              tmem_st4(col_g + 192 + fh * 32 + c * 4, lo);
            } else {
              tmem_st4(col_g + fh * 32 + c * 4, v);
            }
          };
          weights(IntC<0>());
          weights(IntC<1>());
          weights(IntC<2>());
          weights(IntC<3>());
          if (both) {
            weights(IntC<4>());
            weights(IntC<5>());
            weights(IntC<6>());
            weights(IntC<7>());
          }
          tmem_wait_st();
          fence_proxy_async_smem();
          tcgen05_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_pc + 8 * g);
        }
        // ---- dQ: with two CTAs each stores 32 of the 64 columns, its own sums plus the other CTA's
        constexpr int kDQ = 32 / kParts;                             // columns of a thread
        uint32_t own[kDQ], other[kParts == 2 ? 16 : 1];
        ok = mbar_wait(bar_dq + 8 * g, par, prm.status, &abort_flag);
        if (!ok) break;
        tcgen05_fence_after();
        if constexpr (kParts == 2) {
          tmem_ld16(col_g + 64 + peer * 32 + fh * 16, other);
          tmem_ld16(col_g + 64 + rank * 32 + fh * 16, own);
          tmem_wait_ld16(other);
          tmem_wait_ld16(own);
        } else {
          tmem_ld32(col_g + 64 + fh * 32, own);
          tmem_wait_ld(own);
        }
        tcgen05_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_gfree + 8 * g);
        // da of all CTAs complete: P tiles are read; the sums of a head that ends here leave TMEM
        ok = mbar_wait(bar_out + 8 * g, par, prm.status, &abort_flag);
        if (!ok) break;
        if constexpr (kParts == 2) {
          const uint32_t to = map_to_cta(dqx, peer), bar = map_to_cta(bar_y + 8 * g, peer);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            st_async_v4(to + j * 512u, other[4 * j], other[4 * j + 1], other[4 * j + 2], other[4 * j + 3], bar);
          if (q4 == 0 && fh == 0 && lane == 0) mbar_arrive_expect_tx(bar_y + 8 * g, 16384u);
        }
        if (i + 1 == nt || tih + 1 == prm.tiles_per_head) {
          tcgen05_fence_after();
          flush(head);
          tcgen05_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_flush);
        }
        if constexpr (kParts == 2) {
          // (P is written again only after the next bar_x: all eight warps have read what arrived here by then)
          ok = mbar_wait(bar_y + 8 * g, par, prm.status, &abort_flag);
          if (!ok) break;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float a, b, c, d;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(a), "=f"(b), "=f"(c), "=f"(d) : "r"(dqx + j * 512u)
                         : "memory");
            own[4 * j] = __float_as_uint(__uint_as_float(own[4 * j]) + a);
            own[4 * j + 1] = __float_as_uint(__uint_as_float(own[4 * j + 1]) + b);
            own[4 * j + 2] = __float_as_uint(__uint_as_float(own[4 * j + 2]) + c);
            own[4 * j + 3] = __float_as_uint(__uint_as_float(own[4 * j + 3]) + d);
          }
        }
        const int n = tih * 128 + row;
        if (n < prm.N) {
          __nv_bfloat16* o = prm.dQ + (prm.H > 0 ? (((size_t)(head / prm.H) * prm.N + n) * prm.H + (size_t)(head % prm.H)) * 64
                                                 : ((size_t)head * prm.N + n) * 64) + rank * 32 + fh * kDQ;
#pragma unroll
          for (int h = 0; h < kDQ / 16; ++h) {
            uint32_t v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
              v[e] = k4_bf16x2(__uint_as_float(own[16 * h + 2 * e]), __uint_as_float(own[16 * h + 2 * e + 1]));
            k4_store16(o + 16 * h, v, prm.wide != 0);
          }
        }
      }
      if (warp == 4 && lane == 0) grid_launch_dependents();
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  if (kParts == 2) cluster_sync_all();       // nothing is sent to a CTA that has left
  if (warp == 1) tmem_dealloc(tmem, 512);
}

}  // namespace flurka
