// Backward of the query side on tensor cores for d = 64 (bf16; PERFORMER with up to 256 features, RNN).
//
// The forward's query side (arxiv 2306.15799, Eq. (2) with the normalised weights of Appendix D) is
//     O_n = sum_i P_ni a_i,    P_n. = softmax_i(l_n.),    l_ni = w_i . q_n + b_i.
// The paper trains through it but prints no backward formulas; by the chain rule, given dO,
//     g_ni = dO_n . a_i,   delta_n = sum_i P_ni g_ni,   c_ni = P_ni (g_ni - delta_n),
//     dq_n = sum_i c_ni w_i,   da_i = sum_n P_ni dO_n,   db_i = sum_n c_ni = a_i . da_i - sum_n P_ni delta_n.
// A CTA owns 128 features and walks tiles of 128 query rows; with more than 128 features a cluster of two CTAs walks the
// same tiles, half of the features each.  Per tile and CTA, every product a tcgen05 MMA with fp32 accumulators:
//     S = Q W^T + 1 b^T  and  G = dO a^T  (a as two bf16 terms, so g is exact to 2^-17),
//     dQ = C W,   da += P^T dO,   (P^T delta) += P^T [delta_hi delta_mid delta_lo],
// with P and C = bf16 c written to shared memory in the canonical 128-byte-swizzled layout (P doubles as an MN-major
// A operand).  Two threads per row hold their 64 values of S and of G in registers from the one read of TMEM to the
// weights: every exponential and every product is formed once.  (Holding all 256 features in one CTA needs S and G
// twice, in a sweep for delta and one for c, and left MMAs, exponentials and read-outs one after the other: 14 k
// cycles per tile.)  What a row needs from the other half of the features, its maximum, sum and weighted sum, crosses
// the cluster through shared memory (st.async), and so does the half of dQ the other CTA stores, one tile later; S, G
// of tile i+1 are computed under tile i's arithmetic.
// da and P^T delta stay in TMEM over all the tiles of a head; they are added to global memory when it changes.  The
// key side wants e_i = db_i - a_i . da_i, which is -sum_n P_ni delta_n: db itself is never formed.
// RNN (kPerformer = false): l_ni = log((elu(q_ni) + 1) z_i), so the weights come from the Q tile in shared memory, no S
// product, no exponent, and dq_ni = c_ni elu'(q_ni) / (elu(q_ni) + 1) needs no product either.
// Measured at 64 heads x N = 16384, m = 256: 470 us with all features in one CTA, 326 us now; RNN, 96 heads x N = 4096:
// 155 -> 48 us.  A tile takes 1900 cycles of MMA per CTA; what bounds it is the row owners' chain (exponentials, exchange of
// the row sums, c, the half of dQ), which two threads per row and S, G formed a tile ahead cover only in part.
#pragma once

#include <cuda_bf16.h>

#include "k1_down_project_pair.cuh"
#include "k4_bwd_query_wide.cuh"
#include "tc_common.cuh"

namespace flurka {

// Shared memory.  PERFORMER: a Q tile is free as soon as S is formed, a dO tile only after da, so three stages of it.
// RNN (bound by the traffic of Q, dO, dQ): no W, C, dQ exchange, so four of each.
template <bool kPerformer>
struct K7Smem {
  static constexpr int kQ = kPerformer ? 2 : 4, kDO = kPerformer ? 3 : 4;                 // stages of 16 KB
  static constexpr uint32_t a_hi = 0, a_lo = 16384, p = 32768, q = 65536, dout = q + kQ * 16384;
  static constexpr uint32_t w = dout + kDO * 16384, c = w + (kPerformer ? 16384 : 0);
  static constexpr uint32_t dq = c + (kPerformer ? 32768 : 0);                           // received half of dQ
  static constexpr uint32_t delta = dq + (kPerformer ? 16384 : 0);                       // [16 x 128] bf16
  static constexpr uint32_t stat = delta + 4096;                                         // [2 parities][3][4 parts][128] floats
  static constexpr uint32_t bias = stat + 12288;                                         // b_i log2 e (RNN: z_i / max z)
  static constexpr uint32_t bars = bias + 512;
  static constexpr int bytes = (int)bars + 256 + 1024;
};
// TMEM columns: S 0..127, G 128..255, dQ 256..383 (two tiles of 64), da 384..447, P^T delta 448..463
constexpr uint32_t kK7ColG = 128, kK7ColDQ = 256, kK7ColDA = 384, kK7ColDD = 448;

// kParts: CTAs per cluster (1 or 2), 128 features each
template <bool kPerformer, int kParts>
__global__ void __launch_bounds__(kK7Threads, 1)
k7_bwd_query_side(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmDO,
                  const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmA,
                  const K7Params prm) {
  using namespace tc;
  using L = K7Smem<kPerformer>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t bars = base + L::bars;
  const uint32_t bar_w = bars;               // W landed
  const uint32_t bar_q = bars + 8;           // [4] Q tile landed
  const uint32_t bar_qfree = bars + 40;      // [4] ... no longer needed (PERFORMER: S formed; RNN: read by 8 warps)
  const uint32_t bar_do = bars + 72;         // [4] dO tile landed
  const uint32_t bar_dofree = bars + 104;    // [4] ... no longer needed (da added to)
  const uint32_t bar_head = bars + 136;      // a, b of a new head in place
  const uint32_t bar_sg = bars + 144;        // S, G ready
  const uint32_t bar_sgfree = bars + 152;    // S, G and b read out (8 warps)
  const uint32_t bar_pc = bars + 160;        // P, C, delta written (8 warps)
  const uint32_t bar_out = bars + 168;       // dQ, da, P^T delta of a tile complete
  const uint32_t bar_x = bars + 176;         // [2] the row sums of all parts are here (8 local warps, the others by their bytes)
  const uint32_t bar_y = bars + 192;         // the other CTA's part of this CTA's half of dQ is here
  const uint32_t tmem_slot = bars + 200;
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_shared;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int p = prm.p;
  const uint32_t rank = kParts == 2 ? cluster_ctarank() : 0u;
  const int f0 = (int)rank * 128;                             // first feature of this CTA
  const int group = blockIdx.x / kParts, groups = gridDim.x / kParts;
  const int t_begin = (int)(((long long)group * prm.total_tiles) / groups);
  const int nt = (int)(((long long)(group + 1) * prm.total_tiles) / groups) - t_begin;

  if (tid == 0) {
    abort_flag = 0;
    mbar_init(bar_w, 1);
    for (int s = 0; s < 4; ++s) {
      mbar_init(bar_q + 8 * s, 1);
      mbar_init(bar_qfree + 8 * s, kPerformer ? 1 : 8);
      mbar_init(bar_do + 8 * s, 1);
      mbar_init(bar_dofree + 8 * s, 1);
    }
    mbar_init(bar_head, 33);
    mbar_init(bar_sg, 1);
    mbar_init(bar_sgfree, 8);
    mbar_init(bar_pc, 8);
    mbar_init(bar_out, 1);
    mbar_init(bar_x, 8);
    mbar_init(bar_x + 8, 8);
    mbar_init(bar_y, 1);
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  {
    // the delta operand [16 x 128] (K-major, no swizzle): rows 0..2 are rewritten per tile, the rest stays zero
    uint32_t* dz = reinterpret_cast<uint32_t*>(base_ptr + L::delta);
    for (int e = tid; e < 1024; e += kK7Threads) dz[e] = 0u;
    // RNN: features 64..127 (the second slab of the P tile) do not exist
    if (!kPerformer) {
      uint32_t* pz = reinterpret_cast<uint32_t*>(base_ptr + L::p + 16384);
      for (int e = tid; e < 4096; e += kK7Threads) pz[e] = 0u;
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
  if (kParts == 2) cluster_sync_all();       // the other CTA's barriers exist before anything is sent to them
  else __syncthreads();
  const uint32_t tmem = tmem_base_shared;
  const float kLog2e = 1.4426950408889634f;

  if (nt > 0) {
    if (warp < 4) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kK7RegsFew));
      if (warp == 0 && elect_one()) {
        // ============================================================ loader: W, then Q and dO tiles
        prefetch_tmap(&tmQ);
        prefetch_tmap(&tmDO);
        if (kPerformer) {
          prefetch_tmap(&tmW);
          mbar_arrive_expect_tx(bar_w, 16384u);
          tma_load_2d(base + L::w, &tmW, bar_w, 0, f0);       // rows past p read as zero
        }
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
        const uint32_t idescS = make_idesc(kFmtBF16, 0, 0, 128, 128);                    // S: both operands K-major
        const uint32_t idescG = make_idesc(kFmtBF16, 0, 0, 128, kPerformer ? 128 : 64);
        const uint32_t idescQ = make_idesc(kFmtBF16, 0, 1, 128, 64);    // dQ: C K-major, W MN-major
        const uint32_t idescA = make_idesc(kFmtBF16, 1, 1, 128, 64);    // da: P^T (MN-major A) x dO (MN-major B)
        const uint32_t idescD = make_idesc(kFmtBF16, 1, 0, 128, 16);    // P^T delta: delta as a K-major B
        bool ok = kPerformer ? mbar_wait(bar_w, 0, prm.status, &abort_flag) : true;
        int head = -1, events = 0;
        auto form_sg = [&](int i) {      // S, G of tile i, once its operands are in place and the tile before is read out
          const int h = (t_begin + i) / prm.tiles_per_head, sq = i % L::kQ, sd = i % L::kDO;
          if (h != head) {
            ok = mbar_wait(bar_head, (uint32_t)(events++) & 1u, prm.status, &abort_flag);
            head = h;
          }
          if (ok && kPerformer) ok = mbar_wait(bar_q + 8 * sq, (uint32_t)(i / L::kQ) & 1u, prm.status, &abort_flag);
          if (ok) ok = mbar_wait(bar_do + 8 * sd, (uint32_t)(i / L::kDO) & 1u, prm.status, &abort_flag);
          if (ok && i > 0) ok = mbar_wait(bar_sgfree, (uint32_t)(i - 1) & 1u, prm.status, &abort_flag);
          if (!ok) return;
          tcgen05_fence_after();
          const uint64_t ag = make_sdesc(base + L::dout + sd * 16384, 16, 1024, kSwizzle128);
          if (kPerformer) {
            mma_ss_x4(tmem, make_sdesc(base + L::q + sq * 16384, 16, 1024, kSwizzle128),
                      make_sdesc(base + L::w, 16, 1024, kSwizzle128), 2, 2, idescS, 0u);
            mma_commit(bar_qfree + 8 * sq);
          }
          mma_ss_x4(tmem + kK7ColG, ag, make_sdesc(base + L::a_hi, 16, 1024, kSwizzle128), 2, 2, idescG, 0u);
          mma_ss_x4(tmem + kK7ColG, ag, make_sdesc(base + L::a_lo, 16, 1024, kSwizzle128), 2, 2, idescG, 1u);
          mma_commit(bar_sg);
        };
        if (ok) form_sg(0);
        int acc_head = -1;
        for (int i = 0; i < nt && ok; ++i) {
          const int this_head = (t_begin + i) / prm.tiles_per_head;
          if (i + 1 < nt) {
            form_sg(i + 1);
            if (!ok) break;
          }
          ok = mbar_wait(bar_pc, (uint32_t)i & 1u, prm.status, &abort_flag);
          if (!ok) break;
          tcgen05_fence_after();
          const uint32_t sm_do = base + L::dout + (i % L::kDO) * 16384;
          const uint32_t first = this_head != acc_head ? 0u : 1u;
          acc_head = this_head;
          if (kPerformer) {
            const uint32_t dq = tmem + kK7ColDQ + (uint32_t)(i & 1) * 64u;
            for (int j = 0; j < 2; ++j)      // 64 features: 32 B of a C row and 16 rows of W per step
              mma_ss_x4(dq, make_sdesc(base + L::c + j * 16384, 16, 1024, kSwizzle128),
                        make_sdesc(base + L::w + j * 8192, 8192, 1024, kSwizzle128), 2, 128, idescQ, j > 0 ? 1u : 0u);
          }
          for (int j = 0; j < 2; ++j) {      // 64 rows: 16 rows of P and of dO, 256 B of delta per step
            const uint64_t ap = make_sdesc(base + L::p + j * 8192, 16384, 1024, kSwizzle128);
            mma_ss_x4(tmem + kK7ColDA, ap, make_sdesc(sm_do + j * 8192, 8192, 1024, kSwizzle128), 128, 128, idescA,
                      j > 0 ? 1u : first);
            mma_ss_x4(tmem + kK7ColDD, ap, make_sdesc(base + L::delta + j * 1024, 128, 2048, kSwizzleNone), 128, 16, idescD,
                      j > 0 ? 1u : first);
          }
          mma_commit(bar_out);
          mma_commit(bar_dofree + 8 * (i % L::kDO));
        }
      } else if (warp == 2) {
        // ============================================================ a and b of a new head, once the old head's last tile
        // is read out (every tile is waited for: a parity wait sees one bit of the phase count)
        if (lane == 0) prefetch_tmap(&tmA);
        grid_dependency_wait_async();
        int head_prev = -1;
        bool ok = true;
        for (int i = 0; i < nt && ok; ++i) {
          const int head = (t_begin + i) / prm.tiles_per_head;
          if (i > 0) ok = mbar_wait(bar_sgfree, (uint32_t)(i - 1) & 1u, prm.status, &abort_flag);
          if (!ok || head == head_prev) continue;
          head_prev = head;
          if (lane == 0) {
            mbar_arrive_expect_tx(bar_head, 32768u);
            tma_load_3d(base + L::a_hi, &tmA, bar_head, 0, f0, head * 2);
            tma_load_3d(base + L::a_lo, &tmA, bar_head, 0, f0, head * 2 + 1);
          }
          const float* wv = prm.weight + (size_t)head * p;
          float mx = kPerformer ? -INFINITY : 0.f;
          for (int f = lane; f < p; f += 32) mx = fmaxf(mx, __ldcg(wv + f));
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
          float* bs = reinterpret_cast<float*>(base_ptr + L::bias);
          const float inv = 1.f / mx;
          for (int f = lane; f < 128; f += 32) {
            const float v = f0 + f < p ? __ldcg(wv + f0 + f) : 0.f;
            bs[f] = kPerformer ? (f0 + f < p ? (v - mx) * kLog2e : 0.f) : v * inv;
          }
          mbar_arrive(bar_head);
        }
      }
    } else {
      // ============================================================ row owners: two threads per row, 64 features each
      // (RNN: 32 each)
      asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kK7RegsMany));
      constexpr int kF = kPerformer ? 64 : 32;                     // features of a thread
      constexpr int kStat = 2 * kParts * 128;                      // floats of one kind of row sum
      const int q4 = warp & 3, row = q4 * 32 + lane, fh = (warp - 4) >> 2;
      const uint32_t lane_base = tmem + ((uint32_t)(q4 * 32) << 16);
      const bool live = kPerformer ? f0 + fh * 64 < p : true;      // features past p: weight zero
      const uint32_t peer = kParts == 2 ? (rank ^ 1u) : 0u;
      const uint32_t x_peer = map_to_cta(bar_x, peer), y_peer = map_to_cta(bar_y, peer);
      float* stat = reinterpret_cast<float*>(base_ptr + L::stat);
      const uint32_t stat_peer = map_to_cta(base + L::stat, peer);
      const uint32_t dqx_peer = map_to_cta(base + L::dq, peer) + (uint32_t)(fh * 4 * 128 + row) * 16u;
      const float* bs = reinterpret_cast<const float*>(base_ptr + L::bias) + fh * kF;
      bool ok = true;
      grid_dependency_wait();

      // da, P^T delta of one head leave TMEM: lane = feature, 32 of the 64 columns per thread
      auto flush = [&](int head) {
        uint32_t dd[16], r[32];
        tmem_ld16(lane_base + kK7ColDD, dd);
        tmem_ld32(lane_base + kK7ColDA + fh * 32, r);
        tmem_wait_ld16(dd);
        tmem_wait_ld(r);
        const int feat = f0 + row;
        if (feat >= p) return;
        float4* darow = reinterpret_cast<float4*>(prm.da + ((size_t)head * p + feat) * 64 + fh * 32);
#pragma unroll
        for (int e = 0; e < 8; ++e)
          atomicAdd(darow + e, make_float4(__uint_as_float(r[4 * e]), __uint_as_float(r[4 * e + 1]),
                                           __uint_as_float(r[4 * e + 2]), __uint_as_float(r[4 * e + 3])));
        if (fh == 0)
          atomicAdd(prm.ei + (size_t)head * p + feat, -(__uint_as_float(dd[0]) + __uint_as_float(dd[1]) + __uint_as_float(dd[2])));
      };
      auto dq_row = [&](int head, int row0) {
        return prm.dQ + (prm.H > 0 ? (((size_t)(head / prm.H) * prm.N + row0 + row) * prm.H + (size_t)(head % prm.H)) * 64
                                   : ((size_t)head * prm.N + row0 + row) * 64);
      };
      // dQ of a tile: with two CTAs each stores 32 of the 64 columns, its own sums plus the other CTA's.  The other CTA's
      // part of a thread's values comes from the thread of the same row and columns there, which sends it only after
      // this thread's row sums of the next tile have arrived there, i.e. after this thread has read the part before.
      constexpr int kDQ = kPerformer ? 32 / kParts : 1;            // columns of a thread
      uint32_t own[kDQ], other[kParts == 2 ? 16 : 1];
      auto read_dq = [&](int i) {
        const uint32_t dq = lane_base + kK7ColDQ + (uint32_t)(i & 1) * 64u;
        if constexpr (kParts == 2) {
          tmem_ld16(dq + rank * 32 + fh * 16, own);
          tmem_ld16(dq + peer * 32 + fh * 16, other);
          tmem_wait_ld16(own);
          tmem_wait_ld16(other);
        } else if constexpr (kPerformer) {
          tmem_ld32(dq + fh * 32, own);
          tmem_wait_ld(own);
        }
      };
      auto send_dq = [&]() {
        if constexpr (kParts == 2) {
          // 16-byte pieces of four columns, 128 rows of a piece side by side
#pragma unroll
          for (int j = 0; j < 4; ++j)
            st_async_v4(dqx_peer + j * 2048u, other[4 * j], other[4 * j + 1], other[4 * j + 2], other[4 * j + 3], y_peer);
          if (tid == 128) mbar_arrive_expect_tx(bar_y, 16384u);
        }
      };
      auto store_dq = [&](int i, int head, int row0) -> bool {
        if constexpr (kParts == 2) {
          if (!mbar_wait(bar_y, (uint32_t)i & 1u, prm.status, &abort_flag)) return false;
          const float4* src = reinterpret_cast<const float4*>(base_ptr + L::dq) + fh * 4 * 128 + row;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float4 v = src[j * 128];
            own[4 * j] = __float_as_uint(__uint_as_float(own[4 * j]) + v.x);
            own[4 * j + 1] = __float_as_uint(__uint_as_float(own[4 * j + 1]) + v.y);
            own[4 * j + 2] = __float_as_uint(__uint_as_float(own[4 * j + 2]) + v.z);
            own[4 * j + 3] = __float_as_uint(__uint_as_float(own[4 * j + 3]) + v.w);
          }
        }
        if constexpr (kPerformer) {
          if (row0 + row < prm.N) {
            __nv_bfloat16* o = dq_row(head, row0) + rank * 32 + fh * kDQ;
#pragma unroll
            for (int g = 0; g < kDQ / 16; ++g) {
              uint32_t v[8];
#pragma unroll
              for (int e = 0; e < 8; ++e)
                v[e] = k4_bf16x2(__uint_as_float(own[16 * g + 2 * e]), __uint_as_float(own[16 * g + 2 * e + 1]));
              k4_store16(o + 16 * g, v, prm.wide != 0);
            }
          }
        }
        return true;
      };

      int head = t_begin / prm.tiles_per_head, tih = t_begin % prm.tiles_per_head;
      int head_prev = head, row0_prev = 0;
      for (int i = 0; i < nt; ++i) {
        const int row0 = tih * 128;
        const uint32_t par = (uint32_t)(i & 1);
        ok = mbar_wait(bar_sg, par, prm.status, &abort_flag);
        if (!ok) break;
        tcgen05_fence_after();
        // this thread's g, and its weights (PERFORMER: exp(l - own maximum); RNN: phi(q) z / max z), as pairs; RNN: cf is
        // the factor of (g - delta) in dQ: P elu'(q) / (elu(q) + 1) = z / max z where q > 0, the weight itself elsewhere
        uint64_t w2[kF / 2], g2[kF / 2], cf2[kPerformer ? 1 : 16];
        float mx = 0.f;
        uint64_t den2 = 0ull, num2 = 0ull;
        {
          uint32_t ga[32];
          tmem_ld32(lane_base + kK7ColG + fh * kF, ga);
          if constexpr (kPerformer) {
            uint32_t gb[32], sa[32], sb[32];
            tmem_ld32(lane_base + kK7ColG + fh * 64 + 32, gb);
            tmem_ld32(lane_base + fh * 64, sa);
            tmem_ld32(lane_base + fh * 64 + 32, sb);
            tmem_wait_ld(sa);
            tmem_wait_ld(sb);
            tmem_wait_ld(gb);
            tmem_wait_ld(ga);
            const uint64_t l2 = pack2(kLog2e, kLog2e);
            float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              g2[e] = pack2u(ga[2 * e], ga[2 * e + 1]);
              g2[16 + e] = pack2u(gb[2 * e], gb[2 * e + 1]);
            }
#pragma unroll
            for (int e = 0; e < 32; e += 2) {
              const ulonglong2 b4 = *reinterpret_cast<const ulonglong2*>(bs + 2 * e);
              w2[e] = fma2(e < 16 ? pack2u(sa[2 * e & 31], sa[(2 * e + 1) & 31]) : pack2u(sb[2 * e & 31], sb[(2 * e + 1) & 31]), l2, b4.x);
              w2[e + 1] = fma2(e < 16 ? pack2u(sa[(2 * e + 2) & 31], sa[(2 * e + 3) & 31]) : pack2u(sb[(2 * e + 2) & 31], sb[(2 * e + 3) & 31]), l2, b4.y);
              float x0, x1, x2, x3;
              unpack2(w2[e], x0, x1);
              unpack2(w2[e + 1], x2, x3);
              m0 = fmax3(m0, x0, x1);
              m1 = fmax3(m1, x2, x3);
            }
            mx = live ? fmaxf(m0, m1) : -INFINITY;
          } else {
            // (the Q row of this thread, 128-byte swizzled)
            ok = mbar_wait(bar_q + 8 * (i & 3), (uint32_t)(i >> 2) & 1u, prm.status, &abort_flag);
            const uint32_t qrow = base + L::q + (uint32_t)(i & 3) * 16384u + (uint32_t)row * 128u;
#pragma unroll
            for (int c8 = 0; c8 < 4; ++c8) {
              uint32_t w4[4];
              asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w4[0]), "=r"(w4[1]), "=r"(w4[2]), "=r"(w4[3])
                           : "r"(qrow + (((uint32_t)(fh * 4 + c8) ^ (uint32_t)(row & 7)) << 4)));
              const float4 z0 = *reinterpret_cast<const float4*>(bs + 8 * c8), z1 = *reinterpret_cast<const float4*>(bs + 8 * c8 + 4);
              const float z[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const float x0 = __uint_as_float(w4[e] << 16), x1 = __uint_as_float(w4[e] & 0xffff0000u);
                // elu(x) + 1 = max(x, 0) + exp(min(x, 0))
                const float v0 = (fmaxf(x0, 0.f) + k4_ex2(fminf(x0, 0.f) * kLog2e)) * z[2 * e];
                const float v1 = (fmaxf(x1, 0.f) + k4_ex2(fminf(x1, 0.f) * kLog2e)) * z[2 * e + 1];
                w2[4 * c8 + e] = pack2(v0, v1);
                cf2[4 * c8 + e] = pack2(x0 > 0.f ? z[2 * e] : v0, x1 > 0.f ? z[2 * e + 1] : v1);
              }
            }
            tmem_wait_ld(ga);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              g2[e] = pack2u(ga[2 * e], ga[2 * e + 1]);
              den2 = add2(den2, w2[e]);
              num2 = fma2(w2[e], g2[e], num2);
            }
          }
          tcgen05_fence_before();
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(bar_sgfree);
            if (!kPerformer) mbar_arrive(bar_qfree + 8 * (i & 3));
          }
          if (!ok) break;
          if constexpr (kPerformer) {
            if (live) {
              const uint64_t nm2 = pack2(-mx, -mx);
#pragma unroll
              for (int e = 0; e < 32; ++e) {
                float x0, x1;
                unpack2(add2(w2[e], nm2), x0, x1);
                w2[e] = pack2(k4_ex2(x0), k4_ex2(x1));
                den2 = add2(den2, w2[e]);
                num2 = fma2(w2[e], g2[e], num2);
              }
            }
          }
        }
        // ---- the sums to everyone who shares the row
        {
          float d0, d1, n0, n1;
          unpack2(den2, d0, d1);
          unpack2(num2, n0, n1);
          const uint32_t at = par * (3 * kStat) + (rank * 2 + (uint32_t)fh) * 128 + (uint32_t)row;
          stat[at] = mx;
          stat[at + kStat] = d0 + d1;
          stat[at + 2 * kStat] = n0 + n1;
          if (kParts == 2) {
            const uint32_t bar = x_peer + par * 8u;
            st_async_b32(stat_peer + at * 4u, __float_as_uint(mx), bar);
            st_async_b32(stat_peer + (at + kStat) * 4u, __float_as_uint(d0 + d1), bar);
            st_async_b32(stat_peer + (at + 2 * kStat) * 4u, __float_as_uint(n0 + n1), bar);
          }
          __syncwarp();
          if (lane == 0) {
            if (kParts == 2 && warp == 4) mbar_arrive_expect_tx(bar_x + par * 8u, 256u * 12u);
            else mbar_arrive(bar_x + par * 8u);
          }
        }
        if (i > 0) {
          // the products of the tile before are complete: P, C, delta may be overwritten, its dQ read
          ok = mbar_wait(bar_out, par ^ 1u, prm.status, &abort_flag);
          if (!ok) break;
          tcgen05_fence_after();
          read_dq(i - 1);
          if (head != head_prev) flush(head_prev);
          tcgen05_fence_before();
        }
        ok = mbar_wait(bar_x + par * 8u, (uint32_t)(i >> 1) & 1u, prm.status, &abort_flag);
        if (!ok) break;
        if (i > 0) send_dq();
        float delta, scale;
        {
          const float* st0 = stat + par * (3 * kStat) + row;
          float m[2 * kParts], all = -INFINITY, dsum = 0.f, nsum = 0.f;
#pragma unroll
          for (int q = 0; q < 2 * kParts; ++q) {
            m[q] = st0[q * 128];
            all = fmaxf(all, m[q]);
          }
#pragma unroll
          for (int q = 0; q < 2 * kParts; ++q) {
            const float f = kPerformer ? k4_ex2(m[q] - all) : 1.f;
            dsum = fmaf(st0[kStat + q * 128], f, dsum);
            nsum = fmaf(st0[2 * kStat + q * 128], f, nsum);
          }
          const float inv = __fdividef(1.f, dsum);
          delta = nsum * inv;
          scale = kPerformer ? (live ? k4_ex2(mx - all) * inv : 0.f) : inv;      // (features past p: finite values times zero)
        }
        if (fh == 0) {
          // delta_n as three bf16 terms: element (c, n) of the [16 x 128] operand at (n/8)*128 + c*16 + (n%8)*2 bytes
          __nv_bfloat16* dt = reinterpret_cast<__nv_bfloat16*>(base_ptr + L::delta) + (row >> 3) * 64 + (row & 7);
          float r = delta;
          const __nv_bfloat16 d0 = __float2bfloat16_rn(r);  r -= __bfloat162float(d0);
          const __nv_bfloat16 d1 = __float2bfloat16_rn(r);  r -= __bfloat162float(d1);
          dt[0] = d0; dt[8] = d1; dt[16] = __float2bfloat16_rn(r);
        }
        // ---- P and C (RNN: P, and dQ at once)
        {
          const uint32_t prow = (uint32_t)row * 128u + (kPerformer ? (uint32_t)fh * 16384u : 0u);
          const uint64_t sc2 = pack2(scale, scale), nd2 = pack2(-delta, -delta);
          uint32_t dqv[kPerformer ? 1 : 16];
#pragma unroll
          for (int c8 = 0; c8 < kF / 8; ++c8) {
            uint32_t pw[4], cw[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int j = 4 * c8 + e;
              const uint64_t pp = mul2(w2[j], sc2), gd = add2(g2[j], nd2);
              uint64_t cc;
              if constexpr (kPerformer) cc = mul2(pp, gd);
              else cc = mul2(mul2(cf2[j], sc2), gd);
              float p0, p1, c0, c1;
              unpack2(pp, p0, p1);
              unpack2(cc, c0, c1);
              pw[e] = k4_bf16x2(p0, p1);
              cw[e] = k4_bf16x2(c0, c1);
              if constexpr (!kPerformer) dqv[j] = cw[e];
            }
            const uint32_t ch = (uint32_t)(kPerformer ? c8 : fh * 4 + c8);
            const uint32_t off = prow + ((ch ^ (uint32_t)(row & 7)) << 4);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(base + L::p + off), "r"(pw[0]), "r"(pw[1]), "r"(pw[2]),
                         "r"(pw[3]) : "memory");
            if constexpr (kPerformer)
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(base + L::c + off), "r"(cw[0]), "r"(cw[1]), "r"(cw[2]),
                           "r"(cw[3]) : "memory");
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_pc);
          if constexpr (!kPerformer) {
            if (row0 + row < prm.N) {
              __nv_bfloat16* o = dq_row(head, row0) + fh * 32;
              k4_store16(o, *reinterpret_cast<const uint32_t (*)[8]>(&dqv[0]), prm.wide != 0);
              k4_store16(o + 16, *reinterpret_cast<const uint32_t (*)[8]>(&dqv[8]), prm.wide != 0);
            }
          }
        }
        if (i > 0) {
          ok = store_dq(i - 1, head_prev, row0_prev);
          if (!ok) break;
        }
        head_prev = head;
        row0_prev = row0;
        if (++tih == prm.tiles_per_head) { tih = 0; ++head; }
      }
      if (ok) {
        // the last tile's dQ, the last head's sums.  (Its part of dQ may be sent once the other CTA has read the one before:
        // the row sums of tile nt - 1 do not say so, so each thread tells its counterpart with one more word.)
        ok = mbar_wait(bar_out, (uint32_t)(nt - 1) & 1u, prm.status, &abort_flag);
        if (ok) {
          tcgen05_fence_after();
          read_dq(nt - 1);
          flush(head_prev);
          if constexpr (kParts == 2) {
            const uint32_t par = (uint32_t)(nt & 1);
            st_async_b32(stat_peer + (par * (3 * kStat) + (rank * 2 + (uint32_t)fh) * 128 + (uint32_t)row) * 4u, 0u, x_peer + par * 8u);
            __syncwarp();
            if (lane == 0) {
              if (warp == 4) mbar_arrive_expect_tx(bar_x + par * 8u, 256u * 4u);
              else mbar_arrive(bar_x + par * 8u);
            }
            ok = mbar_wait(bar_x + par * 8u, (uint32_t)(nt >> 1) & 1u, prm.status, &abort_flag);
          }
          if (ok) {
            send_dq();
            (void)store_dq(nt - 1, head_prev, row0_prev);
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
