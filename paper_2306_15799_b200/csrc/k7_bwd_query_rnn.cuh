// Backward of the query side on tensor cores for RNN (bf16, d = 64 and 128).
//
// The formulas are those of k8_bwd_query_units.cuh with the feature map of Section 4 (arxiv 2306.15799), phi(x) = elu(x) + 1,
// whose features are the d entries of the row itself: the weights P_ni = phi(q_ni) z_i / sum and
// dq_ni = c_ni phi'(q_ni) / phi(q_ni) come straight from the Q tile, without a product.  Per tile of 128 rows
//     G = dO a^T  (a as two bf16 terms),   da += P^T dO,   (P^T delta) += P^T [delta_hi delta_mid delta_lo]
// are tcgen05 MMAs with fp32 accumulators, P a bf16 tile in shared memory (the MN-major A operand), delta_n = sum_i P_ni g_ni.
// da and P^T delta stay in TMEM over all the tiles of a head.
//
// d = 64 moves 48 KB and takes 1150 cycles of MMA per tile, but a tile's chain from its loads to da is four times that: two
// groups of eight warps (two threads per row) have a tile each.
// kSplit (sequence lengths that are no multiple of 8, and d = 128): P as two bf16 terms, 16 to 17 bits.  With
// d = 64 the second term takes rows 64..127 of the A operand, which has 128 rows either way: da's lanes 64..127 are its share
// of the sums, and the flush adds both.  With d = 128 it is a second product; one group (the operands fill shared memory).
#pragma once

#include <cuda_bf16.h>

#include "k1_down_project_pair.cuh"
#include "k4_bwd_query_wide.cuh"
#include "tc_common.cuh"

namespace flurka {

template <int kD> struct K7Shape {
  static constexpr int kGroups = kD == 64 ? 2 : 1;
  static constexpr int kThreads = 128 + 256 * kGroups;     // loader, MMA issuer, head operands, an idle warp; the row owners
  static constexpr int kRegsFew = kD == 64 ? 32 : 72, kRegsMany = kD == 64 ? 112 : 216;
  // shared memory: stages of a Q and of a dO tile (kD = 128: Q(i+1) is loaded once Q(i) is read, dO(i+1) once da(i) is formed)
  static constexpr int kQ = kD == 64 ? 3 : 1, kDO = kD == 64 ? 4 : 1;
  static constexpr uint32_t kTile = 256u * kD;             // bytes of 128 rows
  static constexpr uint32_t a_hi = 0, a_lo = 2u * kD * kD, p = 2 * a_lo;       // a: [d features x d] per term
  static constexpr uint32_t kP = 32768u * (kD / 64);       // P per group: d = 64 both terms, d = 128 32 KB per term
  static constexpr uint32_t q = p + kGroups * kP, dout = q + kQ * kTile;
  static constexpr uint32_t delta = dout + kDO * kTile;    // [16 x 128] bf16 per group
  static constexpr uint32_t stat = delta + kGroups * 4096; // per group, of two tiles: [2][2 halves][128] floats
  static constexpr uint32_t bias = stat + kGroups * 4096;  // z_i / max z of three heads
  static constexpr uint32_t bars = bias + 1536;
  static constexpr int bytes = (int)bars + 256 + 1024;
};

template <int kD, bool kSplit>
__global__ void __launch_bounds__(K7Shape<kD>::kThreads, 1)
k7_bwd_query_rnn(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmDO,
                 const __grid_constant__ CUtensorMap tmA, const K7Params prm) {
  using namespace tc;
  using L = K7Shape<kD>;
  constexpr int kGroups = L::kGroups, kSlabs = kD / 64, kF = kD / 2;       // kF: features of a thread
  constexpr uint32_t kColG = 0, kColDA = 128, kColDD = kColDA + kD;        // G of group g at 64 g
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t bars = base + L::bars;
  const uint32_t bar_q = bars;               // [3] Q tile landed
  const uint32_t bar_qfree = bars + 24;      // [3] ... read by 8 warps
  const uint32_t bar_do = bars + 48;         // [4] dO tile landed
  const uint32_t bar_dofree = bars + 80;     // [4] ... da added to
  const uint32_t bar_req = bars + 112;       // every product with the old head's a is complete: load the next
  const uint32_t bar_head = bars + 120;      // a, z of a new head in place
  const uint32_t bar_flush = bars + 128;     // da, P^T delta of the old head read out (8 warps)
  // one per group:
  const uint32_t bar_g = bars + 136;         // G ready
  const uint32_t bar_gfree = bars + 152;     // G read out (8 warps)
  const uint32_t bar_x = bars + 168;         // the row sums of both halves are here (8 warps)
  const uint32_t bar_p = bars + 184;         // P, delta written (8 warps)
  const uint32_t bar_out = bars + 200;       // da, P^T delta complete
  const uint32_t tmem_slot = bars + 216;
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_shared;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t_begin = (int)(((long long)blockIdx.x * prm.total_tiles) / gridDim.x);
  const int nt = (int)(((long long)(blockIdx.x + 1) * prm.total_tiles) / gridDim.x) - t_begin;

  if (tid == 0) {
    abort_flag = 0;
    for (int s = 0; s < L::kQ; ++s) {
      mbar_init(bar_q + 8 * s, 1);
      mbar_init(bar_qfree + 8 * s, 8);
    }
    for (int s = 0; s < L::kDO; ++s) {
      mbar_init(bar_do + 8 * s, 1);
      mbar_init(bar_dofree + 8 * s, 1);
    }
    mbar_init(bar_req, 1);
    mbar_init(bar_head, 33);
    mbar_init(bar_flush, 8);
    for (int g = 0; g < kGroups; ++g) {
      mbar_init(bar_g + 8 * g, 1);
      mbar_init(bar_gfree + 8 * g, 8);
      mbar_init(bar_x + 8 * g, 8);
      mbar_init(bar_p + 8 * g, 8);
      mbar_init(bar_out + 8 * g, 1);
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
    for (int e = tid; e < 1024 * kGroups; e += L::kThreads) dz[e] = 0u;
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
  const float kLog2e = 1.4426950408889634f;

  if (nt > 0) {
    if (warp < 4) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(L::kRegsFew));
      if (warp == 0 && elect_one()) {
        // ============================================================ loader of the Q and dO tiles
        prefetch_tmap(&tmQ);
        prefetch_tmap(&tmDO);
        bool ok = true;
        int head = t_begin / prm.tiles_per_head, tih = t_begin % prm.tiles_per_head;
        int nq = 0, nd = 0;                                    // loads issued
        for (int i = 0; i < nt; ++i) {
          const int x = prm.H > 0 ? (head % prm.H) * kD : 0, z = prm.H > 0 ? head / prm.H : head;
          const int sq = i % L::kQ, sd = i % L::kDO;
          if (i >= L::kQ) ok = mbar_wait(bar_qfree + 8 * sq, (uint32_t)(i / L::kQ - 1) & 1u, prm.status, &abort_flag);
          if (!ok) break;
          mbar_arrive_expect_tx(bar_q + 8 * sq, L::kTile);
          for (int s = 0; s < kSlabs; ++s)
            tma_load_3d(base + L::q + sq * L::kTile + s * 16384, &tmQ, bar_q + 8 * sq, x + s * 64, tih * 128, z);
          ++nq;
          if (i >= L::kDO) ok = mbar_wait(bar_dofree + 8 * sd, (uint32_t)(i / L::kDO - 1) & 1u, prm.status, &abort_flag);
          if (!ok) break;
          mbar_arrive_expect_tx(bar_do + 8 * sd, L::kTile);
          for (int s = 0; s < kSlabs; ++s)
            tma_load_3d(base + L::dout + sd * L::kTile + s * 16384, &tmDO, bar_do + 8 * sd, x + s * 64, tih * 128, z);
          ++nd;
          if (++tih == prm.tiles_per_head) { tih = 0; ++head; }
          if (L::kDO == 1 && i + 1 < nt) {
            // the next tiles are loaded when they are wanted: let them wait in L2
            const int x1 = prm.H > 0 ? (head % prm.H) * kD : 0, z1 = prm.H > 0 ? head / prm.H : head;
            for (int s = 0; s < kSlabs; ++s) {
              tma_prefetch_3d(&tmQ, x1 + s * 64, tih * 128, z1);
              tma_prefetch_3d(&tmDO, x1 + s * 64, tih * 128, z1);
            }
          }
        }
        if (!ok) {
          // loads in flight still land in this CTA's shared memory: wait for them (bounded)
          for (int e = max(0, nq - L::kQ); e < nq; ++e)
            (void)mbar_wait(bar_q + 8 * (e % L::kQ), (uint32_t)(e / L::kQ) & 1u, prm.status, &abort_flag);
          for (int e = max(0, nd - L::kDO); e < nd; ++e)
            (void)mbar_wait(bar_do + 8 * (e % L::kDO), (uint32_t)(e / L::kDO) & 1u, prm.status, &abort_flag);
        }
      } else if (warp == 1 && elect_one()) {
        // ============================================================ MMA issuer
        const uint32_t idescG = make_idesc(kFmtBF16, 0, 0, 128, kD);     // G: both operands K-major
        const uint32_t idescA = make_idesc(kFmtBF16, 1, 1, 128, kD);     // da: P^T (MN-major A) x dO (MN-major B)
        const uint32_t idescD = make_idesc(kFmtBF16, 1, 0, 128, 16);     // P^T delta: delta as a K-major B
        bool ok = true;
        int head = -1, events = 0, flushes = 0;
        auto form_g = [&](int i) {       // G of tile i
          const int g = i % kGroups, h = (t_begin + i) / prm.tiles_per_head, sd = i % L::kDO;
          if (h != head) {
            if (i > 0) ok = mbar_wait(bar_g + 8 * ((i - 1) % kGroups), (uint32_t)((i - 1) / kGroups) & 1u, prm.status, &abort_flag);
            if (!ok) return;
            mbar_arrive(bar_req);
            ok = mbar_wait(bar_head, (uint32_t)(events++) & 1u, prm.status, &abort_flag);
            head = h;
          }
          if (ok) ok = mbar_wait(bar_do + 8 * sd, (uint32_t)(i / L::kDO) & 1u, prm.status, &abort_flag);
          if (ok && i >= kGroups) ok = mbar_wait(bar_gfree + 8 * g, (uint32_t)(i / kGroups - 1) & 1u, prm.status, &abort_flag);
          if (!ok) return;
          tcgen05_fence_after();
          const uint32_t dst = tmem + kColG + (uint32_t)g * 64u;
          for (int s = 0; s < kSlabs; ++s) {
            const uint64_t ag = make_sdesc(base + L::dout + sd * L::kTile + s * 16384, 16, 1024, kSwizzle128);
            mma_ss_x4(dst, ag, make_sdesc(base + L::a_hi + s * (kD * 128), 16, 1024, kSwizzle128), 2, 2, idescG, s > 0 ? 1u : 0u);
            mma_ss_x4(dst, ag, make_sdesc(base + L::a_lo + s * (kD * 128), 16, 1024, kSwizzle128), 2, 2, idescG, 1u);
          }
          mma_commit(bar_g + 8 * g);
        };
        // d = 64: G of a group's next tile is formed as soon as the group has read this one's, before this tile's P is there
        constexpr int kAhead = L::kDO > 1 ? kGroups : 0;
        for (int i = 0; i < max(kAhead, 1) && i < nt && ok; ++i) form_g(i);
        int acc_head = -1;
        for (int i = 0; i < nt && ok; ++i) {
          const int g = i % kGroups, this_head = (t_begin + i) / prm.tiles_per_head, sd = i % L::kDO;
          if (kAhead > 0 && i + kAhead < nt) {
            form_g(i + kAhead);
            if (!ok) break;
          }
          ok = mbar_wait(bar_p + 8 * g, (uint32_t)(i / kGroups) & 1u, prm.status, &abort_flag);
          if (!ok) break;
          uint32_t first = 1u;
          if (this_head != acc_head) {
            // the sums of the head before have left TMEM
            if (acc_head >= 0) ok = mbar_wait(bar_flush, (uint32_t)(flushes++) & 1u, prm.status, &abort_flag);
            if (!ok) break;
            acc_head = this_head;
            first = 0u;
          }
          tcgen05_fence_after();
          const uint32_t sm_p = base + L::p + (uint32_t)g * L::kP, sm_d = base + L::delta + (uint32_t)g * 4096u;
          for (int term = 0; term < (kD == 128 && kSplit ? 2 : 1); ++term)
            for (int j = 0; j < 2; ++j) {      // 64 rows: 16 rows of P and of dO, 256 B of delta per step; slabs 16 KB apart
              const uint64_t ap = make_sdesc(sm_p + term * 32768 + j * 8192, 16384, 1024, kSwizzle128);
              mma_ss_x4(tmem + kColDA, ap, make_sdesc(base + L::dout + sd * L::kTile + j * 8192, 16384, 1024, kSwizzle128), 128,
                        128, idescA, first);
              mma_ss_x4(tmem + kColDD, ap, make_sdesc(sm_d + j * 1024, 128, 2048, kSwizzleNone), 128, 16, idescD, first);
              first = 1u;
            }
          mma_commit(bar_dofree + 8 * sd);
          mma_commit(bar_out + 8 * g);
          if (kAhead == 0 && i + 1 < nt) form_g(i + 1);
        }
      } else if (warp == 2) {
        // ============================================================ a and z of a new head, when the issuer asks
        if (lane == 0) prefetch_tmap(&tmA);
        grid_dependency_wait_async();
        const int head0 = t_begin / prm.tiles_per_head, head1 = (t_begin + nt - 1) / prm.tiles_per_head;
        bool ok = true;
        for (int head = head0; head <= head1; ++head) {
          ok = mbar_wait(bar_req, (uint32_t)(head - head0) & 1u, prm.status, &abort_flag);
          if (!ok) break;
          if (lane == 0) {
            mbar_arrive_expect_tx(bar_head, 4u * kD * kD);
            for (int s = 0; s < kSlabs; ++s) {
              tma_load_3d(base + L::a_hi + s * (kD * 128), &tmA, bar_head, s * 64, 0, head * 2);
              tma_load_3d(base + L::a_lo + s * (kD * 128), &tmA, bar_head, s * 64, 0, head * 2 + 1);
            }
          }
          const float* wv = prm.weight + (size_t)head * kD;
          float mx = 0.f;
          for (int f = lane; f < kD; f += 32) mx = fmaxf(mx, __ldcg(wv + f));
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
          // (three heads in turn: the issuer asks for the first tile of a head once it has seen P of the tile three before it)
          float* bs = reinterpret_cast<float*>(base_ptr + L::bias) + (head - head0) % 3 * 128;
          const float inv = 1.f / mx;
          for (int f = lane; f < kD; f += 32) bs[f] = __ldcg(wv + f) * inv;
          mbar_arrive(bar_head);
        }
      }
    } else {
      // ============================================================ row owners: two threads per row, half of the features each
      asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(L::kRegsMany));
      const int g = (warp - 4) >> 3;
      const int q4 = warp & 3, fh = ((warp - 4) >> 2) & 1, row = q4 * 32 + lane;
      const uint32_t lane_base = tmem + ((uint32_t)(q4 * 32) << 16);
      const uint32_t prow = base + L::p + (uint32_t)g * L::kP + (uint32_t)row * 128u;
      const uint32_t swz = (uint32_t)(row & 7);
      bool ok = true;
      grid_dependency_wait();

      // da, P^T delta of one head leave TMEM: lane = feature (d = 64: lanes 64..127 the second term of P), half of the columns
      auto flush = [&](int head) {
        tcgen05_fence_after();
        const int feat = kD == 64 ? row & 63 : row;
        const bool live = kD == 128 || kSplit || row < 64;
        uint32_t r[16];
#pragma unroll 1
        for (int c = 0; c < kD / 2; c += 16) {
          tmem_ld16(lane_base + kColDA + fh * (kD / 2) + c, r);
          tmem_wait_ld16(r);
          if (live) {
            float4* darow = reinterpret_cast<float4*>(prm.da + ((size_t)head * kD + feat) * kD + fh * (kD / 2) + c);
#pragma unroll
            for (int e = 0; e < 4; ++e)
              atomicAdd(darow + e, make_float4(__uint_as_float(r[4 * e]), __uint_as_float(r[4 * e + 1]),
                                               __uint_as_float(r[4 * e + 2]), __uint_as_float(r[4 * e + 3])));
          }
        }
        if (fh == 0) {
          tmem_ld16(lane_base + kColDD, r);
          tmem_wait_ld16(r);
          if (live)
            atomicAdd(prm.ei + (size_t)head * kD + feat, -(__uint_as_float(r[0]) + __uint_as_float(r[1]) + __uint_as_float(r[2])));
        }
        tcgen05_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_flush);
      };

      const int head0 = t_begin / prm.tiles_per_head;
      int ended = -1;                          // the head that ends with this group's last tile: its sums leave TMEM after da
      for (int i = g; i < nt; i += kGroups) {
        const int head = (t_begin + i) / prm.tiles_per_head, tih = (t_begin + i) - head * prm.tiles_per_head;
        const uint32_t par = (uint32_t)(i / kGroups) & 1u;
        // (G's barrier first: with it z of the tile's head is in place)
        ok = mbar_wait(bar_g + 8 * g, par, prm.status, &abort_flag);
        if (ok) ok = mbar_wait(bar_q + 8 * (i % L::kQ), (uint32_t)(i / L::kQ) & 1u, prm.status, &abort_flag);
        if (!ok) break;
        tcgen05_fence_after();
        // this thread's weights phi(q) z / max z and g, as pairs; two bits of `pos` per pair: q > 0
        uint64_t w2[kF / 2], g2[kF / 2];
        uint32_t pos[kF / 32];
        uint64_t den2 = 0ull, num2 = 0ull;
        const float* bs = reinterpret_cast<const float*>(base_ptr + L::bias) + (head - head0) % 3 * 128 + fh * kF;
#pragma unroll
        for (int h = 0; h < kF / 32; ++h) {
          uint32_t ga[32];
          tmem_ld32(lane_base + kColG + g * 64 + fh * kF + h * 32, ga);
          pos[h] = 0u;
          const uint32_t qrow = base + L::q + (uint32_t)(i % L::kQ) * L::kTile + (kD == 128 ? (uint32_t)fh * 16384u : 0u) + (uint32_t)row * 128u;
#pragma unroll
          for (int c8 = 0; c8 < 4; ++c8) {
            const uint32_t ch = kD == 128 ? h * 4 + c8 : fh * 4 + c8;
            uint32_t w4[4];
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w4[0]), "=r"(w4[1]), "=r"(w4[2]), "=r"(w4[3])
                         : "r"(qrow + ((ch ^ swz) << 4)));
            const float4 z0 = *reinterpret_cast<const float4*>(bs + h * 32 + 8 * c8), z1 = *reinterpret_cast<const float4*>(bs + h * 32 + 8 * c8 + 4);
            const float z[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float x0 = __uint_as_float(w4[e] << 16), x1 = __uint_as_float(w4[e] & 0xffff0000u);
              // elu(x) + 1 = max(x, 0) + exp(min(x, 0))
              w2[h * 16 + 4 * c8 + e] = pack2((fmaxf(x0, 0.f) + k4_ex2(fminf(x0, 0.f) * kLog2e)) * z[2 * e],
                                              (fmaxf(x1, 0.f) + k4_ex2(fminf(x1, 0.f) * kLog2e)) * z[2 * e + 1]);
              pos[h] |= (x0 > 0.f ? 1u : 0u) << (8 * c8 + 2 * e) | (x1 > 0.f ? 2u : 0u) << (8 * c8 + 2 * e);
            }
          }
          tmem_wait_ld(ga);
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            g2[h * 16 + e] = pack2u(ga[2 * e], ga[2 * e + 1]);
            den2 = add2(den2, w2[h * 16 + e]);
            num2 = fma2(w2[h * 16 + e], g2[h * 16 + e], num2);
          }
        }
        tcgen05_fence_before();
        // (the sums of two tiles in turn: those of the tile two before are read by whoever has left those of the tile before)
        float* stat = reinterpret_cast<float*>(base_ptr + L::stat) + g * 1024 + par * 512;
        {
          float d0, d1, n0, n1;
          unpack2(den2, d0, d1);
          unpack2(num2, n0, n1);
          stat[fh * 128 + row] = d0 + d1;
          stat[256 + fh * 128 + row] = n0 + n1;
        }
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(bar_gfree + 8 * g);
          mbar_arrive(bar_qfree + 8 * (i % L::kQ));
          mbar_arrive(bar_x + 8 * g);
        }
        ok = mbar_wait(bar_x + 8 * g, par, prm.status, &abort_flag);
        if (!ok) break;
        const float inv = __fdividef(1.f, stat[row] + stat[128 + row]);
        const float delta = (stat[256 + row] + stat[384 + row]) * inv;
        // the products of the group's tile before are complete: P, delta may be overwritten
        if (i >= kGroups) ok = mbar_wait(bar_out + 8 * g, par ^ 1u, prm.status, &abort_flag);
        if (!ok) break;
        if (ended >= 0) flush(ended);
        if (fh == 0) {
          // delta_n as three bf16 terms: element (c, n) of the [16 x 128] operand at (n/8)*128 + c*16 + (n%8)*2 bytes
          __nv_bfloat16* dt = reinterpret_cast<__nv_bfloat16*>(base_ptr + L::delta) + g * 2048 + (row >> 3) * 64 + (row & 7);
          float r = delta;
          const __nv_bfloat16 d0 = __float2bfloat16_rn(r);  r -= __bfloat162float(d0);
          const __nv_bfloat16 d1 = __float2bfloat16_rn(r);  r -= __bfloat162float(d1);
          dt[0] = d0; dt[8] = d1; dt[16] = __float2bfloat16_rn(r);
        }
        // ---- P, and dQ at once: c phi'(q) / phi(q) = P (g - delta) where q <= 0 (phi' = phi), z / max z / sum (g - delta) elsewhere
        const int n = tih * 128 + row;
        __nv_bfloat16* orow = prm.dQ + (prm.H > 0 ? (((size_t)(head / prm.H) * prm.N + n) * prm.H + (size_t)(head % prm.H)) * kD
                                                  : ((size_t)head * prm.N + n) * kD) + fh * kF;
        const uint64_t sc2 = pack2(inv, inv), nd2 = pack2(-delta, -delta);
#pragma unroll
        for (int c16 = 0; c16 < kF / 16; ++c16) {
          uint32_t dqv[8];
#pragma unroll
          for (int c8 = 2 * c16; c8 < 2 * c16 + 2; ++c8) {
            uint32_t pw[4];
            [[maybe_unused]] uint32_t lo[4];
            const float4 z0 = *reinterpret_cast<const float4*>(bs + 8 * c8), z1 = *reinterpret_cast<const float4*>(bs + 8 * c8 + 4);
            const float z[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int j = 4 * c8 + e;
              float w0, w1, p0, p1, c0, c1;
              unpack2(w2[j], w0, w1);
              unpack2(mul2(w2[j], sc2), p0, p1);
              pw[e] = k4_bf16x2(p0, p1);
              if constexpr (kSplit)
                lo[e] = k4_bf16x2(p0 - __uint_as_float(pw[e] << 16), p1 - __uint_as_float(pw[e] & 0xffff0000u));
              const uint32_t bits = pos[j >> 4] >> (2 * (j & 15));
              const uint64_t cf2 = pack2((bits & 1u) ? z[2 * e] : w0, (bits & 2u) ? z[2 * e + 1] : w1);
              unpack2(mul2(mul2(cf2, sc2), add2(g2[j], nd2)), c0, c1);
              dqv[4 * (c8 & 1) + e] = k4_bf16x2(c0, c1);
            }
            const uint32_t ch = (uint32_t)(kD == 128 ? c8 : fh * 4 + c8);
            const uint32_t to = prow + (kD == 128 ? (uint32_t)fh * 16384u : 0u) + ((ch ^ swz) << 4);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(to), "r"(pw[0]), "r"(pw[1]), "r"(pw[2]), "r"(pw[3])
                         : "memory");
            if constexpr (kSplit)
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(to + (kD == 128 ? 32768u : 16384u)), "r"(lo[0]),
                           "r"(lo[1]), "r"(lo[2]), "r"(lo[3]) : "memory");
          }
          if (n < prm.N) k4_store16(orow + 16 * c16, dqv, prm.wide != 0);
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_p + 8 * g);
        ended = i + 1 == nt || tih + 1 == prm.tiles_per_head ? head : -1;
      }
      if (ok && ended >= 0 && mbar_wait(bar_out + 8 * g, (uint32_t)((nt - 1 - g) / kGroups) & 1u, prm.status, &abort_flag)) flush(ended);
      if (warp == 4 && lane == 0) grid_launch_dependents();
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

}  // namespace flurka
