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
// the cluster through shared memory, and so does the half of dQ the other CTA stores; the exchange of tile i's
// sums and of tile i-1's dQ shares one barrier, and S, G of tile i+1 are computed under tile i's arithmetic.
// da and P^T delta stay in TMEM over all the tiles of a head; they are added to global memory when it changes; db
// comes from them there.
// RNN (kPerformer = false): l_ni = log((elu(q_ni) + 1) z_i), so the weights come from the Q tile in shared memory, no S
// product, no exponent, and dq_ni = c_ni elu'(q_ni) / (elu(q_ni) + 1) needs no product either.
// K7_FIG
#pragma once

#include <cuda_bf16.h>

#include "k1_down_project_pair.cuh"
#include "k4_bwd_query_side.cuh"
#include "tc_common.cuh"

namespace flurka {

struct K7Params {
  int N, p, BH, H;              // H > 0: Q, dO, dQ are [B,N,H,d]; H == 0: [BH,N,d]; d = 64
  int tiles_per_head, total_tiles;
  const float* weight;          // [BH][p]      b_i (RNN: z_i)
  const float* a32;             // [BH][p][64]  a_i (fp32)
  __nv_bfloat16* dQ;
  float* da;                    // [BH][p][64]  added to
  float* db;                    // [BH][p]      added to
  int* status;
};

constexpr int kK7Threads = 384;                // loader, MMA issuer, two idle warps; two warpgroups of row owners
// registers: 384 threads x 168 at launch = 128 x 72 + 256 x 216
constexpr int kK7RegsFew = 72, kK7RegsMany = 216;
// shared memory: W 16 KB | a_hi 16 KB | a_lo 16 KB | 2 x (Q tile 16 KB, dO tile 16 KB) | P tile 32 KB | C tile 32 KB |
// received halves of dQ 2 x 16 KB | delta operand 4 KB | row sums 2 x 6 KB | b_i (z_i) 512 B | barriers
constexpr uint32_t kK7W = 0, kK7AHi = 16384, kK7ALo = 32768, kK7In = 49152, kK7P = 114688, kK7C = 147456, kK7DQ = 180224,
                   kK7Delta = 212992, kK7Stat = 217088, kK7Bias = 229376, kK7Bars = 229888;
constexpr int kK7SmemBytes = 229888 + 128 + 1024;
// TMEM columns: S 0..127, G 128..255, dQ 256..383 (two tiles of 64), da 384..447, P^T delta 448..463
constexpr uint32_t kK7ColG = 128, kK7ColDQ = 256, kK7ColDA = 384, kK7ColDD = 448;

namespace tc {
// Stores to a CTA of the cluster that count their bytes on a barrier there: whoever waits for that barrier sees the
// data, and the sender needs no fence (a release at cluster scope would wait for its global stores too: 1400 cycles
// per tile here).
__device__ __forceinline__ void st_async_b32(uint32_t addr, uint32_t v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d), "r"(bar) : "memory");
}
// brings a tile into L2 ahead of its load
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap* m, int x, int y, int z) {
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global [%0, {%1, %2, %3}];"
               ::"l"(reinterpret_cast<uint64_t>(m)), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_wait_ld16(uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
        "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
      :
      : "memory");
}
}  // namespace tc

// kParts: CTAs per cluster (1 or 2), 128 features each
template <bool kPerformer, int kParts>
__global__ void __launch_bounds__(kK7Threads, 1)
k7_bwd_query_side(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmDO,
                  const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmA,
                  const K7Params prm) {
  using namespace tc;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t bars = base + kK7Bars;
  const uint32_t bar_w = bars;               // W landed
  const uint32_t bar_in = bars + 8;          // [2] Q, dO of a tile landed
  const uint32_t bar_free = bars + 24;       // [2] every product that reads them is complete
  const uint32_t bar_head = bars + 40;       // a, b of a new head in place
  const uint32_t bar_sg = bars + 48;         // S, G ready
  const uint32_t bar_sgfree = bars + 56;     // S, G read out (8 warps)
  const uint32_t bar_pc = bars + 64;         // P, C, delta written (8 warps)
  const uint32_t bar_out = bars + 72;        // dQ, da, P^T delta of a tile complete
  const uint32_t bar_x = bars + 80;          // [2] the row sums of all parts (8 local warps; the other CTA's, and its half
                                             //     of the dQ before, by their bytes) are here
  const uint32_t tmem_slot = bars + 96;
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
    for (int s = 0; s < 2; ++s) {
      mbar_init(bar_in + 8 * s, 1);
      mbar_init(bar_free + 8 * s, 1);
    }
    mbar_init(bar_head, 33);
    mbar_init(bar_sg, 1);
    mbar_init(bar_sgfree, 8);
    mbar_init(bar_pc, 8);
    mbar_init(bar_out, 1);
    mbar_init(bar_x, 8);
    mbar_init(bar_x + 8, 8);
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  {
    // the delta operand [16 x 128] (K-major, no swizzle): rows 0..2 are rewritten per tile, the rest stays zero
    uint32_t* dz = reinterpret_cast<uint32_t*>(base_ptr + kK7Delta);
    for (int e = tid; e < 1024; e += kK7Threads) dz[e] = 0u;
    // RNN: features 64..127 (the second slab of the P tile) do not exist
    if (!kPerformer) {
      uint32_t* pz = reinterpret_cast<uint32_t*>(base_ptr + kK7P + 16384);
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
    if (warp == 0) {
      // ============================================================ loader: W, Q and dO tiles, a and b per head
      if (lane == 0) {
        prefetch_tmap(&tmQ);
        prefetch_tmap(&tmDO);
        prefetch_tmap(&tmA);
        if (kPerformer) {
          prefetch_tmap(&tmW);
          mbar_arrive_expect_tx(bar_w, 16384u);
          tma_load_2d(base + kK7W, &tmW, bar_w, 0, f0);       // rows past p read as zero
        }
      }
      __syncwarp();
      grid_dependency_wait_async();
      bool ok = true;
      int head_prev = -1;
      for (int i = 0; i < nt && ok; ++i) {
        const int tile = t_begin + i, head = tile / prm.tiles_per_head;
        const uint32_t st = (uint32_t)(i & 1);
        // (before the head's wait: tile i-2 is complete then, and the one bit of a parity wait is enough for tile i-1)
        if (i >= 2) ok = mbar_wait(bar_free + 8 * st, (uint32_t)((i >> 1) - 1) & 1u, prm.status, &abort_flag);
        if (!ok) break;
        if (head != head_prev) {
          // S, G of the old head's last tile are complete and read, and so is its b: its operands may go
          if (i > 0) ok = mbar_wait(bar_sgfree, (uint32_t)(i - 1) & 1u, prm.status, &abort_flag);
          if (!ok) break;
          if (lane == 0) {
            mbar_arrive_expect_tx(bar_head, 32768u);
            tma_load_3d(base + kK7AHi, &tmA, bar_head, 0, f0, head * 2);
            tma_load_3d(base + kK7ALo, &tmA, bar_head, 0, f0, head * 2 + 1);
          }
          const float* wv = prm.weight + (size_t)head * p;
          float mx = kPerformer ? -INFINITY : 0.f;
          for (int f = lane; f < p; f += 32) mx = fmaxf(mx, __ldcg(wv + f));
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
          float* bs = reinterpret_cast<float*>(base_ptr + kK7Bias);
          const float inv = 1.f / mx;
          for (int f = lane; f < 128; f += 32) {
            const float v = f0 + f < p ? __ldcg(wv + f0 + f) : 0.f;
            bs[f] = kPerformer ? (f0 + f < p ? (v - mx) * kLog2e : 0.f) : v * inv;
          }
          mbar_arrive(bar_head);
          head_prev = head;
        }
        if (lane == 0) {
          const int row0 = (tile % prm.tiles_per_head) * 128;
          const int x = prm.H > 0 ? (head % prm.H) * 64 : 0, z = prm.H > 0 ? head / prm.H : head;
          const uint32_t dst = base + kK7In + st * 32768u;
          mbar_arrive_expect_tx(bar_in + 8 * st, 32768u);
          tma_load_3d(dst, &tmQ, bar_in + 8 * st, x, row0, z);
          tma_load_3d(dst + 16384, &tmDO, bar_in + 8 * st, x, row0, z);
          // a stage only becomes free when the tile two before is done: the next tile's data wait in L2 by then
          if (i + 1 < nt && (int)rank == (i & 1) * (kParts - 1)) {
            const int tile1 = tile + 1, head1 = tile1 / prm.tiles_per_head, row1 = (tile1 % prm.tiles_per_head) * 128;
            const int x1 = prm.H > 0 ? (head1 % prm.H) * 64 : 0, z1 = prm.H > 0 ? head1 / prm.H : head1;
            tma_prefetch_3d(&tmQ, x1, row1, z1);
            tma_prefetch_3d(&tmDO, x1, row1, z1);
          }
        }
        __syncwarp();
      }
      if (!ok && lane == 0) {
        // loads in flight still land in this CTA's shared memory: give them their (bounded) time
        for (int s = 0; s < 2; ++s) {
          (void)mbar_wait(bar_in + 8 * s, 0, prm.status, &abort_flag);
          (void)mbar_wait(bar_in + 8 * s, 1, prm.status, &abort_flag);
        }
      }
    } else if (warp == 1) {
      if (elect_one()) {
        // ============================================================ MMA issuer
        const uint32_t idescS = make_idesc(kFmtBF16, 0, 0, 128, 128);                    // S: both operands K-major
        const uint32_t idescG = make_idesc(kFmtBF16, 0, 0, 128, kPerformer ? 128 : 64);
        const uint32_t idescQ = make_idesc(kFmtBF16, 0, 1, 128, 64);    // dQ: C K-major, W MN-major
        const uint32_t idescA = make_idesc(kFmtBF16, 1, 1, 128, 64);    // da: P^T (MN-major A) x dO (MN-major B)
        const uint32_t idescD = make_idesc(kFmtBF16, 1, 0, 128, 16);    // P^T delta: delta as a K-major B
        auto issue_sg = [&](int i) {
          tcgen05_fence_after();
          const uint32_t sm_q = base + kK7In + (uint32_t)(i & 1) * 32768u;
          if (kPerformer)
            mma_ss_x4(tmem, make_sdesc(sm_q, 16, 1024, kSwizzle128), make_sdesc(base + kK7W, 16, 1024, kSwizzle128), 2, 2,
                      idescS, 0u);
          const uint64_t ag = make_sdesc(sm_q + 16384, 16, 1024, kSwizzle128);
          mma_ss_x4(tmem + kK7ColG, ag, make_sdesc(base + kK7AHi, 16, 1024, kSwizzle128), 2, 2, idescG, 0u);
          mma_ss_x4(tmem + kK7ColG, ag, make_sdesc(base + kK7ALo, 16, 1024, kSwizzle128), 2, 2, idescG, 1u);
          mma_commit(bar_sg);
        };
        bool ok = kPerformer ? mbar_wait(bar_w, 0, prm.status, &abort_flag) : true;
        int head = -1, events = 0;
        auto enter_tile = [&](int i) {      // the operands of tile i's S, G are in place
          const int h = (t_begin + i) / prm.tiles_per_head;
          if (h != head) {
            if (ok) ok = mbar_wait(bar_head, (uint32_t)(events++) & 1u, prm.status, &abort_flag);
            head = h;
          }
          if (ok) ok = mbar_wait(bar_in + 8 * (i & 1), (uint32_t)(i >> 1) & 1u, prm.status, &abort_flag);
          if (ok && i > 0) ok = mbar_wait(bar_sgfree, (uint32_t)(i - 1) & 1u, prm.status, &abort_flag);
        };
        enter_tile(0);
        if (ok) issue_sg(0);
        int acc_head = -1;
        for (int i = 0; i < nt && ok; ++i) {
          const int this_head = (t_begin + i) / prm.tiles_per_head;
          if (i + 1 < nt) {
            enter_tile(i + 1);
            if (!ok) break;
            issue_sg(i + 1);
          }
          ok = mbar_wait(bar_pc, (uint32_t)i & 1u, prm.status, &abort_flag);
          if (!ok) break;
          tcgen05_fence_after();
          const uint32_t sm_do = base + kK7In + (uint32_t)(i & 1) * 32768u + 16384u;
          const uint32_t first = this_head != acc_head ? 0u : 1u;
          acc_head = this_head;
          if (kPerformer) {
            const uint32_t dq = tmem + kK7ColDQ + (uint32_t)(i & 1) * 64u;
            for (int j = 0; j < 2; ++j)      // 64 features: 32 B of a C row and 16 rows of W per step
              mma_ss_x4(dq, make_sdesc(base + kK7C + j * 16384, 16, 1024, kSwizzle128),
                        make_sdesc(base + kK7W + j * 8192, 8192, 1024, kSwizzle128), 2, 128, idescQ, j > 0 ? 1u : 0u);
          }
          for (int j = 0; j < 2; ++j) {      // 64 rows: 16 rows of P and of dO, 256 B of delta per step
            const uint64_t ap = make_sdesc(base + kK7P + j * 8192, 16384, 1024, kSwizzle128);
            mma_ss_x4(tmem + kK7ColDA, ap, make_sdesc(sm_do + j * 8192, 8192, 1024, kSwizzle128), 128, 128, idescA,
                      j > 0 ? 1u : first);
            mma_ss_x4(tmem + kK7ColDD, ap, make_sdesc(base + kK7Delta + j * 1024, 128, 2048, kSwizzleNone), 128, 16, idescD,
                      j > 0 ? 1u : first);
          }
          mma_commit(bar_out);
          mma_commit(bar_free + 8 * (i & 1));
        }
      }
    }
    } else {
      // ============================================================ row owners: two threads per row, 64 features each
      // (RNN: 32 each)
      asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kK7RegsMany));
      const int q4 = warp & 3, row = q4 * 32 + lane, fh = (warp - 4) >> 2;
      const uint32_t lane_base = tmem + ((uint32_t)(q4 * 32) << 16);
      const bool live = kPerformer ? f0 + fh * 64 < p : true;      // features past p: weight zero
      constexpr int kF = kPerformer ? 64 : 32;                     // features of a thread
      const uint32_t peer = kParts == 2 ? (rank ^ 1u) : 0u;
      const uint32_t x_peer = map_to_cta(bar_x, peer);
      float* stat = reinterpret_cast<float*>(base_ptr + kK7Stat);  // [2 parities][3][2 kParts][128]
      const uint32_t stat_peer = map_to_cta(base + kK7Stat, peer);
      const uint32_t dqx_peer = map_to_cta(base + kK7DQ, peer);
      const float* bs = reinterpret_cast<const float*>(base_ptr + kK7Bias) + fh * kF;
      bool ok = true;
      grid_dependency_wait();

      // da, P^T delta of one head leave TMEM: lane = feature, 32 of the 64 columns per thread
      auto flush = [&](int head) {
        tcgen05_fence_after();
        uint32_t dd[16], r[32];
        tmem_ld16(lane_base + kK7ColDD, dd);
        tmem_ld32(lane_base + kK7ColDA + fh * 32, r);
        tmem_wait_ld16(dd);
        tmem_wait_ld(r);
        tcgen05_fence_before();
        const int feat = f0 + row;
        if (feat >= p) return;
        const float4* arow = reinterpret_cast<const float4*>(prm.a32 + ((size_t)head * p + feat) * 64 + fh * 32);
        float4* darow = reinterpret_cast<float4*>(prm.da + ((size_t)head * p + feat) * 64 + fh * 32);
        float dot = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float4 av = __ldcg(arow + e);
          const float4 v = make_float4(__uint_as_float(r[4 * e]), __uint_as_float(r[4 * e + 1]), __uint_as_float(r[4 * e + 2]),
                                       __uint_as_float(r[4 * e + 3]));
          dot = fmaf(av.x, v.x, fmaf(av.y, v.y, fmaf(av.z, v.z, fmaf(av.w, v.w, dot))));
          atomicAdd(darow + e, v);
        }
        if (fh == 0) dot -= __uint_as_float(dd[0]) + __uint_as_float(dd[1]) + __uint_as_float(dd[2]);
        atomicAdd(prm.db + (size_t)head * p + feat, dot);
      };
      auto dq_row = [&](int head, int row0) {
        return prm.dQ + (prm.H > 0 ? (((size_t)(head / prm.H) * prm.N + row0 + row) * prm.H + (size_t)(head % prm.H)) * 64
                                   : ((size_t)head * prm.N + row0 + row) * 64);
      };
      // dQ of a tile: with two CTAs each stores 32 of the 64 columns, its own sums plus the other CTA's
      constexpr int kDQ = kPerformer ? 32 / kParts : 1;            // columns of a thread
      uint32_t own[kDQ];
      auto read_dq = [&](int i) {
        const uint32_t dq = lane_base + kK7ColDQ + (uint32_t)(i & 1) * 64u;
        if constexpr (kParts == 2) {
          uint32_t out[16];
          tmem_ld16(dq + rank * 32 + fh * 16, own);
          tmem_ld16(dq + peer * 32 + fh * 16, out);
          tmem_wait_ld16(own);
          tmem_wait_ld16(out);
          // 16-byte pieces of four columns, 128 rows of a piece side by side
          const uint32_t dst = dqx_peer + (uint32_t)(i & 1) * 16384u + (uint32_t)(fh * 4 * 128 + row) * 16u;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            st_async_v4(dst + j * 2048u, out[4 * j], out[4 * j + 1], out[4 * j + 2], out[4 * j + 3], x_peer + (uint32_t)((i + 1) & 1) * 8u);
        } else if constexpr (kPerformer) {
          tmem_ld32(dq + fh * 32, own);
          tmem_wait_ld(own);
        }
      };
      auto store_dq = [&](int i, int head, int row0) {
        if (row0 + row >= prm.N) return;
        if constexpr (kParts == 2) {
          const float4* src = reinterpret_cast<const float4*>(base_ptr + kK7DQ + (uint32_t)(i & 1) * 16384u) + fh * 4 * 128 + row;
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
          __nv_bfloat16* o = dq_row(head, row0) + rank * 32 + fh * kDQ;
#pragma unroll
          for (int g = 0; g < kDQ / 8; ++g) {
            uint32_t v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = k4_bf16x2(__uint_as_float(own[8 * g + 2 * e]), __uint_as_float(own[8 * g + 2 * e + 1]));
            *reinterpret_cast<uint4*>(o + 8 * g) = make_uint4(v[0], v[1], v[2], v[3]);
          }
        }
      };
      // exchange i: the sums of tile i (unless i == nt) and the dQ halves of tile i - 1 (unless i == 0)
      auto exchange = [&](int i) -> bool {
        const uint32_t bar = bar_x + (uint32_t)(i & 1) * 8u;
        __syncwarp();
        if (lane == 0) {
          if (kParts == 2 && warp == 4) mbar_arrive_expect_tx(bar, (i < nt ? 256u * 12u : 0u) + (i > 0 ? 16384u : 0u));
          else mbar_arrive(bar);
        }
        return mbar_wait(bar, (uint32_t)(i >> 1) & 1u, prm.status, &abort_flag);
      };

      int head = t_begin / prm.tiles_per_head, tih = t_begin % prm.tiles_per_head;
      int head_prev = head, row0_prev = 0;
      for (int i = 0; i < nt && ok; ++i) {
        const int row0 = tih * 128;
        const uint32_t par = (uint32_t)(i & 1);
        const uint32_t sm_q = base + kK7In + par * 32768u;
        ok = mbar_wait(bar_sg, par, prm.status, &abort_flag);
        if (!ok) break;
        tcgen05_fence_after();
        uint32_t s[kF], g[kF];
        float ratio[kPerformer ? 1 : 32];
        {
          uint32_t (&g0)[32] = *reinterpret_cast<uint32_t (*)[32]>(&g[0]);
          tmem_ld32(lane_base + kK7ColG + fh * kF, g0);
          if constexpr (kPerformer) {
            uint32_t (&g1)[32] = *reinterpret_cast<uint32_t (*)[32]>(&g[32]);
            uint32_t (&s0)[32] = *reinterpret_cast<uint32_t (*)[32]>(&s[0]);
            uint32_t (&s1)[32] = *reinterpret_cast<uint32_t (*)[32]>(&s[32]);
            tmem_ld32(lane_base + kK7ColG + fh * 64 + 32, g1);
            tmem_ld32(lane_base + fh * 64, s0);
            tmem_ld32(lane_base + fh * 64 + 32, s1);
            tmem_wait_ld(s0);
            tmem_wait_ld(s1);
            tmem_wait_ld(g1);
          }
          tmem_wait_ld(g0);
        }
        // ---- this thread's part of the row: weights relative to its own maximum, their sum, their sum with g
        float mx = 0.f, den = 0.f, num = 0.f;
        if constexpr (kPerformer) {
          mx = -INFINITY;
          if (live) {
            float m1 = -INFINITY;
#pragma unroll
            for (int e = 0; e < 64; e += 4) {
              const float4 b4 = *reinterpret_cast<const float4*>(bs + e);
              const float x0 = fmaf(__uint_as_float(s[e]), kLog2e, b4.x), x1 = fmaf(__uint_as_float(s[e + 1]), kLog2e, b4.y);
              const float x2 = fmaf(__uint_as_float(s[e + 2]), kLog2e, b4.z), x3 = fmaf(__uint_as_float(s[e + 3]), kLog2e, b4.w);
              mx = fmax3(mx, x0, x1);
              m1 = fmax3(m1, x2, x3);
              s[e] = __float_as_uint(x0);
              s[e + 1] = __float_as_uint(x1);
              s[e + 2] = __float_as_uint(x2);
              s[e + 3] = __float_as_uint(x3);
            }
            mx = fmaxf(mx, m1);
          }
          // (b_i is read here: only now may the next head's replace it)
          tcgen05_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_sgfree);
          if (live) {
#pragma unroll
            for (int e = 0; e < 64; ++e) {
              const float w = k4_ex2(__uint_as_float(s[e]) - mx);
              s[e] = __float_as_uint(w);
              den += w;
              num = fmaf(w, __uint_as_float(g[e]), num);
            }
          }
        } else {
          // (elu(q) + 1) z / max z of this thread's 32 columns of the (128-byte swizzled) Q row, and elu'(q) / (elu(q) + 1)
#pragma unroll
          for (int c8 = 0; c8 < 4; ++c8) {
            const uint32_t ch = (uint32_t)(fh * 4 + c8);
            uint32_t w4[4];
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w4[0]), "=r"(w4[1]), "=r"(w4[2]), "=r"(w4[3])
                         : "r"(sm_q + (uint32_t)row * 128u + ((ch ^ (uint32_t)(row & 7)) << 4)));
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const float x = __uint_as_float((e & 1) ? (w4[e >> 1] & 0xffff0000u) : (w4[e >> 1] << 16));
              const int f = 8 * c8 + e;
              const float phi = fmaxf(x, 0.f) + k4_ex2(fminf(x, 0.f) * kLog2e);      // elu(x) + 1
              const float w = phi * bs[f];
              ratio[f] = x > 0.f ? __fdividef(1.f, phi) : 1.f;
              s[f] = __float_as_uint(w);
              den += w;
              num = fmaf(w, __uint_as_float(g[f]), num);
            }
          }
          tcgen05_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_sgfree);
        }
        // ---- to everyone who shares the row
        {
          const uint32_t part = rank * 2 + (uint32_t)fh;
          const uint32_t at = par * (3 * 2 * kParts * 128) + part * 128 + (uint32_t)row;
          stat[at] = mx;
          stat[at + 2 * kParts * 128] = den;
          stat[at + 4 * kParts * 128] = num;
          if (kParts == 2) {
            const uint32_t bar = x_peer + par * 8u;
            st_async_b32(stat_peer + at * 4u, __float_as_uint(mx), bar);
            st_async_b32(stat_peer + (at + 2 * kParts * 128) * 4u, __float_as_uint(den), bar);
            st_async_b32(stat_peer + (at + 4 * kParts * 128) * 4u, __float_as_uint(num), bar);
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
        ok = exchange(i);
        if (!ok) break;
        float delta, scale;
        {
          const float* st0 = stat + par * (3 * 2 * kParts * 128) + row;
          float m[2 * kParts], all = -INFINITY, dsum = 0.f, nsum = 0.f;
#pragma unroll
          for (int q = 0; q < 2 * kParts; ++q) {
            m[q] = st0[q * 128];
            all = fmaxf(all, m[q]);
          }
#pragma unroll
          for (int q = 0; q < 2 * kParts; ++q) {
            const float f = k4_ex2(m[q] - all);
            dsum = fmaf(st0[(2 * kParts + q) * 128], f, dsum);
            nsum = fmaf(st0[(4 * kParts + q) * 128], f, nsum);
          }
          const float inv = 1.f / dsum;
          delta = nsum * inv;
          scale = live ? k4_ex2(mx - all) * inv : 0.f;         // (features past p: finite values times zero)
        }
        if (fh == 0) {
          // delta_n as three bf16 terms: element (c, n) of the [16 x 128] operand at (n/8)*128 + c*16 + (n%8)*2 bytes
          __nv_bfloat16* dt = reinterpret_cast<__nv_bfloat16*>(base_ptr + kK7Delta) + (row >> 3) * 64 + (row & 7);
          float r = delta;
          const __nv_bfloat16 d0 = __float2bfloat16_rn(r);  r -= __bfloat162float(d0);
          const __nv_bfloat16 d1 = __float2bfloat16_rn(r);  r -= __bfloat162float(d1);
          dt[0] = d0; dt[8] = d1; dt[16] = __float2bfloat16_rn(r);
        }
        // ---- P and C (RNN: P, and dQ at once)
        {
          const uint32_t prow = (uint32_t)row * 128u + (kPerformer ? (uint32_t)fh * 16384u : 0u);
          __nv_bfloat16* dqp = dq_row(head, row0) + fh * 32;
          const bool store = row0 + row < prm.N;
#pragma unroll
          for (int c8 = 0; c8 < kF / 8; ++c8) {
            uint32_t pw[4], cw[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int j = 8 * c8 + 2 * e;
              const float p0 = __uint_as_float(s[j]) * scale, p1 = __uint_as_float(s[j + 1]) * scale;
              pw[e] = k4_bf16x2(p0, p1);
              float c0 = p0 * (__uint_as_float(g[j]) - delta), c1 = p1 * (__uint_as_float(g[j + 1]) - delta);
              if constexpr (!kPerformer) {
                c0 *= ratio[j];
                c1 *= ratio[j + 1];
              }
              cw[e] = k4_bf16x2(c0, c1);
            }
            const uint32_t ch = (uint32_t)(kPerformer ? c8 : fh * 4 + c8);
            const uint32_t off = prow + ((ch ^ (uint32_t)(row & 7)) << 4);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(base + kK7P + off), "r"(pw[0]), "r"(pw[1]), "r"(pw[2]),
                         "r"(pw[3]) : "memory");
            if constexpr (kPerformer)
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(base + kK7C + off), "r"(cw[0]), "r"(cw[1]), "r"(cw[2]),
                           "r"(cw[3]) : "memory");
            else if (store)
              *reinterpret_cast<uint4*>(dqp + 8 * c8) = make_uint4(cw[0], cw[1], cw[2], cw[3]);
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_pc);
        if (i > 0) store_dq(i - 1, head_prev, row0_prev);
        head_prev = head;
        row0_prev = row0;
        if (++tih == prm.tiles_per_head) { tih = 0; ++head; }
      }
      if (ok) {
        // the last tile's dQ, the last head's sums
        ok = mbar_wait(bar_out, (uint32_t)(nt - 1) & 1u, prm.status, &abort_flag);
        if (ok) {
          tcgen05_fence_after();
          read_dq(nt - 1);
          flush(head_prev);
          ok = exchange(nt);
          if (ok) store_dq(nt - 1, head_prev, row0_prev);
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
