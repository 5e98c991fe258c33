// Stage 3 on tensor cores for PERFORMER with d = 64: the query feature map, the associative product and the row division
// (arxiv 2306.15799, Eq. (2); normalisation as in Appendix D), one pass over Q.  The formulas and operands are those of
// k3_query_side.cuh (which serves d = 128 and RNN); what differs is how the work is cut.
//
// Four groups of four warps (one row per thread) walk every fourth tile of 128 query rows, 64 features at a time: S = Q W^T +
// 1 b^T (64 TMEM columns) is read once, into registers; p = exp(S - r) goes back over it as fp16, and O += p a accumulates
// in the other 64 columns of the group's 128.  r is the row's maximum over the first 64 features of the tile; it is raised,
// and O and the sum rescaled, only when a later block's maximum lies more than 2^15 above it (p must stay below fp16's
// 2^16).  The block with the largest b_i comes first, so that this is rare: b decides where the maximum is.  (r at or
// below the maximum costs no precision: fp16 and fp32 are relative, and small weights only come to lie further from
// fp16's subnormal range.)
// With four warps per scheduler in different phases the special-function unit and the FMA pipe of one meet the TMEM reads,
// barrier round trips and read-outs of the others.  Two groups with 256 features at a time (k3_query_side) left them
// half idle: a group's tile took 7390 cycles at m = 256, 3160 of which were exponentials, at 12 cycles each because one
// warp alone does not overlap them (7 with two).  Two groups with 128 features in registers took 7900.
// Measured, two groups -> this kernel: 120 -> 107 us at 64 heads x N = 16384 with m = 256, 64.5 -> 56 us at 96 heads x
// N = 8192 with m = 128, 8.1 -> 7.4 us at 2 heads x N = 1024.  A tile with m = 256 takes 3200 cycles of an SM, 1480 of them
// tensor (N = 64 costs 48 cycles per step with A in shared memory and 32 with A in TMEM: the reads of A bind), 1800
// special-function; what is left is latency: a block's round trip through two chains of products is 1000 cycles.  Three groups
// with S of the next block formed under the exponentials of this one came out the same (108 us).
//
// kSplit: ragged N.  p as two bf16 terms (16 to 17 bits), which fill S's 64 columns, times a as two
// bf16 terms ([feature][column], as stage 2 leaves them for the backward as well): three products instead of one (low x low
// is 2^-18).  a's second term takes the room of the output slabs, so every thread stores its own row.  2 x 8 heads x N = 6001,
// k = m = 256: the call 60.3 us, 51.9 with fp16 weights, 281 with stages 2 and 3 on CUDA cores.
#pragma once

#include "k2_key_side.cuh"
#include "k3_query_side.cuh"

namespace flurka {

constexpr int kK3UThreads = 768;                        // 4 issuers, operand builder, Q loader, 2 idle; 16 warps of row owners
constexpr int kK3URegsFew = 32, kK3URegsMany = 104;     // 768 threads x 80 at launch = 256 x 32 + 512 x 104

struct K3USmem {
  uint32_t w, aT, q, ostage, ones, bias, bars, total;
};
__host__ __device__ inline K3USmem k3u_smem_plan(int p, bool split) {
  K3USmem s;
  uint32_t off = 0;
  s.w = off;      off += (uint32_t)p * 128;              // W: [p rows x 128 B]
  s.aT = off;     off += (uint32_t)p * 128;              // a^T: p/64 K-blocks of [64 rows x 128 B]
  if (split) off += (uint32_t)p * 128;                   // (split: a, two terms of [p rows x 128 B] each)
  s.q = off;      off += 4 * 16384;                      // one Q tile per group
  s.ostage = off; off += split ? 0 : 16 * 4096;          // a [32 x 64] bf16 output slab per row-owner warp
  s.ones = off;   off += 4096;                           // [128 x 16] bf16, no swizzle
  s.bias = off;   off += 8192;                           // [256 x 16] bf16, no swizzle
  s.bars = off;   off += 512;
  s.total = off + 1024;
  return s;
}

template <bool kSplit>
__global__ void __launch_bounds__(kK3UThreads, 1)
k3_query_units(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmW,
               const __grid_constant__ CUtensorMap tmAT, const __grid_constant__ CUtensorMap tmO,
               const K3Params prm) {
  using namespace tc;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const int p = prm.p;
  const K3USmem L = k3u_smem_plan(p, kSplit);
  const int U = p >> 6;                       // blocks of 64 features

  const uint32_t bars = base + L.bars;
  // per group: one phase per tile
  const uint32_t bar_qfull = bars;            // [4]  Q tile landed
  const uint32_t bar_qempty = bars + 32;      // [4]  every S of the tile formed
  const uint32_t bar_ofull = bars + 64;       // [4]  O complete
  // per group: one phase per block of 64 features
  const uint32_t bar_sfull = bars + 96;       // [4]  S ready
  const uint32_t bar_pfull = bars + 128;      // [4]  p written (and O of the tile before read) (4 warps)
  const uint32_t bar_wfull = bars + 160;      //      W resident
  const uint32_t bar_drained = bars + 168;    // [4]  every MMA of a group for the old head is complete
  const uint32_t bar_head = bars + 200;       //      a^T and the bias operand of the new head in place
  const uint32_t tmem_slot = bars + 208;
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_shared;
  __shared__ volatile int first_block;        // of the current head

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t_begin = (int)(((long long)blockIdx.x * prm.total_tiles) / gridDim.x);
  const int t_end = (int)(((long long)(blockIdx.x + 1) * prm.total_tiles) / gridDim.x);
  const int ntiles = t_end - t_begin;
  const int head_first = t_begin / prm.tiles_per_head;
  const int head_last = ntiles > 0 ? (t_end - 1) / prm.tiles_per_head : head_first - 1;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int i = 0; i < 4; ++i) {
      mbar_init(bar_qfull + 8 * i, 1);
      mbar_init(bar_qempty + 8 * i, 1);
      mbar_init(bar_ofull + 8 * i, 1);
      mbar_init(bar_sfull + 8 * i, 1);
      mbar_init(bar_pfull + 8 * i, 4);
      mbar_init(bar_drained + 8 * i, 1);
    }
    mbar_init(bar_wfull, 1);
    mbar_init(bar_head, 33);
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  {
    // the all-ones A operand of the bias step: [128 x 16] bf16, no swizzle, columns 0..2 are 1
    // (element (r, c) at (r/8)*256 + (c/8)*128 + (r%8)*16 + (c%8)*2 bytes)
    uint32_t* ones = reinterpret_cast<uint32_t*>(base_ptr + L.ones);
    for (int e = threadIdx.x; e < 1024; e += kK3UThreads) {
      const int c = (e & 3) + ((e >> 5) & 1) * 4;
      ones[e] = c == 0 ? 0x3f803f80u : (c == 1 ? 0x00003f80u : 0u);
    }
  }
  fence_proxy_async_smem();
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  if (threadIdx.x == 0) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(tmem_slot));
    tmem_base_shared = v;
  }
  __syncthreads();
  const uint32_t tmem = tmem_base_shared;

  if (ntiles > 0) {
    if (warp < 8) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kK3URegsFew));
      if (warp == 5 && elect_one()) {
        // ============================================================ TMA producer: W, then Q tiles.  Neither is stage 2's
        // result, and this kernel only starts once stage 2 has waited for everything before it: no wait here
        prefetch_tmap(&tmQ);
        prefetch_tmap(&tmW);
        mbar_arrive_expect_tx(bar_wfull, (uint32_t)p * 128);
        tma_load_2d(base + L.w, &tmW, bar_wfull, 0, 0);
        bool ok = true;
        int issued = 0, head = head_first, tih = t_begin - head_first * prm.tiles_per_head;
        for (int i = 0; i < ntiles && ok; ++i) {
          const int g = i & 3;
          if (i >= 4) ok = mbar_wait(bar_qempty + 8 * g, (uint32_t)((i >> 2) - 1) & 1u, prm.status, &abort_flag);
          if (!ok) break;
          mbar_arrive_expect_tx(bar_qfull + 8 * g, 16384u);
          if (prm.H > 0) tma_load_3d(base + L.q + g * 16384, &tmQ, bar_qfull + 8 * g, (head % prm.H) * 64, tih * 128, head / prm.H);
          else tma_load_3d(base + L.q + g * 16384, &tmQ, bar_qfull + 8 * g, 0, tih * 128, head);
          ++issued;
          if (++tih == prm.tiles_per_head) { tih = 0; ++head; }
          // four tiles are in flight or in use; the next one waits in L2
          if (i + 1 < ntiles && i >= 3) {
            if (prm.H > 0) tma_prefetch_3d(&tmQ, (head % prm.H) * 64, tih * 128, head / prm.H);
            else tma_prefetch_3d(&tmQ, 0, tih * 128, head);
          }
        }
        if (!ok) {
          for (int i = max(0, issued - 4); i < issued; ++i)
            (void)mbar_wait(bar_qfull + 8 * (i & 3), (uint32_t)(i >> 2) & 1u, prm.status, &abort_flag);
        }
      } else if (warp < 4 && elect_one()) {
        // ============================================================ MMA issuer of group g
        const int g = warp;
        const uint32_t ts = tmem + g * 128, to = ts + 64;
        const uint32_t idescS = make_idesc(kFmtBF16, 0, 0, 128, 64);
        const uint32_t idescO = kSplit ? make_idesc(kFmtBF16, 0, 1, 128, 64) : make_idesc(kFmtF16, 0, 0, 128, 64);
        const uint64_t qd = make_sdesc(base + L.q + g * 16384, 16, 1024, kSwizzle128);
        const uint64_t od = make_sdesc(base + L.ones, 128, 256, kSwizzleNone);
        bool ok = mbar_wait(bar_wfull, 0, prm.status, &abort_flag);
        uint32_t t = 0, n = 0;                                 // the group's tiles and blocks so far
        // S of a block over the p of the block before it, whose product was queued earlier by this thread
        auto form_s = [&](int blk) {
          mma_ss_x4(ts, qd, make_sdesc(base + L.w + blk * 8192, 16, 1024, kSwizzle128), 2, 2, idescS, 0u);
          mma_ss(ts, od, make_sdesc(base + L.bias + blk * 2048, 128, 256, kSwizzleNone), idescS, 1u);
          mma_commit(bar_sfull + 8 * g);
        };
        for (int head = head_first; head <= head_last && ok; ++head) {
          ok = mbar_wait(bar_head, (uint32_t)(head - head_first) & 1u, prm.status, &abort_flag);
          if (!ok) break;
          const int first = first_block;
          auto block = [&](int u) { return u == 0 ? first : (u <= first ? u - 1 : u); };
          const int i_end = min(ntiles, (head + 1) * prm.tiles_per_head - t_begin);
          int i = max(0, head * prm.tiles_per_head - t_begin);
          i += (g - i) & 3;                                    // this group's first tile of the head
          if (i < i_end) {
            ok = mbar_wait(bar_qfull + 8 * g, t & 1u, prm.status, &abort_flag);
            if (!ok) break;
            tcgen05_fence_after();
            form_s(first);
            if (U == 1) mma_commit(bar_qempty + 8 * g);
          }
          for (; i < i_end && ok; i += 4, ++t) {
            for (int u = 0; u < U; ++u, ++n) {
              ok = mbar_wait(bar_pfull + 8 * g, n & 1u, prm.status, &abort_flag);
              if (!ok) break;
              tcgen05_fence_after();
              const uint32_t blk = base + L.aT + block(u) * 8192;
              if constexpr (kSplit) {
                // hi hi + lo hi + hi lo; a lies [feature][column]: an MN-major operand, 16 features = 2048 B per step
                const uint64_t ah = make_sdesc(blk, 8192, 1024, kSwizzle128);
                mma_ts_x4(to, ts, ah, 128, idescO, u > 0 ? 1u : 0u);
                mma_ts_x4(to, ts + 32, ah, 128, idescO, 1u);
                mma_ts_x4(to, ts, make_sdesc(blk + p * 128, 8192, 1024, kSwizzle128), 128, idescO, 1u);
              } else {
                mma_ts_x4(to, ts, make_sdesc(blk, 16, 1024, kSwizzle128), 2, idescO, u > 0 ? 1u : 0u);
              }
              if (u + 1 < U) {
                form_s(block(u + 1));
                if (u + 2 == U) mma_commit(bar_qempty + 8 * g);
              } else {
                mma_commit(bar_ofull + 8 * g);
                if (i + 4 < i_end) {
                  ok = mbar_wait(bar_qfull + 8 * g, (t + 1) & 1u, prm.status, &abort_flag);
                  if (!ok) break;
                  tcgen05_fence_after();
                  form_s(first);
                  if (U == 1) mma_commit(bar_qempty + 8 * g);
                }
              }
            }
          }
          if (ok) mma_commit(bar_drained + 8 * g);
        }
      } else if (warp == 4) {
        // ============================================================ per-head operands
        if (lane == 0) prefetch_tmap(&tmAT);
        grid_dependency_wait_async();
        bool ok = true;
        for (int head = head_first; head <= head_last && ok; ++head) {
          const int e = head - head_first;
          for (int g = 0; g < 4 && e > 0 && ok; ++g) ok = mbar_wait(bar_drained + 8 * g, (uint32_t)(e - 1) & 1u, prm.status, &abort_flag);
          if (!ok) break;
          if (lane == 0) {
            mbar_arrive_expect_tx(bar_head, (uint32_t)p * (kSplit ? 256 : 128));
            for (int kb = 0; kb < U; ++kb) {
              if constexpr (kSplit) {
                tma_load_3d(base + L.aT + kb * 8192, &tmAT, bar_head, 0, kb * 64, head * 2);
                tma_load_3d(base + L.aT + p * 128 + kb * 8192, &tmAT, bar_head, 0, kb * 64, head * 2 + 1);
              } else {
                tma_load_3d(base + L.aT + kb * 8192, &tmAT, bar_head, kb * 64, 0, head);
              }
            }
          }
          const float* wv = prm.weight + (size_t)head * p;
          float mx = -INFINITY;
          int best = 0;
          for (int f = lane; f < p; f += 32) {
            const float b = __ldcg(wv + f);
            if (b > mx) { mx = b; best = f >> 6; }
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            const float m2 = __shfl_xor_sync(0xffffffffu, mx, o);
            const int b2 = __shfl_xor_sync(0xffffffffu, best, o);
            if (m2 > mx || (m2 == mx && b2 < best)) { mx = m2; best = b2; }
          }
          // bias[f][c], c < 16, no swizzle: (f/8)*256 + (c/8)*128 + (f%8)*16 + (c%8)*2 bytes
          for (int f = lane; f < p; f += 32) {
            float b = __ldcg(wv + f) - mx;
            const __nv_bfloat16 h0 = __float2bfloat16_rn(b);  b -= __bfloat162float(h0);
            const __nv_bfloat16 h1 = __float2bfloat16_rn(b);  b -= __bfloat162float(h1);
            const __nv_bfloat16 h2 = __float2bfloat16_rn(b);
            uint4* row = reinterpret_cast<uint4*>(base_ptr + L.bias + (f >> 3) * 256 + (f & 7) * 16);
            row[0] = make_uint4((uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16),
                                (uint32_t)__bfloat16_as_ushort(h2), 0u, 0u);
            row[8] = make_uint4(0u, 0u, 0u, 0u);
          }
          if (lane == 0) first_block = best;
          fence_proxy_async_smem();
          mbar_arrive(bar_head);
        }
      }
    } else {
      // ============================================================ row owners (four groups of 4 warps, one row per thread)
      asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kK3URegsMany));
      const int g = (warp - 8) >> 2;                   // tiles with (i & 3) == g
      const int q4 = warp & 3;                         // TMEM lane quadrant
      const uint32_t ts = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)g * 128u, to = ts + 64;
      const uint32_t slab = base + L.ostage + (uint32_t)(warp - 8) * 4096u;
      const float kLog2e = 1.4426950408889634f;
      const uint64_t l2 = pack2(kLog2e, kLog2e);
      // 32 columns: x = 2^(S log2e - r) as fp16 pairs and the row sum.  One pair in eight takes its exponential as a
      // cubic on the FMA pipe, the others on the special-function unit (three in eight, the mix of k3_query_side, is 2.5 %
      // slower here, where issue slots are the scarcer: 110.3 against 107.2 us; none at all 112.7).
      // kSplit: as two bf16 terms, all exponentials on the special-function unit (the cubic is good for fp16 only).
      auto exp_split = [&](const uint32_t (&r)[32], uint32_t (&hi)[16], uint32_t (&lo)[16], uint64_t ms2, uint64_t& den2) {
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          float x0, x1;
          unpack2(fma2(pack2u(r[2 * e], r[2 * e + 1]), l2, ms2), x0, x1);
          const float e0 = ex2_approx(x0), e1 = ex2_approx(x1);
          den2 = add2(den2, pack2(e0, e1));
          hi[e] = pack_bf16x2(e0, e1);
          lo[e] = pack_bf16x2(e0 - __uint_as_float(hi[e] << 16), e1 - __uint_as_float(hi[e] & 0xffff0000u));
        }
      };
      auto exp_block = [&](const uint32_t (&r)[32], uint32_t (&hh)[16], uint64_t ms2, uint64_t& den2) {
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          float x0, x1, e0, e1;
          unpack2(fma2(pack2u(r[2 * e], r[2 * e + 1]), l2, ms2), x0, x1);
          if ((e & 7) == 4) {
            // far below what fp16 can hold the result is 0 either way; the cubic needs its exponent in range
            exp2_cubic2(pack2(fmaxf(x0, -60.f), fmaxf(x1, -60.f)), e0, e1);
          } else {
            e0 = ex2_approx(x0);
            e1 = ex2_approx(x1);
          }
          den2 = add2(den2, pack2(e0, e1));
          const __half2 h2 = __floats2half2_rn(e0, e1);
          hh[e] = *reinterpret_cast<const uint32_t*>(&h2);
        }
      };
      auto max32 = [&](const uint32_t (&r)[32], float (&m4)[4]) {
#pragma unroll
        for (int e = 0; e < 32; e += 8) {
#pragma unroll
          for (int c = 0; c < 4; ++c) m4[c] = fmax3(m4[c], __uint_as_float(r[e + 2 * c]), __uint_as_float(r[e + 2 * c + 1]));
        }
      };
      bool ok = true;
      uint32_t t = 0, n = 0;
      int head = (t_begin + g) / prm.tiles_per_head, tih = (t_begin + g) % prm.tiles_per_head;
      for (int i = g; i < ntiles && ok; i += 4, ++t) {
        float r = 0.f;                                   // the row's reference, base 2
        uint64_t den2 = pack2(0.f, 0.f);
#pragma unroll 1
        for (int u = 0; u < U; ++u, ++n) {
          ok = mbar_wait(bar_sfull + 8 * g, n & 1u, prm.status, &abort_flag);
          if (!ok) break;
          tcgen05_fence_after();
          uint32_t ra[32], rb[32], hh[16];
          tmem_ld32(ts, ra);
          tmem_ld32(ts + 32, rb);
          float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
          tmem_wait_ld(ra);
          tmem_wait_ld(rb);
          max32(ra, m4);
          max32(rb, m4);
          const float mx = fmaxf(fmax3(m4[0], m4[1], m4[2]), m4[3]) * kLog2e;
          if (u == 0) {
            r = mx;
          } else if (__any_sync(0xffffffffu, mx > r + 15.f)) {
            // raise the reference of the rows that need it (the product of the block before is complete: S came after it)
            const float nr = mx > r + 15.f ? mx : r;
            const float f = ex2_approx(r - nr);
            r = nr;
            den2 = mul2(den2, pack2(f, f));
#pragma unroll 1
            for (int c = 0; c < 64; c += 16) {
              uint32_t o16[16];
              tmem_ld16(to + c, o16);
              tmem_wait_ld16(o16);
#pragma unroll
              for (int e = 0; e < 16; ++e) o16[e] = __float_as_uint(__uint_as_float(o16[e]) * f);
              tmem_st16(to + c, o16);
            }
          }
          const uint64_t ms2 = pack2(-r, -r);
          if constexpr (kSplit) {
            uint32_t lo[16];
            exp_split(ra, hh, lo, ms2, den2);
            tmem_st16(ts, hh);
            tmem_st16(ts + 32, lo);
            exp_split(rb, hh, lo, ms2, den2);
            tmem_st16(ts + 16, hh);
            tmem_st16(ts + 48, lo);
          } else {
            exp_block(ra, hh, ms2, den2);
            tmem_st16(ts, hh);
            exp_block(rb, hh, ms2, den2);
            tmem_st16(ts + 16, hh);
          }
          tmem_wait_st();
          tcgen05_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_pfull + 8 * g);
        }
        if (!ok) break;
        // ---- the tile's O / sum as one TMA store of whole lines per warp
        float d0, d1;
        unpack2(den2, d0, d1);
        const float inv = 1.f / fmaxf(d0 + d1, 1.17549435e-38f);
        ok = mbar_wait(bar_ofull + 8 * g, t & 1u, prm.status, &abort_flag);
        if (!ok) break;
        tcgen05_fence_after();
        if (!kSplit && lane == 0) bulk_wait_group_read0();   // the slab's previous store has been read
        __syncwarp();
        const int row = tih * 128 + q4 * 32 + lane;
        __nv_bfloat16* orow = nullptr;
        if constexpr (kSplit)
          orow = prm.out + (prm.H > 0 ? (((size_t)(head / prm.H) * prm.N + row) * prm.H + (size_t)(head % prm.H)) * 64
                                      : ((size_t)head * prm.N + row) * 64);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t o[32];
          tmem_ld32(to + 32 * c, o);
          tmem_wait_ld(o);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            uint32_t w[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
              const __nv_bfloat162 o2 = __floats2bfloat162_rn(__uint_as_float(o[e * 8 + 2 * x]) * inv, __uint_as_float(o[e * 8 + 2 * x + 1]) * inv);
              w[x] = *reinterpret_cast<const uint32_t*>(&o2);
            }
            if constexpr (kSplit) {
              // (the second term of a has the slabs' room: a thread stores its own row)
              if (row < prm.N) reinterpret_cast<uint4*>(orow)[4 * c + e] = make_uint4(w[0], w[1], w[2], w[3]);
            } else {
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(slab + lane * 128 + (((4 * c + e) ^ (lane & 7)) << 4)),
                           "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
            }
          }
        }
        tcgen05_fence_before();
        if (!kSplit) fence_proxy_async_smem();
        __syncwarp();
        if (!kSplit && lane == 0 && tih * 128 + q4 * 32 < prm.N) {  // rows past the end are clipped by the tensor map
          if (prm.H > 0) tma_store_3d(&tmO, slab, (head % prm.H) * 64, tih * 128 + q4 * 32, head / prm.H);
          else tma_store_3d(&tmO, slab, 0, tih * 128 + q4 * 32, head);
          bulk_commit_group();
        }
        tih += 4;
        while (tih >= prm.tiles_per_head) { tih -= prm.tiles_per_head; ++head; }
      }
      if (!kSplit && lane == 0) bulk_wait_group0();     // this warp's output stores are complete
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

}  // namespace flurka
