// The whole forward pass (arxiv 2306.15799, Eq. (2)) of a small head in one kernel on CUDA cores: a cluster of eight CTAs
// per head of at most 64 columns, for calls whose time is that of launches and of one kernel waiting for the next.
//
// Stage 1: every CTA projects an eighth of the sequence; the partial K', V' meet through distributed shared memory (CTA r
// adds up its eighth of the elements and hands the sums to all eight).  Stage 2: an eighth of the features each; a_i, b_i
// go to all eight.  Stage 3: an eighth of the queries each.  The building blocks, the normalisation with a running maximum
// and the fp32 arithmetic are those of simt_kernels.cuh; K', V', a, b are also left in the workspace.
// One launch instead of four (clear, three stages).  Everything a CTA reads from global memory is in flight at once; what is
// left is a chain of short phases (fp32, N = 256, d = 32, k = 32, m = 64: loads 3, stage 1 3, exchange 4, stage 2 4,
// exchange 1, stage 3 6 thousand cycles).  512 threads with one row each took 31 instead of 25 thousand in all (shared
// memory reads).
#pragma once

#include "k1_down_project_pair.cuh"
#include "simt_kernels.cuh"

namespace flurka {

constexpr int kSmallCtas = 8;                 // CTAs of a cluster (the largest portable cluster)
constexpr int kSmallRows = 32;                // rows per tile
constexpr int kSmallThreads = kSimtThreads;   // two rows of a tile per 16 threads

struct SmallShape {
  int ld;                // floats between rows of W, K', V', Q tiles
  int fpc;               // features per CTA
  int npc;               // positions (and queries) per CTA
  int n32;               // npc, rounded up to 32
  size_t part, kv, w, a, b, q, p, e, x, total;    // float offsets
};
__host__ __device__ inline SmallShape small_shape(int N, int d, int k, int p) {
  SmallShape s;
  s.ld = simt_ld(d);
  s.fpc = (p + kSmallCtas - 1) / kSmallCtas;
  s.npc = ((N + kSmallCtas - 1) / kSmallCtas + 3) & ~3;
  size_t off = 0;
  const int k32 = (k + 31) & ~31;
  s.part = off; off += (size_t)2 * k32 * s.ld;             // this CTA's part of K', V'
  s.kv = off;   off += (size_t)2 * ((k + 63) & ~63) * s.ld;   // K', V'
  s.w = off;    off += (size_t)((p + 63) & ~63) * s.ld;    // W
  s.a = off;    off += (size_t)((p + 63) & ~63) * s.ld;    // a
  s.b = off;    off += (size_t)((p + 63) & ~63);           // b_i (RNN: z_i)
  s.n32 = (s.npc + 31) & ~31;
  s.q = off;    off += (size_t)s.n32 * s.ld;               // this CTA's queries
  s.p = off;    off += (size_t)kSmallRows * 68;            // weights of a tile
  s.e = off;    off += (size_t)2 * k32 * (s.n32 + 4);      // this CTA's columns of E, F
  s.x = off;    off += (size_t)2 * s.n32 * 64;        // this CTA's rows of K, V; then |k'|^2 / 2
  s.total = off + 64;                                 // (the products may read past a tile: columns nobody keeps)
  return s;
}

namespace tc {
__device__ __forceinline__ float4 ld_cluster_v4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void st_cluster_f32(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
}  // namespace tc

// four consecutive elements of a row into shared memory, without waiting for them where no conversion is needed
template <typename T>
__device__ __forceinline__ void small_stage4(float* dst, const T* src, const T* valid, int live, bool vec) {
  if constexpr (sizeof(T) == 4) {
    if (vec) {
      const int bytes = 4 * max(0, min(live, 4));
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_u32(dst)), "l"(bytes > 0 ? src : valid), "r"(bytes)
                   : "memory");
      return;
    }
  }
  *reinterpret_cast<float4*>(dst) = simt_load_row4(src, live, vec);
}

// One tile of 32 rows against up to 64 items at a time; see simt_attend.  Ys: the items' rows, Vs: their vectors (both `ld`
// floats apart), bias: per item (PERFORMER: added to the exponent; RNN, query side: factor).
template <bool kPerformer, bool kKeySide>
__device__ __forceinline__ void small_attend(float (&acc)[2][4], float (&run_max)[2], float (&run_sum)[2], const float* Xs,
                                             const float* Ys, const float* Vs, const float* bias, float* Ps, int ld, int cols,
                                             int items, int feature0) {
  constexpr int kLd = 68;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    run_max[r] = -INFINITY;
    run_sum[r] = 0.f;
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0.f;
  }
#pragma unroll 1
  for (int i0 = 0; i0 < items; i0 += 64) {
    float s[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    if (kPerformer) simt_dots<2>(s, Xs, Ys + (size_t)i0 * ld, ld, cols);
    __syncthreads();                                       // the weights of the step before have been used
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int row = ty + 16 * r;
      if (kPerformer) {
        float cm = -INFINITY;
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          const int i = i0 + tx + 16 * f;
          s[r][f] = i < items ? s[r][f] + bias[i] : -INFINITY;
          cm = fmaxf(cm, s[r][f]);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, o));
        const float new_max = fmaxf(run_max[r], cm);
        const float rescale = expf(run_max[r] - new_max);
        run_max[r] = new_max;
        run_sum[r] *= rescale;
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] *= rescale;
#pragma unroll
        for (int f = 0; f < 4; ++f) s[r][f] = expf(s[r][f] - new_max);
      } else {
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          const int i = i0 + tx + 16 * f;
          float v = 0.f;
          if (i < items) {
            // key side: feature feature0 + row of key i; query side: feature i of the row
            const float x = kKeySide ? Ys[(size_t)i * ld + min(feature0 + row, cols - 1)] : Xs[row * ld + i];
            v = (x > 0.f ? x + 1.f : expf(x)) * (kKeySide ? 1.f : bias[i]);
          }
          s[r][f] = v;
        }
      }
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        run_sum[r] += s[r][f];
        Ps[row * kLd + tx + 16 * f] = s[r][f];
      }
    }
    __syncthreads();
    simt_product<2, 1>(acc, Ps, kLd, Vs + (size_t)i0 * ld, ld, min(64, (items - i0 + 3) & ~3));
  }
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) run_sum[r] += __shfl_xor_sync(0xffffffffu, run_sum[r], o);
}

template <typename T, bool kPerformer>
__global__ void __cluster_dims__(kSmallCtas, 1, 1) __launch_bounds__(kSmallThreads, 1)
simt_small_forward(const T* __restrict__ Q, const T* __restrict__ Kin, const T* __restrict__ Vin, const T* __restrict__ E,
                   const T* __restrict__ Fin, const T* __restrict__ W, float* __restrict__ KpVp, float* __restrict__ weight,
                   float* __restrict__ a32, int* __restrict__ status, T* __restrict__ out, int BH, int N, int d, int k, int p,
                   int seq_major_heads, int ef_heads, int keep_status) {
  using namespace tc;
  extern __shared__ __align__(16) float smem[];
  const SmallShape S = small_shape(N, d, k, p);
  const int ld = S.ld, cols = (d + 3) & ~3, pieces = cols >> 2;
  const int bh = blockIdx.x / kSmallCtas;
  const int rank = (int)cluster_ctarank();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const bool vec = (d & 3) == 0, vec_p = (N & 3) == 0;
  const HeadView hv = head_view(bh, seq_major_heads, N, d);
  const int k32 = (k + 31) & ~31, k64 = (k + 63) & ~63;
  const int n0 = min(N, rank * S.npc), n1 = min(N, n0 + S.npc);
  grid_dependency_wait();
  if (blockIdx.x == 0 && threadIdx.x < 4 && !keep_status) status[threadIdx.x] = 0;

  // ---- everything this CTA reads, all in flight together.  Rows past the last item or position are zeros (the dot
  //      products read them)
  {
    const int lde = S.n32 + 4, xp = 16;
    for (int idx = threadIdx.x; idx < 2 * k32 * (S.n32 >> 2); idx += kSmallThreads) {
      const int nn = (idx % (S.n32 >> 2)) * 4, j = (idx / (S.n32 >> 2)) % k32, t = idx / ((S.n32 >> 2) * k32);
      const T* __restrict__ P = (t ? Fin : E) + (ef_heads > 0 ? (size_t)(bh % ef_heads) * k * N : 0);
      small_stage4(smem + S.e + (size_t)(t * k32 + j) * lde + nn, P + (size_t)j * N + n0 + nn, P, j < k ? n1 - (n0 + nn) : 0, vec_p);
    }
    for (int idx = threadIdx.x; idx < 2 * S.n32 * xp; idx += kSmallThreads) {
      const int c = (idx % xp) * 4, nn = (idx / xp) % S.n32, t = idx / (xp * S.n32);
      const T* __restrict__ X = (t ? Vin : Kin) + hv.base;
      small_stage4(smem + S.x + (size_t)idx * 4, X + (size_t)(n0 + nn) * hv.row_stride + c, X, n0 + nn < n1 ? d - c : 0, vec);
    }
    for (int idx = threadIdx.x; idx < S.n32 * pieces; idx += kSmallThreads) {
      const int r = idx / pieces, c = (idx % pieces) * 4;
      small_stage4(smem + S.q + (size_t)r * ld + c, Q + hv.base + (size_t)(n0 + r) * hv.row_stride + c, Q, n0 + r < n1 ? d - c : 0, vec);
    }
    const int p64 = (p + 63) & ~63;
    for (int idx = threadIdx.x; kPerformer && idx < p64 * pieces; idx += kSmallThreads) {
      const int r = idx / pieces, c = (idx % pieces) * 4;
      small_stage4(smem + S.w + (size_t)r * ld + c, W + (size_t)r * d + c, W, r < p ? d - c : 0, vec);
    }
    if constexpr (sizeof(T) == 4) asm volatile("cp.async.wait_all;" ::: "memory");
  }
  __syncthreads();
  // ---- stage 1: this CTA's part of K', V', 32 rows at a time
  float* Ps = smem + S.p;
#pragma unroll 1
  for (int tj = 0; tj < 2 * (k32 >> 5); ++tj) {
    const int t = tj / (k32 >> 5), j0 = (tj % (k32 >> 5)) * 32;
    float acc[2][4];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[r][c] = 0.f;
    simt_product<2, 1>(acc, smem + S.e + (size_t)(t * k32 + j0) * (S.n32 + 4), S.n32 + 4, smem + S.x + (size_t)t * S.n32 * 64,
                        64, S.n32);
#pragma unroll
    for (int r = 0; r < 2; ++r)
      {
        const int c = tx * 4;
        if (c < ld) *reinterpret_cast<float4*>(smem + S.part + (size_t)(t * k32 + j0 + ty + 16 * r) * ld + c) =
            make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
      }
  }
  cluster_sync_all();
  {
    // this CTA's eighth of the rows of K' and V': the sum of the eight parts, to all eight CTAs (rows past k: zeros)
    const uint32_t sm = smem_u32(smem);
    const int total = 2 * k64 * pieces;
    const int e0 = (int)((long long)total * rank / kSmallCtas), e1 = (int)((long long)total * (rank + 1) / kSmallCtas);
    for (int e = e0 + (int)threadIdx.x; e < e1; e += kSmallThreads) {
      const int c = (e % pieces) * 4, j = (e / pieces) % k64, t = e / (pieces * k64);
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j < k) {
        const uint32_t src = sm + (uint32_t)(S.part + (size_t)(t * k32 + j) * ld + c) * 4u;
        float4 v[kSmallCtas];
#pragma unroll
        for (int r = 0; r < kSmallCtas; ++r) v[r] = ld_cluster_v4(map_to_cta(src, (uint32_t)r));
#pragma unroll
        for (int r = 0; r < kSmallCtas; ++r) { s.x += v[r].x; s.y += v[r].y; s.z += v[r].z; s.w += v[r].w; }
        float* o = KpVp + ((size_t)t * BH + bh) * (size_t)k * d + (size_t)j * d + c;
        if (c < d) o[0] = s.x;
        if (c + 1 < d) o[1] = s.y;
        if (c + 2 < d) o[2] = s.z;
        if (c + 3 < d) o[3] = s.w;
      }
      const uint32_t dst = sm + (uint32_t)(S.kv + (size_t)(t * k64 + j) * ld + c) * 4u;
#pragma unroll
      for (int r = 0; r < kSmallCtas; ++r) st_cluster_v4(map_to_cta(dst, (uint32_t)r), s);
    }
  }
  cluster_sync_all();

  // ---- stage 2: features [f0, f0 + fpc) in tiles of 32
  const float* Ks = smem + S.kv;
  const float* Vs = Ks + (size_t)k64 * ld;
  float* nrm = smem + S.x;
  if (kPerformer) {
    // -|k'_j|^2 / 2, over the K, V tile that is no longer needed
    for (int j = threadIdx.x; j < k; j += kSmallThreads) {
      float sq = 0.f;
      for (int c = 0; c < cols; c += 4) {
        const float4 v = *reinterpret_cast<const float4*>(Ks + (size_t)j * ld + c);
        sq = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, sq))));
      }
      nrm[j] = -0.5f * sq;
    }
    __syncthreads();
  }
  const int f_end = min(p, (rank + 1) * S.fpc);
#pragma unroll 1
  for (int f0 = rank * S.fpc; f0 < f_end; f0 += kSmallRows) {
    float acc[2][4], run_max[2], run_sum[2];
    small_attend<kPerformer, true>(acc, run_max, run_sum, smem + S.w + (size_t)f0 * ld, Ks, Vs, nrm, Ps, ld, cols, k, f0);
    const uint32_t sm = smem_u32(smem);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int f = f0 + ty + 16 * r;
      if (f >= f_end) continue;
      const float inv = 1.f / fmaxf(run_sum[r], 1.17549435e-38f);
      const float b = kPerformer ? run_max[r] + logf(run_sum[r]) : run_sum[r];
      if (tx < kSmallCtas) st_cluster_f32(map_to_cta(sm + (uint32_t)(S.b + f) * 4u, (uint32_t)tx), b);
      if (tx == 0) weight[(size_t)bh * p + f] = b;
      {
        const int c = tx * 4;
        if (c >= cols) continue;
        const float4 v = make_float4(acc[r][0] * inv, acc[r][1] * inv, acc[r][2] * inv, acc[r][3] * inv);
        const uint32_t dst = sm + (uint32_t)(S.a + (size_t)f * ld + c) * 4u;
#pragma unroll
        for (int o = 0; o < kSmallCtas; ++o) st_cluster_v4(map_to_cta(dst, (uint32_t)o), v);
        float* ap = a32 + ((size_t)bh * p + f) * d + c;
        if (c < d) ap[0] = v.x;
        if (c + 1 < d) ap[1] = v.y;
        if (c + 2 < d) ap[2] = v.z;
        if (c + 3 < d) ap[3] = v.w;
      }
    }
  }
  // rows of a past the last feature are multiplied by weights of zero: they have to be finite
  for (int idx = threadIdx.x; idx < (((p + 3) & ~3) - p) * ld; idx += kSmallThreads) smem[S.a + (size_t)p * ld + idx] = 0.f;
  cluster_sync_all();

  // ---- stage 3: this CTA's queries
#pragma unroll 1
  for (int r0 = n0; r0 < n1; r0 += kSmallRows) {
    float acc[2][4], run_max[2], run_sum[2];
    small_attend<kPerformer, false>(acc, run_max, run_sum, smem + S.q + (size_t)(r0 - n0) * ld, smem + S.w, smem + S.a,
                                        smem + S.b, Ps, ld, cols, p, 0);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int n = r0 + ty + 16 * r;
      if (n >= n1) continue;
      const float inv = 1.f / fmaxf(run_sum[r], 1.17549435e-38f);
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (tx * 4 + e < d) store_out(out + hv.base + (size_t)n * hv.row_stride + tx * 4 + e, acc[r][e] * inv);
    }
  }
}

}  // namespace flurka
