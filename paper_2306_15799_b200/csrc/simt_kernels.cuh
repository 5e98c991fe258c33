// CUDA-core (fp32 FFMA) kernels for the three stages of the FLuRKA forward pass
// (arxiv 2306.15799, Eq. (2)).  They serve the float32 I/O configuration, every shape the
// tensor-core kernels do not cover, and stages 2 and 3 where those have no form with more than 16-bit weights.
//
// Stage 1  down-projection   K' = E K, V' = F V          (Section 2.1; sequence contraction)
// Stage 2  key side          per feature i:  b_i = log sum_j exp(L_ji),  a_i = softmax_j(L_.i)^T V'
//                            with L_ji = w_i.k'_j - |k'_j|^2/2            (PERFORMER)
//                            or  z_i = sum_j (elu(k'_ji)+1),  a_i = sum_j (elu(k'_ji)+1) v'_j / z_i  (RNN)
// Stage 3  query side        O_n = sum_i p_ni a_i / sum_i p_ni,  p_ni = exp(w_i.q_n + b_i - r_n)  (PERFORMER)
//                            or  p_ni = (elu(q_ni)+1) z_i                                          (RNN)
//
// Stage 2 + 3 are Eq. (2)'s phi(Q)(phi(K')^T V') / phi(Q)(phi(K')^T 1): phi(K')^T V' = diag(e^b) a and
// phi(K')^T 1 = e^b, so every per-feature scale e^{b_i} moves into the query-side exponent.  The
// 1/sqrt(m), exp(-|q|^2/2) and any per-row r_n cancel in the ratio.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>

#include "tc_common.cuh"

namespace flurka {

// Where head bh of a [B,H,N,d] tensor (H == 0) or of a [B,N,H,d] tensor (H = number of heads) starts,
// and the distance between consecutive sequence positions of that head, in elements.
struct HeadView {
  size_t base, row_stride;
};
__host__ __device__ __forceinline__ HeadView head_view(int bh, int H, int N, int d) {
  HeadView v;
  if (H > 0) {
    v.base = ((size_t)(bh / H) * N * H + (size_t)(bh % H)) * d;
    v.row_stride = (size_t)H * d;
  } else {
    v.base = (size_t)bh * N * d;
    v.row_stride = (size_t)d;
  }
  return v;
}

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ void store_out(float* p, float v) { *p = v; }
__device__ __forceinline__ void store_out(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// ---------------------------------------------------------------------------------------------
// Building blocks.  A block is 256 threads, ty = tid / 16, tx = tid % 16; a thread owns the R rows ty + 16 r and, in
// each of NB 64-wide column blocks, the columns 4 tx .. 4 tx + 3.  Both kinds of product below read shared memory as
// 16-byte pieces only: with R = 8, 12 loads per 128 FFMA of a warp.  B = 2, H = 8, N = 4096, d = 64, k = m = 256, fp32:
// stage 1 443 -> 117 us, stage 3 617 -> 150 us against scalar reads and four rows per thread.  Tried and slower:
// 8 x 8 outputs per thread (half the warps: 120 and 164 us), two-wide FMA on pairs of contraction steps (147 and
// 215 us: it has no higher rate than FFMA and twice the accumulator registers).  Smaller R keeps more blocks busy
// where there are few rows.
// ---------------------------------------------------------------------------------------------
constexpr int kSimtThreads = 256;

__device__ __forceinline__ float4 simt_load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 simt_load4(const __nv_bfloat16* p) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);       // a bf16 is the upper half of an fp32
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                     __uint_as_float(v.y & 0xffff0000u));
}
// the first `live` (<= 0: none) of four consecutive elements, zeros after them; `vec`: p is aligned for one load
template <typename T>
__device__ __forceinline__ float4 simt_load_row4(const T* p, int live, bool vec) {
  if (vec && live >= 4) return simt_load4(p);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (live > 0) v.x = to_f32(p[0]);
  if (live > 1) v.y = to_f32(p[1]);
  if (live > 2) v.z = to_f32(p[2]);
  if (live > 3) v.w = to_f32(p[3]);
  return v;
}
// floats between the rows of a tile that is read row-wise in 16-byte pieces: an odd number of pieces, so that eight
// consecutive rows fall into different banks
__host__ __device__ __forceinline__ int simt_ld(int cols) { return (((cols + 3) >> 2) | 1) << 2; }

// acc[r][..] += A[row][0 .. kk) B[0 .. kk)[cols]; A rows `lda`, B rows `ldb` floats apart; kk a multiple of 4
template <int R, int NB>
__device__ __forceinline__ void simt_product(float (&acc)[R][NB * 4], const float* A, int lda, const float* Bt, int ldb, int kk) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  for (int t = 0; t < kk; t += 4) {
    float4 b[4][NB];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int q = 0; q < NB; ++q) b[u][q] = *reinterpret_cast<const float4*>(Bt + (t + u) * ldb + q * 64 + tx * 4);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float4 a = *reinterpret_cast<const float4*>(A + (ty + 16 * r) * lda + t);
      const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int q = 0; q < NB; ++q) {
          acc[r][q * 4 + 0] = fmaf(av[u], b[u][q].x, acc[r][q * 4 + 0]);
          acc[r][q * 4 + 1] = fmaf(av[u], b[u][q].y, acc[r][q * 4 + 1]);
          acc[r][q * 4 + 2] = fmaf(av[u], b[u][q].z, acc[r][q * 4 + 2]);
          acc[r][q * 4 + 3] = fmaf(av[u], b[u][q].w, acc[r][q * 4 + 3]);
        }
    }
  }
}

// s[r][f] += X[row] . Y[tx + 16 f] over `cols` (a multiple of 4) columns; rows of both `ld` floats apart
template <int R>
__device__ __forceinline__ void simt_dots(float (&s)[R][4], const float* X, const float* Y, int ld, int cols) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  for (int c = 0; c < cols; c += 4) {
    float4 y[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) y[f] = *reinterpret_cast<const float4*>(Y + (tx + 16 * f) * ld + c);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float4 x = *reinterpret_cast<const float4*>(X + (ty + 16 * r) * ld + c);
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        s[r][f] = fmaf(x.x, y[f].x, s[r][f]);
        s[r][f] = fmaf(x.y, y[f].y, s[r][f]);
        s[r][f] = fmaf(x.z, y[f].z, s[r][f]);
        s[r][f] = fmaf(x.w, y[f].w, s[r][f]);
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Stage 1.  grid = (ceil(k / 16R), B*H, 2*nsplit).
// blockIdx.z = t*nsplit + s: t = 0 projects K with E, t = 1 projects V with F; split s covers the
// sequence range [s*chunk, min(N,(s+1)*chunk)).  Partial sums are added into KpVp (zeroed before).
// KpVp layout: [2][B*H][k][d] fp32.  E, F: [k][N] shared by all heads, or [H][k][N] (ef_heads = H).
// The next 32 positions travel in registers while the current ones are multiplied.
// ---------------------------------------------------------------------------------------------
constexpr int kSimtTN = 32;            // sequence positions per step
template <typename T, int R, int NB>
__global__ void __launch_bounds__(kSimtThreads, R == 8 && NB == 2 ? 1 : 2)
simt_down_project(const T* __restrict__ Kin, const T* __restrict__ Vin, const T* __restrict__ E,
                  const T* __restrict__ Fin, float* __restrict__ KpVp, int BH, int N, int d, int k,
                  int nsplit, int chunk, int seq_major_heads, int ef_heads) {
  constexpr int kRows = 16 * R, kLd = kSimtTN + 4;
  __shared__ __align__(16) float Ps[kRows * kLd];      // [j][n]
  __shared__ __align__(16) float Xs[kSimtTN * 64 * NB];  // [n][c]
  tc::grid_launch_dependents();
  const int t = blockIdx.z / nsplit, s = blockIdx.z % nsplit;
  const int bh = blockIdx.y, j0 = blockIdx.x * kRows;
  // ef_heads > 0: E and F are [ef_heads][k][N], one pair per head (head = bh % ef_heads)
  const T* __restrict__ P = (t ? Fin : E) + (ef_heads > 0 ? (size_t)(bh % ef_heads) * k * N : 0);
  const HeadView hv = head_view(bh, seq_major_heads, N, d);
  const T* __restrict__ X = (t ? Vin : Kin) + hv.base;
  float* __restrict__ out = KpVp + ((size_t)t * BH + bh) * (size_t)k * d;
  const int n_begin = s * chunk, n_end = min(N, n_begin + chunk);
  const bool vec_p = (N & 3) == 0, vec_x = (d & 3) == 0;

  constexpr int kPV = R / 2, kXV = 2 * NB;             // 16-byte pieces of each tile per thread
  float4 rp[kPV], rx[kXV];
  auto fetch = [&](int n0) {
#pragma unroll
    for (int i = 0; i < kPV; ++i) {
      const int idx = threadIdx.x + i * kSimtThreads, jj = idx >> 3, nn = (idx & 7) * 4;
      rp[i] = simt_load_row4(P + (size_t)(j0 + jj) * N + n0 + nn, j0 + jj < k ? n_end - (n0 + nn) : 0, vec_p);
    }
#pragma unroll
    for (int i = 0; i < kXV; ++i) {
      const int idx = threadIdx.x + i * kSimtThreads, nn = idx / (16 * NB), c = (idx % (16 * NB)) * 4;
      rx[i] = simt_load_row4(X + (size_t)(n0 + nn) * hv.row_stride + c, n0 + nn < n_end ? d - c : 0, vec_x);
    }
  };
  float acc[R][NB * 4];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < NB * 4; ++c) acc[r][c] = 0.f;
  fetch(n_begin);
  for (int n0 = n_begin; n0 < n_end; n0 += kSimtTN) {
#pragma unroll
    for (int i = 0; i < kPV; ++i) {
      const int idx = threadIdx.x + i * kSimtThreads;
      *reinterpret_cast<float4*>(Ps + (idx >> 3) * kLd + (idx & 7) * 4) = rp[i];
    }
#pragma unroll
    for (int i = 0; i < kXV; ++i) *reinterpret_cast<float4*>(Xs + (threadIdx.x + i * kSimtThreads) * 4) = rx[i];
    __syncthreads();
    if (n0 + kSimtTN < n_end) fetch(n0 + kSimtTN);
    simt_product<R, NB>(acc, Ps, kLd, Xs, 64 * NB, kSimtTN);
    __syncthreads();
  }
  tc::grid_dependency_wait();          // KpVp has been zeroed
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int j = j0 + ty + 16 * r;
    if (j >= k) continue;
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int c = q * 64 + tx * 4;
      float* o = out + (size_t)j * d + c;
      if (vec_x && c < d) {
        atomicAdd(reinterpret_cast<float4*>(o), make_float4(acc[r][q * 4], acc[r][q * 4 + 1], acc[r][q * 4 + 2], acc[r][q * 4 + 3]));
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (c + e < d) atomicAdd(o + e, acc[r][q * 4 + e]);
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Stages 2 and 3 share one form: every row (a feature i on the key side, a query n on the query side) weighs a list
// of items (projected keys j, or features i), normalises the weights, and takes the weighted mean of the items'
// vectors (v'_j, or a_i), items in steps of 64 with a running maximum.
//   key side    rows W_i, items K'_j with bias -|k'_j|^2/2 and vectors V'_j   (PERFORMER)
//               weight elu(k'_ji) + 1                                          (RNN)
//               out: weight[bh][i] (b_i or z_i), a32[bh][i][c] fp32, aT16[bh][c][i] fp16 (either may be NULL)
//   query side  rows Q_n, items W_i with bias b_i and vectors a_i               (PERFORMER)
//               weight (elu(q_ni) + 1) z_i                                      (RNN)
// grid = (ceil(rows / 16R), B*H).  Dynamic shared memory: simt_attend_smem().
// ---------------------------------------------------------------------------------------------
inline size_t simt_attend_smem(int R, int NB, int d) {
  return ((size_t)(16 * R + 64) * simt_ld(d) + (size_t)64 * 64 * NB + (size_t)16 * R * 68 + 64) * 4;
}

template <typename T, bool kPerformer, bool kKeySide, int R, int NB>
__global__ void __launch_bounds__(kSimtThreads, R == 8 && NB == 2 ? 1 : 2)
simt_attend(const T* __restrict__ Q, const T* __restrict__ W, const float* __restrict__ KpVp, float* __restrict__ weight,
            float* __restrict__ a32, __half* __restrict__ aT16, T* __restrict__ out, int BH, int N, int d, int k, int p,
            int seq_major_heads) {
  extern __shared__ __align__(16) float smem[];
  constexpr int kRows = 16 * R, kLd = 68;
  const int ld = simt_ld(d), cols = (d + 3) & ~3;
  float* Xs = smem;                        // [16R][ld]    rows
  float* Ys = Xs + kRows * ld;             // [64][ld]     items
  float* Vs = Ys + 64 * ld;                // [64][64 NB]  the items' vectors
  float* Ps = Vs + 64 * 64 * NB;           // [16R][68]    weights
  float* bias = Ps + kRows * kLd;          // [64]
  tc::grid_launch_dependents();
  const int bh = blockIdx.y, row0 = blockIdx.x * kRows;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const bool vec = (d & 3) == 0;
  const int rows = kKeySide ? p : N, items = kKeySide ? k : p;
  const HeadView hv = head_view(bh, seq_major_heads, N, d);
  const float* __restrict__ Vh = kKeySide ? KpVp + ((size_t)BH + bh) * (size_t)k * d : a32 + (size_t)bh * p * d;

  if (kPerformer || !kKeySide) {
    for (int idx = threadIdx.x; idx < kRows * (cols >> 2); idx += kSimtThreads) {
      const int r = idx / (cols >> 2), c = (idx % (cols >> 2)) * 4;
      const T* src = kKeySide ? W + (size_t)(row0 + r) * d : Q + hv.base + (size_t)(row0 + r) * hv.row_stride;
      *reinterpret_cast<float4*>(Xs + r * ld + c) = simt_load_row4(src + c, row0 + r < rows ? d - c : 0, vec);
    }
  }
  // rows are inputs of the call, or complete because the key side was an ordinary launch; the rest comes from the kernels before
  tc::grid_dependency_wait();
  float run_max[R], run_sum[R], acc[R][NB * 4];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    run_max[r] = -INFINITY;
    run_sum[r] = 0.f;
#pragma unroll
    for (int c = 0; c < NB * 4; ++c) acc[r][c] = 0.f;
  }
  for (int i0 = 0; i0 < items; i0 += 64) {
    __syncthreads();
    if (kPerformer || kKeySide) {
      for (int idx = threadIdx.x; idx < 64 * (cols >> 2); idx += kSimtThreads) {
        const int r = idx / (cols >> 2), c = (idx % (cols >> 2)) * 4;
        const int live = i0 + r < items ? d - c : 0;
        float4 y;
        if (kKeySide) y = simt_load_row4(KpVp + ((size_t)bh * k + i0 + r) * d + c, live, vec);
        else y = simt_load_row4(W + (size_t)(i0 + r) * d + c, live, vec);
        *reinterpret_cast<float4*>(Ys + r * ld + c) = y;
      }
    }
    for (int idx = threadIdx.x; idx < 64 * 16 * NB; idx += kSimtThreads) {
      const int r = idx / (16 * NB), c = (idx % (16 * NB)) * 4;
      *reinterpret_cast<float4*>(Vs + idx * 4) = simt_load_row4(Vh + (size_t)(i0 + r) * d + c, i0 + r < items ? d - c : 0, vec);
    }
    if (!kKeySide && threadIdx.x < 64) bias[threadIdx.x] = i0 + threadIdx.x < items ? weight[(size_t)bh * p + i0 + threadIdx.x] : 0.f;
    __syncthreads();
    if (kKeySide && kPerformer) {
      // -|k'_j|^2 / 2: a few threads per key
      constexpr int kPer = kSimtThreads / 64;
      const int r = threadIdx.x / kPer;
      float sq = 0.f;
      for (int c = (threadIdx.x % kPer) * 4; c < cols; c += 4 * kPer) {
        const float4 v = *reinterpret_cast<const float4*>(Ys + r * ld + c);
        sq = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, sq))));
      }
#pragma unroll
      for (int o = 1; o < kPer; o <<= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
      if (threadIdx.x % kPer == 0) bias[r] = -0.5f * sq;
      __syncthreads();
    }
    float s[R][4];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int f = 0; f < 4; ++f) s[r][f] = 0.f;
    if (kPerformer) simt_dots<R>(s, Xs, Ys, ld, cols);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = ty + 16 * r;
      if (kPerformer) {
        float cm = -INFINITY;
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          s[r][f] = i0 + tx + 16 * f < items ? s[r][f] + bias[tx + 16 * f] : -INFINITY;
          cm = fmaxf(cm, s[r][f]);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, o));
        const float new_max = fmaxf(run_max[r], cm);
        const float rescale = expf(run_max[r] - new_max);       // exp(-inf) = 0 on the first step
        run_max[r] = new_max;
        run_sum[r] *= rescale;
#pragma unroll
        for (int c = 0; c < NB * 4; ++c) acc[r][c] *= rescale;
#pragma unroll
        for (int f = 0; f < 4; ++f) s[r][f] = expf(s[r][f] - new_max);
      } else {
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          const int i = tx + 16 * f;
          float v = 0.f;
          if (i0 + i < items) {
            const float x = kKeySide ? (row0 + row < rows ? Ys[i * ld + row0 + row] : 0.f) : Xs[row * ld + i0 + i];
            v = (x > 0.f ? x + 1.f : expf(x)) * (kKeySide ? 1.f : bias[i]);
          }
          s[r][f] = v;
        }
      }
      float part = 0.f;                                           // this thread's share of the row
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        part += s[r][f];
        Ps[row * kLd + tx + 16 * f] = s[r][f];
      }
      run_sum[r] += part;
    }
    __syncthreads();
    simt_product<R, NB>(acc, Ps, kLd, Vs, 64 * NB, min(64, (items - i0 + 3) & ~3));
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    float sum = run_sum[r];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const int row = row0 + ty + 16 * r;
    if (row >= rows) continue;
    const float inv = 1.f / fmaxf(sum, 1.17549435e-38f);
    if (kKeySide && tx == 0) weight[(size_t)bh * p + row] = kPerformer ? run_max[r] + logf(sum) : sum;
#pragma unroll
    for (int q = 0; q < NB; ++q) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int c = q * 64 + tx * 4 + e;
        if (c >= d) continue;
        const float v = acc[r][q * 4 + e] * inv;
        if (kKeySide) {
          if (a32) a32[((size_t)bh * p + row) * d + c] = v;
          if (aT16) aT16[((size_t)bh * d + c) * p + row] = __float2half_rn(v);
        } else {
          store_out(out + hv.base + (size_t)row * hv.row_stride + c, v);
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// The linear maps of Eq. (2) and the contraction of un-projected inputs on CUDA cores: a plain
// batched C = A B with fp32 accumulation.  A: [Z][M][K] (batch stride a_stride, 0 = shared),
// B: [Z][K][ncols] (b_stride likewise), both row-major.  grid = (ceil(ncols/32), ceil(M/32), Z),
// block = 256 (a 32 x 32 tile of C, four rows per thread).
// head_d == 0: C is [Z][M][ncols] row-major.  head_d > 0: C is the K', V' workspace, fp32
// [(z0 + z) * ncols/head_d + col/head_d][M][head_d]: column block h of the product is head h's.
// ---------------------------------------------------------------------------------------------
template <typename TA, typename TB, typename TC>
__global__ void __launch_bounds__(256)
simt_linear_map(const TA* __restrict__ A, const TB* __restrict__ Bm, TC* __restrict__ C, int M, int K, int ncols,
                size_t a_stride, size_t b_stride, int head_d, int z0) {
  __shared__ float sa[32][33];
  __shared__ float sb[32][33];
  const int z = blockIdx.z;
  const TA* Az = A + (size_t)z * a_stride;
  const TB* Bz = Bm + (size_t)z * b_stride;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;      // ty: 0..7
  const int row0 = blockIdx.y * 32, col0 = blockIdx.x * 32;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int k0 = 0; k0 < K; k0 += 32) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int ar = row0 + ty + 8 * r, ak = k0 + tx;
      sa[ty + 8 * r][tx] = (ar < M && ak < K) ? to_f32(Az[(size_t)ar * K + ak]) : 0.f;
      const int bk = k0 + ty + 8 * r, bc = col0 + tx;
      sb[ty + 8 * r][tx] = (bk < K && bc < ncols) ? to_f32(Bz[(size_t)bk * ncols + bc]) : 0.f;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < 32; ++kk) {
      const float b = sb[kk][tx];
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[r] = fmaf(sa[ty + 8 * r][kk], b, acc[r]);
    }
    __syncthreads();
  }
  const int col = col0 + tx;
  if (col >= ncols) return;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int row = row0 + ty + 8 * r;
    if (row >= M) continue;
    if (head_d > 0) {
      const size_t head = (size_t)(z0 + z) * (ncols / head_d) + col / head_d;
      store_out(C + (head * M + row) * head_d + col % head_d, acc[r]);
    } else {
      store_out(C + ((size_t)z * M + row) * ncols + col, acc[r]);
    }
  }
}

}  // namespace flurka
