// Backward pass of the FLuRKA forward (arxiv 2306.15799, Eq. (2); the paper trains these models but
// prints no backward formulas: this is the chain rule through the three stages, CUDA cores, fp32).
//
// With the forward's per-feature summaries  a_i (a d-vector) and b_i = log z_i,  the output is
//     O_n = sum_i P_ni a_i,     P_n. = softmax_i(l_ni),   l_ni = w_i.q_n + b_i          (PERFORMER)
//                                                          l_ni = log(elu(q_ni)+1) + b_i  (RNN)
// and   a_i = sum_j A_ij v'_j,  b_i = log sum_j exp(L_ji),  A_i. = softmax_j(L_.i),
//     L_ji = w_i.k'_j - |k'_j|^2/2  (PERFORMER),   L_ji = log(elu(k'_ji)+1)  (RNN).
// Given dO:
//   query side   c_ni = P_ni (a_i.dO_n - O_n.dO_n)   (sums to zero over i)
//                dq_n = sum_i c_ni w_i  (PERFORMER; the -q_n sum_i c_ni term vanishes),
//                dq_ni = c_ni elu'(q_ni)/(elu(q_ni)+1)  (RNN)
//                da_i = sum_n P_ni dO_n,   db_i = sum_n c_ni
//   key side     g_ij = da_i.v'_j + e_i with e_i = db_i - da_i.a_i = -sum_n P_ni (O_n.dO_n) (db itself is never formed),
//                 dL_ji = A_ij g_ij,   dv'_j = sum_i A_ij da_i,
//                dk'_j = sum_i dL_ji (w_i - k'_j)  (PERFORMER),  dk'_ji = dL_ji elu'(k'_ji)/(elu(k'_ji)+1)  (RNN)
//   projections  dK = E^T dK',  dV = F^T dV',  dE = sum_heads dK' K^T,  dF = sum_heads dV' V^T.
#pragma once

#include "simt_kernels.cuh"

namespace flurka {

__device__ __forceinline__ float elu1(float x) { return x > 0.f ? x + 1.f : expf(x); }
__device__ __forceinline__ float elu1_slope(float x) { return x > 0.f ? 1.f : expf(x); }

// ---------------------------------------------------------------------------------------------
// Query side.  grid = (ceil(N / 16R), B*H); block = 256 (the building blocks of simt_kernels.cuh); 64 features at a time.
// With g_ni = a_i . dO_n, O_n . dO_n = sum_i P_ni g_ni: sweep 1 is the dot products l and g with a running maximum, sum and
// weighted sum; sweep 2 forms them again, then c_ni, dq += C W, da += P^T dO (C and P^T through shared memory), e_i.
// RNN: the weights come from the Q tile, no l, no dq product.  da, e (fp32, zeroed before) are added to with atomics: every
// row tile of a head contributes.  Six units of 2 N m d operations (RNN: three) at the FFMA rate of the register tiles.
// fp32, B = 2, H = 8, N = 4096, d = 64, m = 256, against one feature per lane and scalar reads: 1667 -> 543 us
// (B = 1, H = 2, N = 1024, m = 128: 78 -> 30; RNN, first sizes: 250 -> 109; RNN, bf16, d = 128: 655 -> 399).
// R = 2 (tiles of 32 rows) where tiles of 64 would be fewer than SMs.
// ---------------------------------------------------------------------------------------------
// floats of shared memory; a product reads up to 64 NB columns of a row, so a tile it reads has another one behind it
__host__ __device__ inline size_t simt_bwd_query_floats(int d, int R, bool performer) {
  return (size_t)simt_ld(d) * (2 * 16 * R + (performer ? 2 : 1) * 64) + 64 * (16 * R + 4) + (performer ? 16 * R * 68 : 0) + 128;
}
template <typename T, bool kPerformer, int R, int NB>
__global__ void __launch_bounds__(kSimtThreads, NB == 1 ? 2 : 1)
simt_bwd_query_side(const T* __restrict__ Q, const T* __restrict__ W, const T* __restrict__ dO,
                    const float* __restrict__ weight, const float* __restrict__ a32, T* __restrict__ dQ,
                    float* __restrict__ da, float* __restrict__ ei, int N, int d, int p, int seq_major_heads) {
  extern __shared__ __align__(16) float smem[];
  constexpr int kRows = 16 * R, kLdP = kRows + 4, kLdC = 68;
  const int ld = simt_ld(d), cols = (d + 3) & ~3;
  float* Gs = smem;                          // [kRows][ld]  dO tile
  float* Qs = Gs + kRows * ld;               // [kRows][ld]
  float* As = Qs + kRows * ld;               // [64][ld]     a of the chunk's features
  float* Ws = As + 64 * ld;                  // [64][ld]     PERFORMER: W of the chunk's features
  float* Pt = Ws + (kPerformer ? 64 * ld : 0);   // [64 features][kRows]
  float* Cs = Pt + 64 * kLdP;                // [kRows][64]  PERFORMER
  __shared__ float ws[64];
  __shared__ float es[8][64];

  const int bh = blockIdx.y, n0 = blockIdx.x * kRows;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, warp = tid >> 5, lane = tid & 31;
  const HeadView hv = head_view(bh, seq_major_heads, N, d);
  const float* __restrict__ ah = a32 + (size_t)bh * p * d;
  const float* __restrict__ wh = weight + (size_t)bh * p;
  const bool vec_d = (d & 3) == 0;
  const int pieces = ld >> 2;

  for (int e = tid; e < kRows * pieces; e += kSimtThreads) {
    const int r = e / pieces, c = (e % pieces) * 4, live = n0 + r < N ? d - c : 0;
    const size_t at = hv.base + (size_t)(n0 + r) * hv.row_stride + c;
    *reinterpret_cast<float4*>(Qs + r * ld + c) = simt_load_row4(Q + at, live, vec_d);
    *reinterpret_cast<float4*>(Gs + r * ld + c) = simt_load_row4(dO + at, live, vec_d);
  }
  auto stage_chunk = [&](int i0) {
    __syncthreads();
    for (int e = tid; e < 64 * pieces; e += kSimtThreads) {
      const int i = e / pieces, c = (e % pieces) * 4, live = i0 + i < p ? d - c : 0;
      const size_t at = (size_t)(i0 + i) * d + c;
      if (kPerformer) *reinterpret_cast<float4*>(Ws + i * ld + c) = simt_load_row4(W + at, live, vec_d);
      *reinterpret_cast<float4*>(As + i * ld + c) = simt_load_row4(ah + at, live, vec_d);
    }
    if (tid < 64) ws[tid] = i0 + tid < p ? wh[i0 + tid] : 0.f;
    __syncthreads();
  };
  // this thread's rows ty + 16 r x features i0 + tx + 16 f: PERFORMER the logit, RNN the weight itself; and g
  auto form = [&](int i0, float (&s)[R][4], float (&g)[R][4]) {
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int f = 0; f < 4; ++f) s[r][f] = g[r][f] = 0.f;
    if (kPerformer) simt_dots<R>(s, Qs, Ws, ld, cols);
    simt_dots<R>(g, Gs, As, ld, cols);
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const int i = tx + 16 * f;
        const bool live = i0 + i < p;
        if (kPerformer) s[r][f] = live ? s[r][f] + ws[i] : -INFINITY;
        else s[r][f] = live ? elu1(Qs[(ty + 16 * r) * ld + i0 + i]) * ws[i] : 0.f;
      }
  };

  // ---- sweep 1: row maximum, sum and weighted sum of g
  float run_max[R], sum[R], t[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    run_max[r] = kPerformer ? -INFINITY : 0.f;
    sum[r] = t[r] = 0.f;
  }
  for (int i0 = 0; i0 < p; i0 += 64) {
    stage_chunk(i0);
    float s[R][4], g[R][4];
    form(i0, s, g);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (kPerformer) {
        float cm = fmaxf(fmaxf(s[r][0], s[r][1]), fmaxf(s[r][2], s[r][3]));
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, o));
        const float new_max = fmaxf(run_max[r], cm);
        const float rescale = expf(run_max[r] - new_max);
        run_max[r] = new_max;
        sum[r] *= rescale;
        t[r] *= rescale;
      }
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const float pv = kPerformer ? expf(s[r][f] - run_max[r]) : s[r][f];
        sum[r] += pv;
        t[r] = fmaf(pv, g[r][f], t[r]);
      }
    }
  }
  float inv_sum[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      sum[r] += __shfl_xor_sync(0xffffffffu, sum[r], o);
      t[r] += __shfl_xor_sync(0xffffffffu, t[r], o);
    }
    const bool row_live = n0 + ty + 16 * r < N;
    inv_sum[r] = row_live ? 1.f / fmaxf(sum[r], 1.17549435e-38f) : 0.f;     // rows past the end weigh nothing
    t[r] *= inv_sum[r];
  }

  // ---- sweep 2: c_ni, dq_n, da_i, e_i
  float dq[R][NB * 4];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < NB * 4; ++c) dq[r][c] = 0.f;
  for (int i0 = 0; i0 < p; i0 += 64) {
    stage_chunk(i0);
    float s[R][4], g[R][4];
    form(i0, s, g);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const int i = tx + 16 * f;
      float e_part = 0.f;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int row = ty + 16 * r;
        const float P = (kPerformer ? expf(s[r][f] - run_max[r]) : s[r][f]) * inv_sum[r];
        const float cv = P * (g[r][f] - t[r]);
        e_part = fmaf(-P, t[r], e_part);
        Pt[i * kLdP + row] = P;
        if (kPerformer) {
          Cs[row * kLdC + i] = cv;
        } else if (i0 + i < p && n0 + row < N) {
          // feature i is column i of the row: d log(elu(x)+1)/dx = elu'(x)/(elu(x)+1)
          const float x = Qs[row * ld + i0 + i];
          store_out(dQ + hv.base + (size_t)(n0 + row) * hv.row_stride + i0 + i, cv * elu1_slope(x) / elu1(x));
        }
      }
      e_part += __shfl_xor_sync(0xffffffffu, e_part, 16);
      if (lane < 16) es[warp][i] = e_part;
    }
    __syncthreads();
    if (kPerformer) simt_product<R, NB>(dq, Cs, kLdC, Ws, ld, 64);
    float acc[4][NB * 4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < NB * 4; ++c) acc[r][c] = 0.f;
    simt_product<4, NB>(acc, Pt, kLdP, Gs, ld, kRows);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = i0 + ty + 16 * r;
      if (i >= p) continue;
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        const int c = q * 64 + tx * 4;
        float* at = da + ((size_t)bh * p + i) * d + c;
        if (vec_d && c < d) {
          atomicAdd(reinterpret_cast<float4*>(at), make_float4(acc[r][q * 4], acc[r][q * 4 + 1], acc[r][q * 4 + 2], acc[r][q * 4 + 3]));
        } else {
#pragma unroll
          for (int x = 0; x < 4; ++x)
            if (c + x < d) atomicAdd(at + x, acc[r][q * 4 + x]);
        }
      }
    }
    if (tid < 64 && i0 + tid < p) {
      float e = 0.f;
#pragma unroll
      for (int w8 = 0; w8 < 8; ++w8) e += es[w8][tid];
      atomicAdd(ei + (size_t)bh * p + i0 + tid, e);
    }
  }
  if (kPerformer) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int n = n0 + ty + 16 * r;
      if (n >= N) continue;
#pragma unroll
      for (int q = 0; q < NB; ++q)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int c = q * 64 + tx * 4 + x;
          if (c < d) store_out(dQ + hv.base + (size_t)n * hv.row_stride + c, dq[r][q * 4 + x]);
        }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Key side.  grid = (ceil(k / 16R), B*H); block = 256 (the building blocks of simt_kernels.cuh): a block owns 16 R
// projected keys and walks the features 64 at a time: the exponents k'_j . w_i and the products v'_j . da_i are dot
// products of rows, the weights A and dL go through shared memory, and dv'_j = sum_i A_ij da_i,
// dk'_j = sum_i dL_ij w_i - k'_j sum_i dL_ij are register-tile products that read da and W where the dot products left
// them.  Inputs: K', V' (KpVp), W, b (weight), da, e.  Outputs: dK', dV' as two bf16 terms into `split`
// ([2][2 terms][k][BH][d], what k5_bwd_projections reads), or, split == NULL, as fp32 into dKpVp [2][B*H][k][d].
// kD: the head dimension where it is known at compile time (all loads of a step are then in flight together, and
// the next step's travel in registers under this step's products), or 0.
// ---------------------------------------------------------------------------------------------
inline size_t simt_bwd_key_side_smem(int R, int d) {
  return ((size_t)(2 * 64 + 2 * 16 * R) * simt_ld(d) + (size_t)2 * 16 * R * 68 + 128 + 128) * 4;
}
// four consecutive values of a row of dK' or dV'
__device__ __forceinline__ void simt_put4(float* f32, __nv_bfloat16* hi, size_t term, const float (&v)[4], int live, bool vec) {
  if (hi) {
    uint32_t h[2], l[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const __nv_bfloat162 h2 = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
      const __nv_bfloat162 l2 = __floats2bfloat162_rn(v[2 * e] - __low2float(h2), v[2 * e + 1] - __high2float(h2));
      h[e] = *reinterpret_cast<const uint32_t*>(&h2);
      l[e] = *reinterpret_cast<const uint32_t*>(&l2);
    }
    *reinterpret_cast<uint2*>(hi) = make_uint2(h[0], h[1]);            // (only for d = 64, 128: live is 4 or <= 0)
    *reinterpret_cast<uint2*>(hi + term) = make_uint2(l[0], l[1]);
  } else if (vec && live >= 4) {
    *reinterpret_cast<float4*>(f32) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (e < live) f32[e] = v[e];
  }
}

template <typename T, bool kPerformer, int R, int NB, int kD>
__global__ void __launch_bounds__(256, NB == 1 && kD > 0 && !kPerformer ? 3 : (NB == 1 ? 2 : 1))
simt_bwd_key_side(const float* __restrict__ KpVp, const T* __restrict__ W, const float* __restrict__ weight,
                  const float* __restrict__ da, const float* __restrict__ ei, float* __restrict__ dKpVp,
                  __nv_bfloat16* __restrict__ split, int BH, int d_rt, int k, int p) {
  extern __shared__ __align__(16) float smem[];
  constexpr int kRows = 16 * R, kLd = 68;
  const int d = kD > 0 ? kD : d_rt;
  const int ld = kD > 0 ? kD + 4 : simt_ld(d), cols = (d + 3) & ~3, pieces = cols >> 2;
  float* Ks = smem;                        // [16R][ld]
  float* Vs = Ks + kRows * ld;             // [16R][ld]
  float* Ws = Vs + kRows * ld;             // [64][ld]
  float* Ds = Ws + 64 * ld;                // [64][ld]  da (the products below may read past its end: columns nobody keeps)
  float* As = Ds + 64 * ld;                // [16R][68] A
  float* Ls = As + kRows * kLd;            // [16R][68] dL (RNN: dk')
  float* bs = Ls + kRows * kLd;            // [64] b_i (RNN: 1 / z_i)
  float* es = bs + 64;                     // [64] e_i
  float* nrm = es + 64;                    // [16R] |k'_j|^2 / 2
  const int bh = blockIdx.y, j0 = blockIdx.x * kRows;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const bool vec = kD > 0 || (d & 3) == 0;
  const float* __restrict__ Kp = KpVp + (size_t)bh * k * d;
  const float* __restrict__ Vp = KpVp + ((size_t)BH + bh) * (size_t)k * d;
  const float* __restrict__ dah = da + (size_t)bh * p * d;
  tc::grid_launch_dependents();
  tc::grid_dependency_wait();

  // the step's W and da: into registers first where d is known
  constexpr int kPre = kD > 0 ? 64 * (kD / 4) / kSimtThreads : 1;
  float4 rw[kPre], rd[kPre];
  float rb = 0.f, re = 0.f;
  auto fetch = [&](int i0) {
    if constexpr (kD > 0) {
#pragma unroll
      for (int u = 0; u < kPre; ++u) {
        const int idx = threadIdx.x + u * kSimtThreads, r = idx / (kD / 4), c = (idx % (kD / 4)) * 4;
        const int live = i0 + r < p ? 4 : 0;
        rd[u] = simt_load_row4(dah + (size_t)(i0 + r) * kD + c, live, true);
        if (kPerformer) rw[u] = simt_load_row4(W + (size_t)(i0 + r) * kD + c, live, true);
      }
    }
    if (threadIdx.x < 64) {
      const bool in = i0 + threadIdx.x < p;
      rb = in ? weight[(size_t)bh * p + i0 + threadIdx.x] : 1.f;
      re = in ? ei[(size_t)bh * p + i0 + threadIdx.x] : 0.f;
    }
  };
  if constexpr (kD > 0) {
    constexpr int kKV = kRows * (kD / 4) / kSimtThreads;
    float4 rk[kKV], rv[kKV];
#pragma unroll
    for (int u = 0; u < kKV; ++u) {
      const int idx = threadIdx.x + u * kSimtThreads, r = idx / (kD / 4), c = (idx % (kD / 4)) * 4;
      const int live = j0 + r < k ? 4 : 0;
      rk[u] = simt_load_row4(Kp + (size_t)(j0 + r) * kD + c, live, true);
      rv[u] = simt_load_row4(Vp + (size_t)(j0 + r) * kD + c, live, true);
    }
    fetch(0);
#pragma unroll
    for (int u = 0; u < kKV; ++u) {
      const int idx = threadIdx.x + u * kSimtThreads, r = idx / (kD / 4), c = (idx % (kD / 4)) * 4;
      *reinterpret_cast<float4*>(Ks + r * ld + c) = rk[u];
      *reinterpret_cast<float4*>(Vs + r * ld + c) = rv[u];
    }
  } else {
    for (int idx = threadIdx.x; idx < kRows * pieces; idx += kSimtThreads) {
      const int r = idx / pieces, c = (idx % pieces) * 4;
      const int live = j0 + r < k ? d - c : 0;
      *reinterpret_cast<float4*>(Ks + r * ld + c) = simt_load_row4(Kp + (size_t)(j0 + r) * d + c, live, vec);
      *reinterpret_cast<float4*>(Vs + r * ld + c) = simt_load_row4(Vp + (size_t)(j0 + r) * d + c, live, vec);
    }
    fetch(0);
  }
  float dk[kPerformer ? R : 1][NB * 4], dv[R][NB * 4], dl_sum[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    dl_sum[r] = 0.f;
#pragma unroll
    for (int c = 0; c < NB * 4; ++c) {
      dv[r][c] = 0.f;
      if (kPerformer) dk[r][c] = 0.f;
    }
  }
  const size_t hd = (size_t)BH * d, term = (size_t)k * hd;
  if (kPerformer) {
    __syncthreads();
    if (threadIdx.x < kRows) {
      // as the forward's key side adds them up, rounding for rounding: its error then cancels between L_ij and b_i
      float s[4] = {0.f, 0.f, 0.f, 0.f};
      for (int c = 0; c < cols; c += 16) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (c + 4 * q >= cols) break;
          const float4 v = *reinterpret_cast<const float4*>(Ks + threadIdx.x * ld + c + 4 * q);
          s[q] = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, s[q]))));
        }
      }
      nrm[threadIdx.x] = 0.5f * ((s[0] + s[1]) + (s[2] + s[3]));
    }
  }
  for (int i0 = 0; i0 < p; i0 += 64) {
    if (i0 > 0) __syncthreads();
    if constexpr (kD > 0) {
#pragma unroll
      for (int u = 0; u < kPre; ++u) {
        const int idx = threadIdx.x + u * kSimtThreads, r = idx / (kD / 4), c = (idx % (kD / 4)) * 4;
        *reinterpret_cast<float4*>(Ds + r * ld + c) = rd[u];
        if (kPerformer) *reinterpret_cast<float4*>(Ws + r * ld + c) = rw[u];
      }
    } else {
      for (int idx = threadIdx.x; idx < 64 * pieces; idx += kSimtThreads) {
        const int r = idx / pieces, c = (idx % pieces) * 4;
        const int live = i0 + r < p ? d - c : 0;
        if (kPerformer) *reinterpret_cast<float4*>(Ws + r * ld + c) = simt_load_row4(W + (size_t)(i0 + r) * d + c, live, vec);
        *reinterpret_cast<float4*>(Ds + r * ld + c) = simt_load_row4(dah + (size_t)(i0 + r) * d + c, live, vec);
      }
    }
    if (threadIdx.x < 64) {
      bs[threadIdx.x] = kPerformer ? rb : 1.f / rb;
      es[threadIdx.x] = re;
    }
    __syncthreads();
    if (i0 + 64 < p) fetch(i0 + 64);
    float s[R][4], t[R][4];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int f = 0; f < 4; ++f) s[r][f] = t[r][f] = 0.f;
    if (kPerformer) simt_dots<R>(s, Ks, Ws, ld, cols);
    simt_dots<R>(t, Vs, Ds, ld, cols);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = ty + 16 * r;
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const int i = tx + 16 * f;
        const bool live = i0 + i < p && j0 + row < k;
        float A, factor = 1.f;
        if (kPerformer) {
          A = expf(s[r][f] - nrm[row] - bs[i]);         // b_i = log sum_j exp(L_ji): A <= 1
        } else {
          // RNN: feature i is column i0 + i (p = d); d log(elu(x) + 1) / dx = elu'(x) / (elu(x) + 1)
          const float x = live ? Ks[row * ld + i0 + i] : 0.f;
          A = (fmaxf(x, 0.f) + expf(fminf(x, 0.f))) * bs[i];
          factor = x > 0.f ? 1.f / (x + 1.f) : 1.f;
        }
        if (!live) A = 0.f;
        const float dL = A * (t[r][f] + es[i]);
        dl_sum[r] += dL;
        As[row * kLd + i] = A;
        Ls[row * kLd + i] = dL * factor;
      }
    }
    __syncthreads();
    const int kk = min(64, (p - i0 + 3) & ~3);
    if constexpr (!kPerformer) {
      // dk' of these 64 columns, four at a time
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const int row = ty + 16 * u, c = tx * 4;
        const float4 x = *reinterpret_cast<const float4*>(Ls + row * kLd + c);
        const float v[4] = {x.x, x.y, x.z, x.w};
        if (j0 + row < k && i0 + c < d)
          simt_put4(dKpVp + ((size_t)bh * k + j0 + row) * d + i0 + c,
                    split ? split + (size_t)(j0 + row) * hd + (size_t)bh * d + i0 + c : nullptr, term, v, d - i0 - c, vec);
      }
    }
    simt_product<R, NB>(dv, As, kLd, Ds, ld, kk);
    if constexpr (kPerformer) simt_product<R, NB>(dk, Ls, kLd, Ws, ld, kk);
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    float ds = dl_sum[r];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) ds += __shfl_xor_sync(0xffffffffu, ds, o);
    const int row = ty + 16 * r;
    if (j0 + row >= k) continue;
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int c0 = q * 64 + tx * 4;
      if (c0 >= d) continue;
      __nv_bfloat16* sp = split ? split + (size_t)(j0 + row) * hd + (size_t)bh * d + c0 : nullptr;
      float v[4];
      if constexpr (kPerformer) {
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = dk[r][q * 4 + e] - Ks[row * ld + c0 + e] * ds;
        simt_put4(dKpVp + ((size_t)bh * k + j0 + row) * d + c0, sp, term, v, d - c0, vec);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = dv[r][q * 4 + e];
      simt_put4(dKpVp + (((size_t)BH + bh) * k + j0 + row) * d + c0, sp ? sp + 2 * term : nullptr, term, v, d - c0, vec);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// dK = E^T dK', dV = F^T dV'.  grid = (ceil(N / 16R), B*H, 2 ceil(d / 64)); block = 256.  E, F: [k][N] (or [H][k][N],
// ef_heads = H).  Both operands lie [j][..], so a thread's R consecutive positions x 4 columns are an outer product per
// projected key, read from shared memory in 16-byte pieces (3 per 32 FFMA with R = 8; FFMA-bound, as stage 1); the next
// 32 keys travel in registers under this step's products.  B = 2, H = 8, N = 4096, d = 64, k = 256, fp32, against scalar
// reads and four rows per warp: 335 -> 115 us (B = 1, H = 2, N = 1024, k = 128: 20.5 -> 6.6).  R = 2 keeps more blocks busy where 128-row tiles would be fewer than SMs.
// ---------------------------------------------------------------------------------------------
template <typename T, int R>
__global__ void __launch_bounds__(kSimtThreads)
simt_bwd_inputs(const T* __restrict__ E, const T* __restrict__ F, const float* __restrict__ dKpVp,
                T* __restrict__ dK, T* __restrict__ dV, int BH, int N, int d, int k, int seq_major_heads,
                int ef_heads) {
  constexpr int kRows = 16 * R, kA = kRows / 32;   // 16-byte pieces of the E tile per thread
  __shared__ __align__(16) float Ps[32][kRows];    // [j][n]
  __shared__ __align__(16) float Gs[32][64];       // [j][c]
  const int cb = (d + 63) / 64;
  const int t = blockIdx.z / cb, c0 = (blockIdx.z % cb) * 64, bh = blockIdx.y, n0 = blockIdx.x * kRows;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const T* __restrict__ P = (t ? F : E) + (ef_heads > 0 ? (size_t)(bh % ef_heads) * k * N : 0);
  const float* __restrict__ G = dKpVp + ((size_t)t * BH + bh) * (size_t)k * d;
  const HeadView hv = head_view(bh, seq_major_heads, N, d);
  T* __restrict__ out = (t ? dV : dK) + hv.base;
  const bool vec_n = (N & 3) == 0, vec_d = (d & 3) == 0;
  float4 pa[kA], pg[2];
  auto fetch = [&](int j0) {
#pragma unroll
    for (int q = 0; q < kA; ++q) {
      const int e = threadIdx.x + q * kSimtThreads, jj = e / (kRows / 4), n = n0 + (e % (kRows / 4)) * 4;
      pa[q] = simt_load_row4(P + (size_t)(j0 + jj) * N + n, j0 + jj < k ? N - n : 0, vec_n);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = threadIdx.x + q * kSimtThreads, jj = e >> 4, c = c0 + (e & 15) * 4;
      pg[q] = simt_load_row4(G + (size_t)(j0 + jj) * d + c, j0 + jj < k ? d - c : 0, vec_d);
    }
  };
  float acc[R][4];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[r][b] = 0.f;
  fetch(0);
  for (int j0 = 0; j0 < k; j0 += 32) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kA; ++q) reinterpret_cast<float4*>(&Ps[0][0])[threadIdx.x + q * kSimtThreads] = pa[q];
#pragma unroll
    for (int q = 0; q < 2; ++q) reinterpret_cast<float4*>(&Gs[0][0])[threadIdx.x + q * kSimtThreads] = pg[q];
    __syncthreads();
    if (j0 + 32 < k) fetch(j0 + 32);
#pragma unroll 4
    for (int jj = 0; jj < 32; ++jj) {
      const float4 g = *reinterpret_cast<const float4*>(&Gs[jj][tx * 4]);
      float p[R];
#pragma unroll
      for (int r = 0; r < R; r += 2) {
        const float2 v = *reinterpret_cast<const float2*>(&Ps[jj][ty * R + r]);
        p[r] = v.x;
        p[r + 1] = v.y;
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        acc[r][0] = fmaf(p[r], g.x, acc[r][0]);
        acc[r][1] = fmaf(p[r], g.y, acc[r][1]);
        acc[r][2] = fmaf(p[r], g.z, acc[r][2]);
        acc[r][3] = fmaf(p[r], g.w, acc[r][3]);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int n = n0 + ty * R + r;
    if (n >= N) continue;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int c = c0 + tx * 4 + b;
      if (c < d) store_out(out + (size_t)n * hv.row_stride + c, acc[r][b]);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// dE = sum over heads of dK' K^T, dF = sum over heads of dV' V^T.  grid = (ceil(N / 64), ceil(k / 16R),
// 2 * max(ef_heads, 1)); block = 256.  With shared E, F the sum runs over all B*H heads; with one pair per head over the
// batch only.  Both operands are rows of d values: dot products 32 columns at a time (simt_dots), the next step's
// operands in registers.  B = 2, H = 8, N = 4096, d = 64, k = 256, fp32, against scalar reads and four outputs per
// thread: 431 -> 128 us (small as above: 12.9 -> 6.1).  R as above.
// ---------------------------------------------------------------------------------------------
template <typename T, int R>
__global__ void __launch_bounds__(kSimtThreads)
simt_bwd_projections(const T* __restrict__ Kin, const T* __restrict__ Vin, const float* __restrict__ dKpVp,
                     T* __restrict__ dE, T* __restrict__ dF, int BH, int N, int d, int k, int seq_major_heads,
                     int ef_heads) {
  constexpr int kLd = 36, kG = (16 * R) / 32 > 0 ? (16 * R) / 32 : 1;   // simt_ld(32); pieces of dK' per thread
  __shared__ __align__(16) float Gs[16 * R][kLd];  // [j][c]
  __shared__ __align__(16) float Xs[64][kLd];      // [n][c]
  const int groups = ef_heads > 0 ? ef_heads : 1;
  const int t = blockIdx.z / groups, eh = blockIdx.z % groups;
  const int n0 = blockIdx.x * 64, j0 = blockIdx.y * (16 * R);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int row8 = threadIdx.x >> 3, col4 = (threadIdx.x & 7) * 4;
  const bool vec_d = (d & 3) == 0;
  const T* __restrict__ Xin = t ? Vin : Kin;
  float4 pg[kG], px[2];
  auto fetch = [&](int bh, int c0) {
    const float* __restrict__ G = dKpVp + ((size_t)t * BH + bh) * (size_t)k * d;
    const HeadView hv = head_view(bh, seq_major_heads, N, d);
    const int c = c0 + col4;
#pragma unroll
    for (int q = 0; q < kG; ++q) {
      const int j = j0 + row8 + 32 * q;
      pg[q] = simt_load_row4(G + (size_t)j * d + c, j < k ? d - c : 0, vec_d);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int n = n0 + row8 + 32 * q;
      px[q] = simt_load_row4(Xin + hv.base + (size_t)n * hv.row_stride + c, n < N ? d - c : 0, vec_d);
    }
  };
  float acc[R][4];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int f = 0; f < 4; ++f) acc[r][f] = 0.f;
  int bh = eh, c0 = 0;
  fetch(bh, c0);
  while (bh < BH) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kG; ++q)
      if (row8 + 32 * q < 16 * R) *reinterpret_cast<float4*>(&Gs[row8 + 32 * q][col4]) = pg[q];
#pragma unroll
    for (int q = 0; q < 2; ++q) *reinterpret_cast<float4*>(&Xs[row8 + 32 * q][col4]) = px[q];
    __syncthreads();
    const int cols = min(32, (d - c0 + 3) & ~3);
    c0 += 32;
    if (c0 >= d) { c0 = 0; bh += groups; }
    if (bh < BH) fetch(bh, c0);
    simt_dots<R>(acc, &Gs[0][0], &Xs[0][0], kLd, cols);
  }
  T* __restrict__ out = (t ? dF : dE) + (size_t)eh * k * N;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int j = j0 + ty + 16 * r;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const int n = n0 + tx + 16 * f;
      if (j < k && n < N) store_out(out + (size_t)j * N + n, acc[r][f]);
    }
  }
}

}  // namespace flurka
