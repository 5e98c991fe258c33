// Host side of the tensor-core (tcgen05 / TMEM / TMA) kernels: tensor-map encoding and launches.
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <string.h>

#include <algorithm>

#include "clear.cuh"
#include "k0_linear_maps.cuh"
#include "k1_down_project.cuh"
#include "k1_down_project_pair.cuh"
#include "k2_key_side.cuh"
#include "k3_query_side.cuh"
#include "k3_query_units.cuh"
#include "k4_bwd_query_wide.cuh"
#include "k5_bwd_projections.cuh"
#include "k6_bwd_key_side.cuh"
#include "k7_bwd_query_rnn.cuh"
#include "k8_bwd_query_units.cuh"
#include "k10_bwd_key_performer.cuh"
#include "k9_bwd_key_rnn.cuh"
#include "pad_rows.cuh"

namespace flurka {

// Launch with programmatic stream serialisation: the kernel may be scheduled while the previous
// kernel in the stream is finishing (its CTAs call griddepcontrol.launch_dependents) and waits in
// griddepcontrol.wait before it touches that kernel's results.  Every kernel of a chain waits somewhere before it
// ends, so that the completion of one says that all before it are complete.
// chained = false: an ordinary launch, which starts when everything before it in the stream is complete.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_cluster_after_predecessor(int cluster, void (*fn)(KArgs...), dim3 grid, int block, size_t smem,
                                                    cudaStream_t st, bool chained, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)block, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = chained ? 1 : 0;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, fn, KArgs(args)...);
}
// (kernels with __cluster_dims__ bring their own cluster size)
template <typename... KArgs, typename... Args>
inline cudaError_t launch_after_predecessor(void (*fn)(KArgs...), dim3 grid, int block, size_t smem, cudaStream_t st,
                                            Args... args) {
  return launch_cluster_after_predecessor(1, fn, grid, block, smem, st, true, args...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained(bool chained, void (*fn)(KArgs...), dim3 grid, int block, size_t smem, cudaStream_t st,
                                  Args... args) {
  return launch_cluster_after_predecessor(1, fn, grid, block, smem, st, chained, args...);
}

// Zeroes [p0, p0 + n0) and [p1, p1 + n1) (16-byte aligned; lengths are rounded up to 16 bytes).
inline cudaError_t launch_clear(void* p0, size_t n0, void* p1, size_t n1, int sms, cudaStream_t st) {
  ClearRanges r;
  r.ptr[0] = reinterpret_cast<uint4*>(p0);
  r.ptr[1] = reinterpret_cast<uint4*>(p1);
  r.count[0] = (n0 + 15) >> 4;
  r.count[1] = (n1 + 15) >> 4;
  // four 16-byte words per thread, at most eight blocks per SM
  size_t blocks = (std::max(r.count[0], r.count[1]) + 1023) / 1024;
  blocks = std::max<size_t>(1, std::min<size_t>(blocks, (size_t)sms * 8));
  return launch_after_predecessor(clear_ranges, dim3((unsigned)blocks), 256, 0, st, r);
}

// Optional per-stage timing: events recorded on the launch stream around the three stages.
struct StageTimer {
  bool on = false;
  bool have = false;
  cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
  // creates the events on the current device on first use; returns a cudaError_t as int
  int create() {
    for (int i = 0; i < 4; ++i) {
      if (!ev[i]) {
        cudaError_t e = cudaEventCreate(&ev[i]);
        if (e != cudaSuccess) return (int)e;
      }
    }
    return 0;
  }
  void mark(int i, cudaStream_t st) {
    if (on && ev[i]) cudaEventRecord(ev[i], st);
  }
};

// ---------------------------------------------------------------------------------------------
// cuTensorMapEncodeTiled is fetched from the driver at run time, so the library links against
// the CUDA runtime only and still loads on machines without a driver.
// ---------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_tiled_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess) {
      (void)cudaGetLastError();
      return nullptr;
    }
    fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// A tensor map together with the arguments it was built from (re-encoded only when they change).
struct CachedMap {
  CUtensorMap map;
  const void* ptr = nullptr;
  unsigned long long key[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  bool valid = false;
};

// rank <= 3; dims/box in elements (innermost first); 128-byte swizzle; out-of-range reads give zero.
// pitch: elements between rows where they are further apart than dims[0] (0: dense)
inline bool encode_map(CachedMap* cm, CUtensorMapDataType dt, int esize, int rank, const void* ptr,
                       const unsigned long long* dims, const unsigned* box, unsigned long long pitch = 0) {
  if (!pitch) pitch = dims[0];
  unsigned long long key[9] = {(unsigned long long)dt, (unsigned long long)rank, dims[0], dims[1],
                               rank > 2 ? dims[2] : 1ull, box[0], box[1], rank > 2 ? box[2] : 1u, pitch};
  if (cm->valid && cm->ptr == ptr && memcmp(key, cm->key, sizeof(key)) == 0) return true;
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  cuuint64_t gdim[3] = {dims[0], dims[1], rank > 2 ? dims[2] : 1};
  cuuint64_t gstride[2] = {pitch * (cuuint64_t)esize, pitch * dims[1] * (cuuint64_t)esize};
  cuuint32_t bdim[3] = {box[0], box[1], rank > 2 ? box[2] : 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(&cm->map, dt, (cuuint32_t)rank, const_cast<void*>(ptr), gdim, gstride, bdim, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) { cm->valid = false; return false; }
  cm->ptr = ptr;
  memcpy(cm->key, key, sizeof(key));
  cm->valid = true;
  return true;
}

struct TensorMaps {
  CachedMap E, F, K, V, kpvp, Q, W, W2, Wb, aT, aS, O;
  CachedMap dO, abf;                            // backward of the query side
  CachedMap bE, bF, bK, bV, split64, split128, gK, gV, gE, gF;   // backward of the down-projection
  CachedMap A3, Wk, Wv, Xq, Wq, Qp, kpvp2;      // the linear maps of the entry point with un-projected inputs
};

// Per-device context of the tensor-core kernels: the cached tensor maps (their pointers are device
// addresses), the SM count, and whether the kernels' shared-memory limits have been raised there.
struct TensorContext {
  TensorMaps maps;
  int sms = 0;
  // shared-memory limits raised so far (a call that raises them again costs the host as much as a quarter of a launch)
  struct { const void* fn; int bytes; } raised[48] = {};
  cudaError_t raise_smem(const void* fn, int bytes) {
    int i = 0;
    for (; i < 48 && raised[i].fn; ++i)
      if (raised[i].fn == fn) {
        if (raised[i].bytes >= bytes) return cudaSuccess;
        break;
      }
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && i < 48) {
      raised[i].bytes = bytes;
      raised[i].fn = fn;
    }
    return e;
  }
  int sm_total() {
    if (!sms) {
      int dev = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      if (sms <= 0) sms = 148;
    }
    return sms;
  }
  // SMs the persistent kernels may use (the test knob caps it)
  int sm_count();
};

// whether stage 1 may run as pairs of CTAs (tcgen05.mma.cta_group::2) where the shape allows
inline int& stage1_pairs() {
  static int on = 1;
  return on;
}

// 0 = use every SM; otherwise the persistent kernels are launched with at most this many CTAs
inline int& cta_limit() {
  static int limit = 0;
  return limit;
}

inline int TensorContext::sm_count() {
  const int n = sm_total();
  const int lim = cta_limit();
  return (lim > 0 && lim < n) ? lim : n;
}

// ---- E, F with rows on 16-byte boundaries (N no multiple of 8), and dE, dF back ------------------------------
inline int launch_pad_rows(const void* E, const void* F, void* Ep, void* Fp, int rows, int N, int pitch, cudaStream_t st,
                           int* cuda_err) {
  dim3 grid((N + 2047) / 2048, rows < 65535 ? rows : 65535, 2);
  cudaError_t e = launch_after_predecessor(pad_rows, grid, 256, 0, st, (const uint16_t*)E, (const uint16_t*)F,
                                           (uint16_t*)Ep, (uint16_t*)Fp, rows, N, pitch);
  if (e != cudaSuccess) { *cuda_err = (int)e; return -6; }
  return 0;
}
inline int launch_unpad_rows(const void* dEp, const void* dFp, void* dE, void* dF, int rows, int N, int pitch,
                             cudaStream_t st, int* cuda_err) {
  const long long blocks = ((long long)rows * N + 2047) / 2048;
  dim3 grid((unsigned)(blocks < 65535 ? blocks : 65535), 1, 2);
  unpad_rows<<<grid, 256, 0, st>>>((const uint16_t*)dEp, (const uint16_t*)dFp, (uint16_t*)dE, (uint16_t*)dF, rows, N, pitch);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { *cuda_err = (int)e; return -6; }
  return 0;
}

// Sequence splits of stage 1: as few as fill the machine once.  Every split adds a full copy of
// the output to the fp32 reduction (measured: the reduce-add traffic of all CTAs drains at about
// 2.5 TB/s after the last MMA, so more, shorter CTAs lose more in that tail than they gain).
inline int k1_choose_nsplit(int sms, int units, int chunks) {
  int ns = sms / units;
  if (ns < 1) ns = 1;
  if (ns > chunks) ns = chunks;
  return ns;
}

// ---- stage 1: K' = E K, V' = F V into kpvp (already zeroed) ----------------------------------
// H > 0: K, V are [B,N,H,d] (H heads merged into the row); H == 0: [B,H,N,d]
// ef_heads > 0: E, F are [ef_heads][k][N] (one pair per head; head index = bh % ef_heads)
// ef_pitch: elements between the rows of E, F (N, or a multiple of 8 above it)
inline int launch_k1(TensorContext& tc, const void* K, const void* V, const void* E, const void* F, float* kpvp,
                     int BH, int H, int N, int d, int k, int* status, cudaStream_t st, int* cuda_err,
                     int ef_heads, int ef_pitch) {
  TensorMaps& tm = tc.maps;
  const unsigned long long dE[3] = {(unsigned long long)N, (unsigned long long)k,
                                    (unsigned long long)(ef_heads > 0 ? ef_heads : 1)};
  const unsigned bE[3] = {64, 128, 1};
  // [B,N,H,d] is a 3-D tensor too: rows of H*d elements, head h at columns h*d .. h*d+d-1
  const unsigned long long dX[3] = {(unsigned long long)(H > 0 ? H * d : d), (unsigned long long)N,
                                    (unsigned long long)(H > 0 ? BH / H : BH)};
  const unsigned bX[3] = {64, 64, 1};
  const unsigned long long dO[3] = {(unsigned long long)d, (unsigned long long)k, (unsigned long long)2 * BH};
  const unsigned bO[3] = {32, 32, 1};
  if (!encode_map(&tm.E, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 3, E, dE, bE, ef_pitch) ||
      !encode_map(&tm.F, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 3, F, dE, bE, ef_pitch) ||
      !encode_map(&tm.K, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 3, K, dX, bX) ||
      !encode_map(&tm.V, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 3, V, dX, bX) ||
      !encode_map(&tm.kpvp, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, 3, kpvp, dO, bO)) {
    *cuda_err = (int)cudaErrorInvalidValue;
    return -6;
  }
  if (stage1_pairs() && ef_heads == 0 && k % 256 == 0 && (BH * d) % 256 == 0) {
    // two CTAs per output tile: 256 projection rows x 512 columns per pair
    K1PairParams pp;
    pp.N = N; pp.d = d; pp.k = k; pp.BH = BH; pp.H = H;
    pp.col_groups = (BH * d + 511) / 512;
    pp.k_halves = k / 256;
    pp.nsplit = k1_choose_nsplit(tc.sm_count() / 2, 2 * pp.col_groups * pp.k_halves, (N + 63) / 64);
    pp.wait_inputs = ef_pitch != N;
    pp.status = status;
    cudaError_t e = tc.raise_smem((const void*)k1_down_project_pair, kK1PSmemBytes);
    if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
    const int pairs = 2 * pp.k_halves * pp.col_groups * pp.nsplit;
    e = launch_after_predecessor(k1_down_project_pair, 2 * pairs, kK1PThreads, kK1PSmemBytes, st, tm.E.map,
                                             tm.F.map, tm.K.map, tm.V.map, tm.kpvp.map, pp);
    if (e != cudaSuccess) { *cuda_err = (int)e; return -6; }
    return 0;
  }
  K1Params p;
  p.N = N; p.d = d; p.k = k; p.BH = BH; p.H = H;
  p.ef_heads = ef_heads;
  p.group_cols = ef_heads > 0 ? d : 256;
  p.col_groups = (BH * d + p.group_cols - 1) / p.group_cols;
  p.k_halves = (k + 255) / 256;
  p.nsplit = k1_choose_nsplit(tc.sm_count(), 2 * p.col_groups * p.k_halves, (N + 63) / 64);
  p.wait_inputs = ef_pitch != N;
  p.status = status;
  cudaError_t e = tc.raise_smem((const void*)k1_down_project, kK1SmemBytes);
  if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  const int grid = 2 * p.k_halves * p.col_groups * p.nsplit;
  e = launch_after_predecessor(k1_down_project, grid, kK1Threads, kK1SmemBytes, st, tm.E.map, tm.F.map,
                                           tm.K.map, tm.V.map, tm.kpvp.map, p);
  if (e != cudaSuccess) { *cuda_err = (int)e; return -6; }
  return 0;
}

inline int k0_set_attr(TensorContext& tc, int* cuda_err) {
  const cudaError_t e = tc.raise_smem((const void*)k0_linear_map, kK0SmemBytes);
  if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  return 0;
}

// ---- the linear maps on the k contracted rows: K', V' (fp32, [2][B*H][k][d], already zeroed) from
//      kt = stage 1's output for the un-projected inputs ([2][B][dm/64][k][64] fp32)
inline int launch_k0_key_value_maps(TensorContext& tc, const float* kt, __nv_bfloat16* a3, const void* Wk,
                                    const void* Wv, float* kpvp, int B, int H, int dm, int d, int k, int* status,
                                    cudaStream_t st, int* cuda_err) {
  TensorMaps& tm = tc.maps;
  {
    const long long total = (long long)2 * B * k * (dm >> 2);
    int grid = (int)((total + 255) / 256);
    if (grid > tc.sm_total() * 8) grid = tc.sm_total() * 8;
    cudaError_t e = launch_after_predecessor(k0_split_rows, grid, 256, 0, st, kt, a3, 2 * B, k, dm);
    if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  }
  const unsigned long long dA[3] = {(unsigned long long)3 * dm, (unsigned long long)k, (unsigned long long)2 * B};
  const unsigned bA[3] = {64, 128, 1};
  const unsigned long long dB[2] = {(unsigned long long)H * d, (unsigned long long)dm};
  const unsigned bB[2] = {64, 64};
  const unsigned long long dO[3] = {(unsigned long long)d, (unsigned long long)k, (unsigned long long)2 * B * H};
  const unsigned bO[3] = {32, 32, 1};
  if (!encode_map(&tm.A3, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 3, a3, dA, bA) ||
      !encode_map(&tm.Wk, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 2, Wk, dB, bB) ||
      !encode_map(&tm.Wv, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 2, Wv, dB, bB) ||
      !encode_map(&tm.kpvp2, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, 3, kpvp, dO, bO)) {
    *cuda_err = (int)cudaErrorInvalidValue;
    return -6;
  }
  K0Params p;
  p.mode = 0; p.M = k; p.chunks = 3 * dm / 64; p.b_chunks = dm / 64; p.ncols = H * d; p.d = d; p.H = H;
  p.Z = 2 * B; p.zb_shift = B;
  p.row_blocks = (k + 255) / 256;
  p.col_groups = (H * d + 255) / 256;
  const int units = p.row_blocks * p.col_groups * p.Z;
  p.nsplit = k1_choose_nsplit(tc.sm_count(), units, p.chunks);
  p.status = status;
  int rc = k0_set_attr(tc, cuda_err);
  if (rc) return rc;
  cudaError_t e = launch_after_predecessor(k0_linear_map, units * p.nsplit, kK0Threads, kK0SmemBytes, st, tm.A3.map,
                                           tm.Wk.map, tm.Wv.map, tm.kpvp2.map, p);
  if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  return 0;
}

// ---- the query map: Qp [B*N][H*d] bf16 = Xq [B*N][dm] Wq [dm][H*d]
inline int launch_k0_query_map(TensorContext& tc, const void* Xq, const void* Wq, void* Qp, int B, int N, int H, int dm,
                               int d, int* status, cudaStream_t st, int* cuda_err) {
  TensorMaps& tm = tc.maps;
  const unsigned long long dA[3] = {(unsigned long long)dm, (unsigned long long)B * N, 1ull};
  const unsigned bA[3] = {64, 128, 1};
  const unsigned long long dB[2] = {(unsigned long long)H * d, (unsigned long long)dm};
  const unsigned bB[2] = {64, 64};
  const unsigned long long dO[2] = {(unsigned long long)H * d, (unsigned long long)B * N};
  const unsigned bO[2] = {64, 32};
  if (!encode_map(&tm.Xq, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 3, Xq, dA, bA) ||
      !encode_map(&tm.Wq, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 2, Wq, dB, bB) ||
      !encode_map(&tm.Qp, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 2, Qp, dO, bO)) {
    *cuda_err = (int)cudaErrorInvalidValue;
    return -6;
  }
  K0Params p;
  p.mode = 1; p.M = B * N; p.chunks = dm / 64; p.b_chunks = dm / 64; p.ncols = H * d; p.d = d; p.H = H;
  p.Z = 1; p.zb_shift = 1; p.nsplit = 1;
  p.row_blocks = (p.M + 255) / 256;
  p.col_groups = (H * d + 255) / 256;
  p.status = status;
  if (stage1_pairs() && (H * d) % 256 == 0) {
    // as pairs of CTAs: 256 rows x 512 columns per pair
    p.col_groups = (H * d + 511) / 512;
    cudaError_t e = tc.raise_smem((const void*)k0_query_map_pair, kK0PSmemBytes);
    if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
    const int pairs = std::max(1, std::min(tc.sm_count() / 2, p.row_blocks * p.col_groups));
    e = launch_after_predecessor(k0_query_map_pair, 2 * pairs, kK0PThreads, kK0PSmemBytes, st, tm.Xq.map,
                                             tm.Wq.map, tm.Qp.map, p);
    if (e != cudaSuccess) { *cuda_err = (int)e; return -6; }
    return 0;
  }
  int rc = k0_set_attr(tc, cuda_err);
  if (rc) return rc;
  cudaError_t e = launch_after_predecessor(k0_linear_map, p.row_blocks * p.col_groups, kK0Threads, kK0SmemBytes, st,
                                           tm.Xq.map, tm.Wq.map, tm.Wq.map, tm.Qp.map, p);
  if (e != cudaSuccess) { *cuda_err = (int)e; return -6; }
  return 0;
}

// Key splits of stage 2: with few (head, feature tile) pairs the key blocks are divided over up to four
// CTAs per pair, as long as all of them fit on the machine at once.  (A block is not divided: the merge costs
// about what half a block does.)
inline int k2_nsplit(int sms, bool performer, int BH, int d, int k, int p) {
  if (!performer) return 1;
  const int units = BH * ((p + 127) / 128);
  const int chunks = (k * d + kK2BlockElems - 1) / kK2BlockElems;
  int ns = sms / units;
  if (ns > chunks) ns = chunks;
  if (ns > 4) ns = 4;
  return ns < 1 ? 1 : ns;
}

// scratch floats for the partial results of a split stage 2, sized for the largest split the
// problem could get on any device (so the workspace size does not depend on the device)
inline size_t k2_part_floats(bool performer, int BH, int d, int k, int p) {
  if (!performer) return 0;
  int chunks = (k * d + kK2BlockElems - 1) / kK2BlockElems;
  if (chunks > 4) chunks = 4;
  if (chunks < 2) return 0;
  return (size_t)BH * ((p + 127) / 128) * chunks * (size_t)(d + 2) * 128;
}

// ---- stage 2: per-feature summaries a (fp16, transposed) and weights b / z from K', V' --------
// terms: the weights and V' inside as two bf16 terms (for ragged lengths; not PERFORMER with d = 128) or, PERFORMER, as three, and
// then a as three terms too
// chained: W is an input of a call whose chain of launches began before this kernel (it is read before the wait)
inline int launch_k2(TensorContext& tc, bool performer, const float* kpvp, const void* W, float* weight,
                     __half* aT16, float* part, int* counters, int BH, int d, int k, int p, int* status,
                     cudaStream_t st, int* cuda_err, float* a32 = nullptr, __nv_bfloat16* abf = nullptr, int terms = 0,
                     bool chained = true) {
  TensorMaps& tm = tc.maps;
  if (performer) {
    const unsigned long long dW[2] = {(unsigned long long)d, (unsigned long long)p};
    const unsigned bW[2] = {64, 128};
    if (!encode_map(&tm.W2, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 2, W, dW, bW)) {
      *cuda_err = (int)cudaErrorInvalidValue;
      return -6;
    }
  }
  K2Params prm;
  prm.d = d; prm.k = k; prm.p = p; prm.BH = BH;
  prm.ftiles = (p + 127) / 128;
  prm.kpvp = kpvp;
  prm.weight = weight;
  prm.aT16 = aT16;
  prm.a32 = a32;
  prm.abf = abf;
  prm.status = status;
  prm.nsplit = (part && counters) ? k2_nsplit(tc.sm_total(), performer, BH, d, k, p) : 1;
  prm.part = part;
  prm.counters = counters;
  auto fn = terms == 3 ? k2_key_side<true, 64, 3>
            : terms == 2 ? (performer ? k2_key_side<true, 64, 2> : (d == 64 ? k2_key_side<false, 64, 2> : k2_key_side<false, 128, 2>))
                         : (d == 64 ? (performer ? k2_key_side<true, 64> : k2_key_side<false, 64>)
                                    : (performer ? k2_key_side<true, 128> : k2_key_side<false, 128>));
  const int smem = terms == 3 ? K2Smem<3>::bytes : K2Smem<0>::bytes;
  cudaError_t e = tc.raise_smem((const void*)fn, smem);
  if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  // the RNN kernel ignores tmW; pass any valid map
  e = launch_chained(chained, fn, BH * prm.ftiles * prm.nsplit, kK2Threads, smem, st,
                     performer ? tm.W2.map : tm.kpvp.map, prm);
  if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  e = cudaGetLastError();
  if (e != cudaSuccess) { *cuda_err = (int)e; return -6; }
  return 0;
}

// ---- stage 3: O from Q, W and the key-side summaries ------------------------------------------
// abf != NULL (not PERFORMER with d = 128): a as two bf16 terms, [BH][2][p][d], in place of aT16; weights as two terms too
inline int launch_k3(TensorContext& tc, bool performer, const void* Q, const void* W, const __half* aT16,
                     const __nv_bfloat16* abf, const float* weight, void* out, int BH, int H, int N, int d, int p,
                     int* status, cudaStream_t st, int* cuda_err) {
  TensorMaps& tm = tc.maps;
  const unsigned long long dQ[3] = {(unsigned long long)(H > 0 ? H * d : d), (unsigned long long)N,
                                    (unsigned long long)(H > 0 ? BH / H : BH)};
  const unsigned bQ[3] = {64, 128, 1};
  const unsigned long long dA[3] = {(unsigned long long)p, (unsigned long long)d, (unsigned long long)BH};
  const unsigned bA[3] = {64, (unsigned)d, 1};
  const unsigned bO[3] = {64, 32, 1};                 // d = 64: one row-owner warp's slab of the output
  if (d == 64 && !encode_map(&tm.O, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 3, out, dQ, bO)) {
    *cuda_err = (int)cudaErrorInvalidValue;
    return -6;
  }
  const unsigned long long dS[3] = {(unsigned long long)d, (unsigned long long)p, (unsigned long long)BH * 2};
  const unsigned bS[3] = {64, 64, 1};
  if (!encode_map(&tm.Q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 3, Q, dQ, bQ) ||
      !(abf ? encode_map(&tm.aS, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 3, abf, dS, bS)
            : encode_map(&tm.aT, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, 3, aT16, dA, bA))) {
    *cuda_err = (int)cudaErrorInvalidValue;
    return -6;
  }
  if (performer) {
    const unsigned long long dW[2] = {(unsigned long long)d, (unsigned long long)p};
    const unsigned bW[2] = {64, (unsigned)p};
    if (!encode_map(&tm.W, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 2, W, dW, bW)) {
      *cuda_err = (int)cudaErrorInvalidValue;
      return -6;
    }
  }
  K3Params prm;
  prm.N = N; prm.d = d; prm.p = p; prm.BH = BH; prm.H = H;
  prm.tiles_per_head = (N + 127) / 128;
  prm.total_tiles = prm.tiles_per_head * BH;
  prm.weight = weight;
  prm.out = reinterpret_cast<__nv_bfloat16*>(out);
  prm.abf = abf;
  prm.wide = ((uintptr_t)out & 31) == 0;
  prm.status = status;
  // PERFORMER, d = 64: four tiles at a time (64 columns of S and 64 of O each fill TMEM; with d = 128 O alone would)
  const bool units = performer && d == 64;
  const uint32_t smem = units ? k3u_smem_plan(p, abf != nullptr).total : k3_smem_plan(d, p, performer, abf != nullptr).total;
  auto fn = units ? (abf ? k3_query_units<true> : k3_query_units<false>)
                  : (performer ? k3_query_side<true, 128>
                                : (d == 128 ? (abf ? k3_query_side<false, 128, true> : k3_query_side<false, 128>)
                                            : (abf ? k3_query_side<false, 64, true> : k3_query_side<false, 64>)));
  cudaError_t e = tc.raise_smem((const void*)fn, (int)smem);
  if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  int grid = tc.sm_count();
  if (grid > prm.total_tiles) grid = prm.total_tiles;
  // the RNN kernel ignores tmW and only d = 64 stores through tmO; pass any valid map otherwise
  e = launch_after_predecessor(fn, grid, units ? kK3UThreads : k3_threads(d), smem, st, tm.Q.map, performer ? tm.W.map : tm.Q.map,
                               abf ? tm.aS.map : tm.aT.map, d == 64 ? tm.O.map : tm.Q.map, prm);
  if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  e = cudaGetLastError();
  if (e != cudaSuccess) { *cuda_err = (int)e; return -6; }
  return 0;
}

// ---- backward of the query side: dQ, and da, e added to -----------------------------------------
// abf: a as two bf16 terms, [BH][2][p][d], or (PERFORMER with split) three; split: weights as two (RNN with d = 128: always)
inline int bwd_query_a_terms(bool performer, bool split) { return performer && split ? 3 : 2; }
inline int launch_bwd_query(TensorContext& tc, bool performer, bool split, const void* Q, const void* dO, const void* W,
                            const float* weight, const __nv_bfloat16* abf, void* dQ, float* da, float* ei, int BH, int H,
                            int N, int d, int p, int* status, cudaStream_t st, int* cuda_err) {
  TensorMaps& tm = tc.maps;
  const unsigned long long dQd[3] = {(unsigned long long)(H > 0 ? H * d : d), (unsigned long long)N,
                                     (unsigned long long)(H > 0 ? BH / H : BH)};
  const unsigned bQ[3] = {64, 128, 1};
  const unsigned long long dW[2] = {(unsigned long long)d, (unsigned long long)p};
  const unsigned bW[2] = {64, 128};                       // 128 features of a CTA; rows past p read as zero
  const unsigned long long dA[3] = {(unsigned long long)d, (unsigned long long)p,
                                    (unsigned long long)(BH * bwd_query_a_terms(performer, split))};
  const unsigned bA[3] = {64, performer ? 128u : (unsigned)d, 1};
  const CUtensorMapDataType bf = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  if (!encode_map(&tm.Q, bf, 2, 3, Q, dQd, bQ) || !encode_map(&tm.dO, bf, 2, 3, dO, dQd, bQ) ||
      (performer && !encode_map(&tm.W2, bf, 2, 2, W, dW, bW)) || !encode_map(&tm.abf, bf, 2, 3, abf, dA, bA)) {
    *cuda_err = (int)cudaErrorInvalidValue;
    return -6;
  }
  K7Params prm;
  prm.N = N; prm.p = p; prm.BH = BH; prm.H = H;
  prm.tiles_per_head = (N + 127) / 128;
  prm.total_tiles = prm.tiles_per_head * BH;
  prm.weight = weight;
  prm.dQ = reinterpret_cast<__nv_bfloat16*>(dQ);
  prm.wide = ((uintptr_t)dQ & 31) == 0;
  prm.da = da; prm.ei = ei; prm.status = status;
  const int parts = performer ? (p + 127) / 128 : 1;      // 1 or 2 CTAs share a tile
  const int units = std::max(1, std::min(tc.sm_count() / parts, prm.total_tiles));
  cudaError_t e;
  if (!performer) {
    auto fn = d == 128 ? k7_bwd_query_rnn<128, true> : (split ? k7_bwd_query_rnn<64, true> : k7_bwd_query_rnn<64, false>);
    const int smem = d == 128 ? K7Shape<128>::bytes : K7Shape<64>::bytes;
    const int threads = d == 128 ? K7Shape<128>::kThreads : K7Shape<64>::kThreads;
    e = tc.raise_smem((const void*)fn, smem);
    if (e == cudaSuccess) e = launch_after_predecessor(fn, units, threads, smem, st, tm.Q.map, tm.dO.map, tm.abf.map, prm);
  } else {
    auto fn = d == 128 ? (parts == 2 ? k4_bwd_query_wide<2> : k4_bwd_query_wide<1>)
              : split  ? (parts == 2 ? k8_bwd_query_units<2, true> : k8_bwd_query_units<1, true>)
                       : (parts == 2 ? k8_bwd_query_units<2, false> : k8_bwd_query_units<1, false>);
    const int smem = d == 128 ? K4Smem::bytes : (split ? K8Smem<true>::bytes : K8Smem<false>::bytes);
    const int threads = d == 128 ? kK7Threads : (split ? K8Shape<true>::kThreads : K8Shape<false>::kThreads);
    e = tc.raise_smem((const void*)fn, smem);
    if (e == cudaSuccess)
      e = launch_cluster_after_predecessor(parts, fn, units * parts, threads, smem, st, true, tm.Q.map, tm.dO.map, tm.W2.map,
                                           tm.abf.map, prm);
  }
  if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  return 0;
}

// ---- backward of the down-projection: dK, dV, dE, dF from dK', dV' as two bf16 terms ----------------------------
// split: [2][2 terms][k][BH][d] bf16; ef_heads > 0: E, F, dE, dF are [ef_heads][k][N]
// ef_pitch: elements between the rows of E, F, dE, dF.  When it is not N, E, F are padded copies that the last
// product overwrites with dE, dF (dE == E, dF == F), and the caller copies those to their dense form.
template <int kMode, int kN, int kParts = 1>
inline cudaError_t launch_k5_as(TensorContext& tc, const CachedMap& p0, const CachedMap& p1, const CachedMap& s,
                                const CachedMap& o0, const CachedMap& o1, K5Params p, cudaStream_t st) {
  using Sh = K5Shape<kMode, kN>;
  const int rows = kMode == 0 ? p.N : p.k, cols = kMode == 0 ? p.slabs * 64 : p.N;
  p.row_tiles = (rows + 255) / 256;
  p.col_tiles = (cols + kN - 1) / kN;
  p.tiles = 2 * p.groups * p.row_tiles * p.col_tiles;
  auto fn = k5_bwd_projections<kMode, kN, kParts>;
  cudaError_t e = tc.raise_smem((const void*)fn, Sh::kSmemBytes);
  if (e != cudaSuccess) return e;
  const int pairs = kParts == 2 ? p.tiles : std::max(1, std::min(tc.sm_count() / 2, p.tiles));
  return launch_cluster_after_predecessor(2 * kParts, fn, dim3(2 * kParts * pairs), kK5Threads, Sh::kSmemBytes, st, true, p0.map,
                                          p1.map, s.map, o0.map, o1.map, p);
}
inline int launch_k5(TensorContext& tc, const void* E, const void* F, const void* K, const void* V,
                     const __nv_bfloat16* split, void* dK, void* dV, void* dE, void* dF, int BH, int H, int N, int d, int k,
                     int ef_heads, int ef_pitch, int* status, cudaStream_t st, int* cuda_err) {
  TensorMaps& tm = tc.maps;
  const int groups = ef_heads > 0 ? ef_heads : 1;
  K5Params p;
  p.N = N; p.k = k; p.d = d; p.BH = BH; p.H = H; p.status = status;
  p.groups = groups;
  p.slabs = BH / groups * (d >> 6);
  // 256 x 128 tiles where 256 x 256 ones would leave more than a third of the pairs of SMs without one: such a
  // launch is bound by the length of one tile
  const int few = tc.sm_count() / 3;
  const bool narrow0 = 2 * groups * ((N + 255) / 256) * ((p.slabs + 3) / 4) < few;
  const int row_tiles1 = 2 * groups * ((k + 255) / 256);
  // mode 1 with so few tiles that two pairs of CTAs can share each: clusters of four, of which an SM count of 148 holds 32 at
  // once, and enough column blocks that half of them are worth the exchange.  us per launch, one pair per tile / two, k = 256: 128 columns,
  // N = 1024: 16 blocks 11.3 / 12.0, 20 12.1 / 12.2, 24 13.5 / 12.9, 48 22.0 / 17.7, 96 44.2 / 29.9 (N = 2048: 16 12.5 / 13.7, 24 15.0 / 14.8, 96
  // 47 / 33); 256 columns, N = 3000: 32 21.0 / 24.0, 48 28.4 / 29.6, 64 35.4 / 34.4, 96 50 / 45 (N = 4096: 48 29.9 / 30.6, 64 37.2 / 36.1)
  const int at_once = tc.sm_count() * 32 / 148;
  const bool shared128 = row_tiles1 * ((N + 127) / 128) <= at_once && p.slabs >= 24;
  const bool shared256 = !shared128 && row_tiles1 * ((N + 255) / 256) <= at_once && p.slabs >= 64;
  const bool narrow1 = shared128 || (!shared256 && row_tiles1 * ((N + 255) / 256) < few);
  const unsigned long long hd = (unsigned long long)BH * d;
  const unsigned long long dEF[3] = {(unsigned long long)N, (unsigned long long)k, (unsigned long long)groups};
  const unsigned bEF[3] = {64, 64, 1}, bGE[3] = {64, 32, 1};
  const unsigned long long dKV[3] = {(unsigned long long)(H > 0 ? H * d : d), (unsigned long long)N,
                                     (unsigned long long)(H > 0 ? BH / H : BH)};
  const unsigned bKV[3] = {64, narrow1 ? 64u : 128u, 1}, bGK[3] = {64, 32, 1};
  const unsigned long long dS[3] = {hd, (unsigned long long)k, 4};
  const unsigned bS64[3] = {64, 64, 1}, bS128[3] = {64, 128, 1};
  const CUtensorMapDataType bf = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  if (!encode_map(&tm.bE, bf, 2, 3, E, dEF, bEF, ef_pitch) || !encode_map(&tm.bF, bf, 2, 3, F, dEF, bEF, ef_pitch) ||
      !encode_map(&tm.bK, bf, 2, 3, K, dKV, bKV) || !encode_map(&tm.bV, bf, 2, 3, V, dKV, bKV) ||
      !encode_map(&tm.split64, bf, 2, 3, split, dS, bS64) || !encode_map(&tm.split128, bf, 2, 3, split, dS, bS128) ||
      !encode_map(&tm.gK, bf, 2, 3, dK, dKV, bGK) || !encode_map(&tm.gV, bf, 2, 3, dV, dKV, bGK) ||
      !encode_map(&tm.gE, bf, 2, 3, dE, dEF, bGE, ef_pitch) || !encode_map(&tm.gF, bf, 2, 3, dF, dEF, bGE, ef_pitch)) {
    *cuda_err = (int)cudaErrorInvalidValue;
    return -6;
  }
  cudaError_t e = narrow0 ? launch_k5_as<0, 128>(tc, tm.bE, tm.bF, tm.split64, tm.gK, tm.gV, p, st)
                          : launch_k5_as<0, 256>(tc, tm.bE, tm.bF, tm.split64, tm.gK, tm.gV, p, st);
  if (e == cudaSuccess)
    e = shared128   ? launch_k5_as<1, 128, 2>(tc, tm.bK, tm.bV, tm.split128, tm.gE, tm.gF, p, st)
        : shared256 ? launch_k5_as<1, 256, 2>(tc, tm.bK, tm.bV, tm.split128, tm.gE, tm.gF, p, st)
        : narrow1   ? launch_k5_as<1, 128>(tc, tm.bK, tm.bV, tm.split128, tm.gE, tm.gF, p, st)
                    : launch_k5_as<1, 256>(tc, tm.bK, tm.bV, tm.split128, tm.gE, tm.gF, p, st);
  if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  return 0;
}

// ---- backward of the key side (PERFORMER, d = 64): dK', dV' from da, e ----------------------------------
inline int launch_k6(TensorContext& tc, const void* W, const float* kpvp, const float* weight,
                     const float* da, const float* ei, __nv_bfloat16* split, int BH, int k, int p, int* status,
                     cudaStream_t st, int* cuda_err) {
  TensorMaps& tm = tc.maps;
  const unsigned long long dW[2] = {64ull, (unsigned long long)p};
  const unsigned bW[2] = {64, 128};
  if (!encode_map(&tm.W2, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 2, W, dW, bW)) {
    *cuda_err = (int)cudaErrorInvalidValue;
    return -6;
  }
  K6Params prm;
  prm.k = k; prm.p = p; prm.BH = BH;
  prm.kpvp = kpvp; prm.weight = weight; prm.da = da; prm.ei = ei; prm.split = split; prm.status = status;
  cudaError_t e = tc.raise_smem((const void*)k6_bwd_key_side, kK6SmemBytes);
  if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  e = launch_after_predecessor(k6_bwd_key_side, BH * ((k + 127) / 128), kK6Threads, kK6SmemBytes, st, tm.W2.map, prm);
  if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  return 0;
}

// ---- the same with 24 bits
inline int launch_k10(TensorContext& tc, const void* W, const float* kpvp, const float* weight, const float* da,
                      const float* ei, __nv_bfloat16* split, int BH, int d, int k, int p, int* status, cudaStream_t st,
                      int* cuda_err) {
  TensorMaps& tm = tc.maps;
  const unsigned long long dW[2] = {(unsigned long long)d, (unsigned long long)p};
  const unsigned bW[2] = {64, kK10Feats};
  if (!encode_map(&tm.Wb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 2, W, dW, bW)) {
    *cuda_err = (int)cudaErrorInvalidValue;
    return -6;
  }
  K6Params prm;
  prm.k = k; prm.p = p; prm.BH = BH;
  prm.kpvp = kpvp; prm.weight = weight; prm.da = da; prm.ei = ei; prm.split = split; prm.status = status;
  auto fn = d == 128 ? k10_bwd_key_performer<128> : k10_bwd_key_performer<64>;
  const int smem = d == 128 ? K10Shape<128>::bytes : K10Shape<64>::bytes;
  cudaError_t e = tc.raise_smem((const void*)fn, smem);
  if (e == cudaSuccess)
    e = launch_after_predecessor(fn, BH * ((k + 127) / 128), kK10Threads, smem, st, tm.Wb.map, prm);
  if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  return 0;
}

// ---- backward of the key side (RNN): dK', dV' from da, e ------------------------------------------------
inline int launch_k9(TensorContext& tc, const float* kpvp, const float* weight, const float* da, const float* ei,
                     __nv_bfloat16* split, int BH, int d, int k, int* status, cudaStream_t st, int* cuda_err) {
  K9Params prm;
  prm.k = k; prm.BH = BH;
  prm.kpvp = kpvp; prm.weight = weight; prm.da = da; prm.ei = ei; prm.split = split; prm.status = status;
  auto fn = d == 128 ? k9_bwd_key_rnn<128> : k9_bwd_key_rnn<64>;
  const int smem = d == 128 ? K9Shape<128>::bytes : K9Shape<64>::bytes;
  cudaError_t e = tc.raise_smem((const void*)fn, smem);
  if (e == cudaSuccess) e = launch_after_predecessor(fn, BH * ((k + 127) / 128), kK9Threads, smem, st, prm);
  if (e != cudaSuccess) { *cuda_err = (int)e; (void)cudaGetLastError(); return -6; }
  return 0;
}

}  // namespace flurka
