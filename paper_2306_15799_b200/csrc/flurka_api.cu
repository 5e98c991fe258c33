// Host side of the FLuRKA forward library: argument checks, workspace, path selection, launches.
// The C ABI is declared and documented in include/flurka.h.
#include "flurka.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <stdint.h>

#include "simt_backward.cuh"
#include "simt_kernels.cuh"
#include "simt_small.cuh"
#include "tensor_path.cuh"

namespace {

using namespace flurka;

struct Problem {
  int kernel;      // FLURKA_PERFORMER / FLURKA_RNN
  bool fp32;       // element type of the I/O tensors
  bool bnhd;       // Q, K, V, out are [B,N,H,d] (heads merged into the row) instead of [B,H,N,d]
  bool ef_per_head;  // E, F are [H,k,N]: one pair per head, shared over the batch
  int B, H, N, d, k, m;
  int seq_major_heads() const { return bnhd ? H : 0; }   // what head_view() takes
  int ef_heads() const { return ef_per_head ? H : 0; }
  int BH() const { return B * H; }
  int p() const { return kernel == FLURKA_PERFORMER ? m : d; }   // feature dimension
  size_t esize() const { return fp32 ? 4 : 2; }
  size_t qkv_elems() const { return (size_t)B * H * N * d; }
  size_t ef_elems() const { return (size_t)k * N * (ef_per_head ? H : 1); }
  size_t w_elems() const { return kernel == FLURKA_PERFORMER ? (size_t)m * d : 0; }
};

// Workspace layout (all offsets 256-byte aligned):
//   status  int32[4] at offset 0 whatever the problem, then one arrival counter per
//           (head, 128-feature tile) of stage 2
//   kpvp    fp32 [2][BH][k][d]     K' then V'
//           (status and kpvp are adjacent: one range to clear per forward)
//   weight  fp32 [BH][p]           b_i (PERFORMER) or z_i (RNN)
//   a32     fp32 [BH][p][d]        key-side summary, feature-major (ragged lengths on tensor cores: two bf16 terms,
//                                  [BH][2][p][d], in the same bytes)
//   aT16    fp16 [BH][d][p]        the same, transposed, as the tensor-core B operand
//   part    fp32 partial results of a key-split stage 2 (tensor-core path only)
//   efpad   E, F with padded rows (tensor-core path, N no multiple of 8); last, the only part that depends on N
struct Layout {
  size_t status, status_bytes, kpvp, kpvp_end, weight, a32, aT16, part, efpad, total;
};

// Ragged lengths (N no multiple of 8) pay a copy of E, F into rows on 16-byte boundaries (pad_rows.cuh).  With all three stages
// on tensor cores that is a gain over the CUDA-core kernels at every length tried from 257 on (two heads, d = 64, m = 128, us per call:
// k = 64 22 / 27, k = 256 27 / 48); shorter ones were not tried.
constexpr int kRaggedMin = 256;

bool tensor_path_ok(const Problem& pr) {
  if (pr.fp32) return false;
  if (pr.d != 64 && pr.d != 128) return false;
  if (pr.N % 8 && pr.N < kRaggedMin) return false;
  if (pr.k % 64 || pr.k > 512) return false;
  if (pr.kernel == FLURKA_PERFORMER && (pr.m % 64 || pr.m > 256)) return false;
  return true;
}

// Ragged lengths: they came to the tensor cores from the CUDA-core kernels, whose weights, a and V' are
// fp32, while the kernels of the other lengths round weights and a to fp16 (the backward: P, c to bf16).  Stage 1 gives
// fp32 sums of exact products either way.  Stages 2 and 3 have a form with two bf16 terms of everything (16 to 17 bits, fp32's range; error of
// the output against 64 bits as with fp32 weights, 1.649e-3 at B H = 8, N = 3001, k = m = 256, all of it the output's own
// rounding, where fp16 weights give 1.667e-3); PERFORMER with d = 128, where those terms do not fit beside W, runs on CUDA cores.
bool ragged(const Problem& pr) { return pr.N % 8 != 0; }
bool tensor_stages23_ok(const Problem& pr) { return !(ragged(pr) && pr.kernel == FLURKA_PERFORMER && pr.d == 128); }
// Which path a tensor-core shape is said to take: ragged lengths TENSOR_STAGE1 but for PERFORMER with d = 64, whichever
// kernels stages 2 and 3 run on.
int tensor_path_name(const Problem& pr) {
  return !ragged(pr) || (pr.kernel == FLURKA_PERFORMER && pr.d == 64) ? FLURKA_PATH_TENSOR : FLURKA_PATH_TENSOR_STAGE1;
}
// With stages 2 and 3 on CUDA cores, stage 1 on tensor cores (and the copy of E, F) pays from about 2^24 multiply-adds on.
// us per call, stage 1 on tensor cores / on CUDA cores: 10.5 M (BH = 2, N = 643, k = 64, PERFORMER d = 128) 44.6 / 43.5, 12.6 M
// (2, 385, 256, RNN d = 64) 37.5 / 36.2, 16.8 M (16, 257, 64, RNN d = 64) 21.5 / 25.2, 21 M (2, 643, 256, RNN d = 64) 37.8 / 42.6.
double projection_fmas(const Problem& pr) { return (double)pr.BH() * pr.N * pr.k * pr.d; }
int auto_path(const Problem& pr) {
  if (!tensor_path_ok(pr)) return FLURKA_PATH_SIMT;
  if (tensor_path_name(pr) == FLURKA_PATH_TENSOR) return FLURKA_PATH_TENSOR;
  return projection_fmas(pr) >= (double)(1 << 24) ? FLURKA_PATH_TENSOR_STAGE1 : FLURKA_PATH_SIMT;
}

int path_without_copies(const Problem& pr, int path) { return ragged(pr) ? FLURKA_PATH_SIMT : path; }

// Whether a path that the caller forces may take the problem: ragged lengths need a copy of E, F first, which only the
// library's own choice of path makes.
bool forced_tensor_ok(const Problem& pr) { return tensor_path_ok(pr) && !ragged(pr); }

// Elements between the rows of E, F as the tensor-core kernels read them: N, or whole 128-byte lines above it
// where N is ragged and the rows are copied.
int ef_pitch(const Problem& pr) { return ragged(pr) ? (pr.N + 63) & ~63 : pr.N; }
size_t efpad_bytes(const Problem& pr) {
  return ragged(pr) && tensor_path_ok(pr) ? (size_t)2 * pr.k * (pr.ef_per_head ? pr.H : 1) * ef_pitch(pr) * 2 : 0;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// `with_split_scratch`: reserve room for the partial results of a key-split tensor-core stage 2
// (the SIMT path never needs it)
Layout make_layout(const Problem& pr, bool with_split_scratch = true) {
  Layout L;
  size_t off = 0;
  L.status_bytes = 16 + (with_split_scratch ? (size_t)pr.BH() * ((pr.p() + 127) / 128) * 4 : 0);
  L.status = off; off = align256(off + L.status_bytes);
  L.kpvp = off;   L.kpvp_end = off + (size_t)2 * pr.BH() * pr.k * pr.d * 4; off = align256(L.kpvp_end);
  L.weight = off; off = align256(off + (size_t)pr.BH() * pr.p() * 4);
  L.a32 = off;    off = align256(off + (size_t)pr.BH() * pr.p() * pr.d * 4);
  L.aT16 = off;   off = align256(off + (size_t)pr.BH() * pr.p() * pr.d * 2);
  const size_t part_floats = (with_split_scratch && !pr.fp32)
                                 ? k2_part_floats(pr.kernel == FLURKA_PERFORMER, pr.BH(), pr.d, pr.k, pr.p())
                                 : 0;
  L.part = off;   off = align256(off + part_floats * 4);
  L.efpad = off;  off = align256(off + (with_split_scratch ? efpad_bytes(pr) : 0));
  L.total = off;
  return L;
}

// Everything that belongs to one GPU: scratch, staging, streams, events, tensor maps and the record
// of the last forward.  Slot = CUDA device ordinal of the device that is current at the call.
struct DeviceState {
  void* user_ws = nullptr;
  size_t user_ws_bytes = 0;
  void* own_ws = nullptr;
  size_t own_ws_bytes = 0;
  int last_path = 0;
  int last_launches = 0;
  // most recent forward (for flurka_debug_copy / flurka_last_status)
  bool have_last = false;
  bool partial_pending = false;        // the last call was the first half of a sequence-sharded forward
  Problem last_problem{};
  char* last_ws = nullptr;
  // host-buffer entry point: device staging
  void* stage = nullptr;
  size_t stage_bytes = 0;
  cudaStream_t out_stream = nullptr;   // device-to-host copies of finished head groups
  cudaEvent_t group_done[8] = {};      // one per head group of a host-buffer call
  cudaEvent_t out_done = nullptr;
  StageTimer timer;
  TensorContext tc;
};

constexpr int kMaxDevices = 64;
DeviceState g_dev[kMaxDevices];

// Process-wide settings
int g_path = FLURKA_PATH_AUTO;
bool g_stage_timing = false;
int g_last_cuda_error = 0;

// The slot of the current device (slot 0 when there is no usable device: the calls that reach
// this without one only touch host-side fields).
DeviceState& dev_state() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); dev = 0; }
  if (dev < 0 || dev >= kMaxDevices) dev = 0;
  return g_dev[dev];
}

// SMs of the current device
int device_sms() { return dev_state().tc.sm_total(); }

int cuda_fail(cudaError_t e) {
  g_last_cuda_error = (int)e;
  (void)cudaGetLastError();
  return FLURKA_ERR_CUDA;
}

int parse_problem(int variant, int B, int H, int N, int d, int k, int m, Problem* pr) {
  const int kernel = variant & 0xff;
  const int io = variant & 0x100;
  const int layout = variant & 0x200;
  if (kernel != FLURKA_PERFORMER && kernel != FLURKA_RNN) return FLURKA_ERR_VARIANT;
  if (variant & ~0x7ff) return FLURKA_ERR_VARIANT;
  if (B <= 0 || H <= 0 || N <= 0 || d <= 0 || k <= 0) return FLURKA_ERR_SHAPE;
  if (d > 128 || k > 4096) return FLURKA_ERR_SHAPE;
  if (kernel == FLURKA_PERFORMER && m <= 0) return FLURKA_ERR_SHAPE;
  if ((long long)B * H > 65535) return FLURKA_ERR_SHAPE;
  pr->kernel = kernel;
  pr->fp32 = io == FLURKA_IO_FP32;
  pr->bnhd = layout == FLURKA_LAYOUT_BNHD;
  pr->ef_per_head = (variant & FLURKA_EF_PER_HEAD) != 0;
  pr->B = B; pr->H = H; pr->N = N; pr->d = d; pr->k = k;
  pr->m = kernel == FLURKA_PERFORMER ? m : 0;
  return FLURKA_OK;
}

bool overlaps(const void* a, size_t na, const void* b, size_t nb) {
  const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
  return x < y + nb && y < x + na;
}

// The library-owned workspace grows in stream order: the old block is released and the new one
// obtained on the call's stream, so nothing waits on the host and earlier work queued on that
// stream still finds its block.
int get_workspace(DeviceState& ds, size_t need, cudaStream_t st, char** ws) {
  if (ds.user_ws) {
    if (ds.user_ws_bytes < need) return FLURKA_ERR_WORKSPACE;
    *ws = (char*)ds.user_ws;
    return FLURKA_OK;
  }
  if (ds.own_ws_bytes < need) {
    if (ds.own_ws) {
      cudaError_t e = cudaFreeAsync(ds.own_ws, st);
      if (e != cudaSuccess) return cuda_fail(e);
      ds.own_ws = nullptr;
      ds.own_ws_bytes = 0;
      ds.have_last = false;
    }
    cudaError_t e = cudaMallocAsync(&ds.own_ws, need, st);
    if (e != cudaSuccess) { cuda_fail(e); ds.own_ws = nullptr; return FLURKA_ERR_WORKSPACE; }
    ds.own_ws_bytes = need;
  }
  *ws = (char*)ds.own_ws;
  return FLURKA_OK;
}

// Whether the workspace of the next call holds (the library's own: will hold) that much.  A caller's workspace that is large
// enough but for the copies of E, F of a ragged length gets the CUDA-core kernels, which make none: without the copies the
// size does not depend on N, and a workspace may have been sized at another N.
bool workspace_holds(const DeviceState& ds, size_t need) { return !ds.user_ws || ds.user_ws_bytes >= need; }

int check_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); return FLURKA_ERR_DEVICE; }
  if (dev < 0 || dev >= kMaxDevices) return FLURKA_ERR_DEVICE;
  int major = 0;
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return FLURKA_ERR_DEVICE;
  }
  return major == 10 ? FLURKA_OK : FLURKA_ERR_DEVICE;
}

// Copies E, F into `pad` with padded rows where the tensor-core kernels need that, and points *E, *F there.
int pad_projections(const Problem& pr, char* pad, const void** E, const void** F, cudaStream_t st, int* launches) {
  if (!ragged(pr)) return FLURKA_OK;
  const int rows = pr.k * (pr.ef_per_head ? pr.H : 1);
  char* Fp = pad + efpad_bytes(pr) / 2;
  int cuda_err = 0;
  const int rc = launch_pad_rows(*E, *F, pad, Fp, rows, pr.N, ef_pitch(pr), st, &cuda_err);
  if (rc) { g_last_cuda_error = cuda_err; return rc; }
  *E = pad;
  *F = Fp;
  ++*launches;
  return FLURKA_OK;
}

template <typename T, int R, int NB>
cudaError_t launch_simt_down_project_as(const Problem& pr, const void* K, const void* V, const void* E, const void* Fin,
                                 float* kpvp, cudaStream_t st) {
  // enough sequence splits for about four blocks per SM; a split is a multiple of one step
  const int jt = (pr.k + 16 * R - 1) / (16 * R);
  int nsplit = 4 * device_sms() / (jt * pr.BH() * 2);
  const int max_split = (pr.N + kSimtTN - 1) / kSimtTN;
  nsplit = std::max(1, std::min(nsplit, std::min(max_split, 16384)));
  int chunk = (pr.N + nsplit - 1) / nsplit;
  chunk = (chunk + kSimtTN - 1) / kSimtTN * kSimtTN;
  nsplit = (pr.N + chunk - 1) / chunk;
  dim3 grid(jt, pr.BH(), 2 * nsplit);
  return launch_after_predecessor(simt_down_project<T, R, NB>, grid, kSimtThreads, 0, st, (const T*)K, (const T*)V,
                                  (const T*)E, (const T*)Fin, kpvp, pr.BH(), pr.N, pr.d, pr.k, nsplit, chunk,
                                  pr.seq_major_heads(), pr.ef_heads());
}

template <typename T>
int launch_simt_down_project(const Problem& pr, const void* K, const void* V, const void* E,
                             const void* F, float* kpvp, cudaStream_t st, int* launches) {
  // rows per block: the largest tile that k fills (the larger the tile, the fewer shared memory reads per FMA).
  const bool wide = pr.d > 64;
  cudaError_t e;
  // (bf16 with more than 64 columns: 64 rows, two blocks per SM, which hide the conversions and, with N no multiple of 4, the
  // element-wise loads; RNN, 24 heads, k = 1024, the call, us, 64 / 128 rows: N = 4096, d = 128 2284 / 2628, N = 4097, d = 127
  // 2759 / 3490, N = 4097, d = 66 2472 / 3025; fp32 N = 4096, d = 128 1897 / 1813)
  constexpr int kWideRows = sizeof(T) == 2 ? 4 : 8;
  if (pr.k > 64) e = wide ? launch_simt_down_project_as<T, kWideRows, 2>(pr, K, V, E, F, kpvp, st)
                          : launch_simt_down_project_as<T, 8, 1>(pr, K, V, E, F, kpvp, st);
  else if (pr.k > 32) e = wide ? launch_simt_down_project_as<T, 4, 2>(pr, K, V, E, F, kpvp, st)
                               : launch_simt_down_project_as<T, 4, 1>(pr, K, V, E, F, kpvp, st);
  else e = wide ? launch_simt_down_project_as<T, 2, 2>(pr, K, V, E, F, kpvp, st)
                : launch_simt_down_project_as<T, 2, 1>(pr, K, V, E, F, kpvp, st);
  if (e != cudaSuccess) return cuda_fail(e);
  ++*launches;
  return FLURKA_OK;
}

template <typename T, bool P, bool kKeySide, int R, int NB>
int launch_simt_attend_as(const Problem& pr, const void* Q, const void* W, const float* kpvp, float* weight, float* a32,
                          __half* aT16, void* out, cudaStream_t st, bool chained) {
  const size_t smem = simt_attend_smem(R, NB, pr.d);
  auto fn = simt_attend<T, P, kKeySide, R, NB>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e);
  }
  dim3 grid(((kKeySide ? pr.p() : pr.N) + 16 * R - 1) / (16 * R), pr.BH());
  cudaError_t e = launch_chained(chained, fn, grid, kSimtThreads, smem, st, (const T*)Q, (const T*)W, kpvp, weight, a32,
                                 aT16, (T*)out, pr.BH(), pr.N, pr.d, pr.k, pr.p(), pr.seq_major_heads());
  if (e != cudaSuccess) return cuda_fail(e);
  return FLURKA_OK;
}

// chained: everything that the kernel and the query side after it read before they wait (their rows: W, and Q) was complete
// when the call's chain of launches began.  Otherwise it is launched ordinarily and starts when all before it is complete.
template <typename T, bool P, bool kKeySide>
int launch_simt_attend(const Problem& pr, const void* Q, const void* W, const float* kpvp, float* weight, float* a32,
                       __half* aT16, void* out, cudaStream_t st, int* launches, bool chained) {
  // 128 rows per block as soon as that gives every SM a block; 32 below, where the length of one block is the time
  const bool big = (long long)(((kKeySide ? pr.p() : pr.N) + 127) / 128) * pr.BH() >= device_sms();
  ++*launches;
  if (pr.d > 64)
    return big ? launch_simt_attend_as<T, P, kKeySide, 8, 2>(pr, Q, W, kpvp, weight, a32, aT16, out, st, chained)
               : launch_simt_attend_as<T, P, kKeySide, 2, 2>(pr, Q, W, kpvp, weight, a32, aT16, out, st, chained);
  return big ? launch_simt_attend_as<T, P, kKeySide, 8, 1>(pr, Q, W, kpvp, weight, a32, aT16, out, st, chained)
             : launch_simt_attend_as<T, P, kKeySide, 2, 1>(pr, Q, W, kpvp, weight, a32, aT16, out, st, chained);
}

template <typename T, bool P>
int launch_simt_key_side(const Problem& pr, const float* kpvp, const void* W, float* weight, float* a32,
                         __half* aT16, cudaStream_t st, int* launches, bool chained = true) {
  return launch_simt_attend<T, P, true>(pr, nullptr, W, kpvp, weight, a32, aT16, nullptr, st, launches, chained);
}

template <typename T, bool P>
int launch_simt_query_side(const Problem& pr, const void* Q, const void* W, float* weight, float* a32, void* out,
                           cudaStream_t st, int* launches) {
  return launch_simt_attend<T, P, false>(pr, Q, W, nullptr, weight, a32, nullptr, out, st, launches, true);
}

template <typename T>
int key_side_dispatch(const Problem& pr, const float* kpvp, const void* W, float* weight, float* a32,
                      __half* aT16, cudaStream_t st, int* launches, bool chained) {
  return pr.kernel == FLURKA_PERFORMER
             ? launch_simt_key_side<T, true>(pr, kpvp, W, weight, a32, aT16, st, launches, chained)
             : launch_simt_key_side<T, false>(pr, kpvp, W, weight, a32, aT16, st, launches, chained);
}

// The three stages in order.  tc1 / tc3 choose the tensor-core kernel for stage 1 / stage 3
// (bf16 only); tc2 (which needs tc3) does the same for stage 2.  `timer` (may be NULL) gets an
// event before and after each stage.  `keep_status`: the status words are left as they are (a
// later head group of one host-buffer call; they only ever gain bits).
// `stage1(kpvp, status, launches)` fills the (zeroed) K', V' accumulators: the down-projection of
// already projected heads, or the contraction and the linear maps of un-projected inputs.
template <typename T, typename Stage1>
int run_pipeline_with(const Problem& pr, const Layout& L, char* ws, const void* Q, const void* W, void* out,
                      cudaStream_t st, bool tc2, bool tc3, TensorContext* tc, StageTimer* timer, bool keep_status,
                      int* launches, Stage1&& stage1, int phases = 3, void* more = nullptr, size_t more_bytes = 0,
                      bool own_queries = false) {
  // more: one further range of the workspace that has to start at zero
  // own_queries: Q is a result of stage 1, written by a kernel that the last one of stage 1 does not wait for
  // phases: bit 0 = clear the accumulators and run stage 1, bit 1 = run stages 2 and 3 (a sequence-sharded
  // forward does the two halves in separate calls, with the sum over the shards in between)
  float* kpvp = (float*)(ws + L.kpvp);
  float* weight = (float*)(ws + L.weight);
  float* a32 = (float*)(ws + L.a32);
  __half* aT16 = (__half*)(ws + L.aT16);
  int* status = (int*)(ws + L.status);
  const bool performer = pr.kernel == FLURKA_PERFORMER;
  int cuda_err = 0;
  // one range: the status words, the arrival counters and the K', V' accumulators the kernels add into
  const size_t clear_from = L.status + (keep_status ? 16 : 0);
  cudaError_t e = cudaSuccess;
  int rc = FLURKA_OK;
  if (phases & 1) {
    e = launch_clear(ws + clear_from, L.kpvp_end - clear_from, more, more_bytes, device_sms(), st);
    if (e != cudaSuccess) return cuda_fail(e);
    if (timer) timer->mark(0, st);
    rc = stage1(kpvp, status, launches);
    if (rc) return rc;
    if (timer) timer->mark(1, st);
  }
  if (!(phases & 2)) {
    e = cudaGetLastError();
    return e == cudaSuccess ? FLURKA_OK : cuda_fail(e);
  }
  // The kernels of stages 2 and 3 read W and Q before they wait: inputs that were complete before the clearing kernel let
  // the chain begin.  Without that kernel (phases without bit 0), or with Q computed by an ordinary launch in the call, stage
  // 2 starts a chain of its own.
  const bool chained = (phases & 1) && !own_queries;
  // ragged lengths: a as two bf16 terms, which together are as large as the fp32 a they lie in place of
  __nv_bfloat16* abf = tc2 && ragged(pr) ? (__nv_bfloat16*)a32 : nullptr;
  if (tc2) {
    float* part = L.total > L.part ? (float*)(ws + L.part) : nullptr;
    rc = launch_k2(*tc, performer, kpvp, W, weight, abf ? nullptr : aT16, part, status + 4, pr.BH(), pr.d, pr.k, pr.p(), status,
                   st, &cuda_err, nullptr, abf, abf ? 2 : 0, chained);
    if (rc) { g_last_cuda_error = cuda_err; return rc; }
    ++*launches;
  } else {
    rc = key_side_dispatch<T>(pr, kpvp, W, weight, tc3 ? nullptr : a32, tc3 ? aT16 : nullptr, st, launches, chained);
    if (rc) return rc;
  }
  if (timer) timer->mark(2, st);
  if (tc3) {
    rc = launch_k3(*tc, performer, Q, W, aT16, abf, weight, out, pr.BH(), pr.seq_major_heads(), pr.N, pr.d, pr.p(),
                   status, st, &cuda_err);
    if (rc) { g_last_cuda_error = cuda_err; return rc; }
    ++*launches;
  } else {
    rc = performer ? launch_simt_query_side<T, true>(pr, Q, W, weight, a32, out, st, launches)
                   : launch_simt_query_side<T, false>(pr, Q, W, weight, a32, out, st, launches);
    if (rc) return rc;
  }
  if (timer) timer->mark(3, st);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e);
  return FLURKA_OK;
}

template <typename T>
int run_pipeline(const Problem& pr, const Layout& L, char* ws, const void* Q, const void* K, const void* V,
                 const void* E, const void* F, const void* W, void* out, cudaStream_t st, bool tc1, bool tc2,
                 bool tc3, TensorContext* tc, StageTimer* timer, bool keep_status, int* launches, int phases = 3) {
  auto stage1 = [&](float* kpvp, int* status, int* n) -> int {
    if (tc1) {
      int cuda_err = 0;
      const void *Ep = E, *Fp = F;
      int rc = pad_projections(pr, ws + L.efpad, &Ep, &Fp, st, n);
      if (rc) return rc;
      rc = launch_k1(*tc, K, V, Ep, Fp, kpvp, pr.BH(), pr.seq_major_heads(), pr.N, pr.d, pr.k, status, st, &cuda_err,
                     pr.ef_heads(), ef_pitch(pr));
      if (rc) { g_last_cuda_error = cuda_err; return rc; }
      ++*n;
      return FLURKA_OK;
    }
    return launch_simt_down_project<T>(pr, K, V, E, F, kpvp, st, n);
  };
  return run_pipeline_with<T>(pr, L, ws, Q, W, out, st, tc2, tc3, tc, timer, keep_status, launches, stage1, phases);
}

// Whether the one-kernel forward pass takes the problem: everything fits the shared memory of a cluster of eight CTAs per
// head, and a thread has few enough multiply-adds (padding included) that no shape measured is slower than as four launches.
// us per call, one kernel / four launches, on 170 shapes:
//   up to 15 heads (that many clusters of eight run at once with an SM per CTA): 2048 multiply-adds 12.6 / 18.0 (d = 32, k = m =
//   32, N = 256) to 17.5 / 18.0; 2304 14.7 / 18.5 (d = 16, k = m = 64, N = 200); 2432 20.4 / 22.4; 2560 15.0 / 18.4 (d = 32, k = 64,
//   m = 32, N = 128) but also 19.2 / 17.2 (RNN, bf16, d = 64, k = 32, N = 384); 3072 17.5 / 18.3 to 20.8 / 19.8; 3584 19.0 / 17.2;
//   16 heads, RNN, d = k = 48, N = 64 (131 KB of shared memory: one CTA on an SM) 26.7 / 17.3, 15 heads 14.4 / 17.4;
//   16 heads, two CTAs on an SM: 1536 12.7 / 17.7, 1792 16.5 / 18.4, 2048 16.2 / 18.0 to 18.6 / 17.3, 2304 20.3 / 18.2.
constexpr int kSmallHeads = 15;
constexpr long long kSmallFma = 2500, kSmallFmaTwo = 1800;
constexpr size_t kSmallSmem = 200 * 1024, kSmallSmemTwo = 112 * 1024;
bool small_forward_ok(const Problem& pr) {
  if ((long long)pr.BH() * kSmallCtas > device_sms() || pr.d > 64 || pr.k > 1024) return false;
  const SmallShape S = small_shape(pr.N, pr.d, pr.k, pr.p());
  const bool two = pr.BH() > kSmallHeads;
  if (S.total * 4 > (two ? kSmallSmemTwo : kSmallSmem)) return false;
  const long long n = S.n32, f = (S.fpc + 31) & ~31, k32 = (pr.k + 31) & ~31, k64 = (pr.k + 63) & ~63,
                  p64 = (pr.p() + 63) & ~63, per_item = 64 + (pr.kernel == FLURKA_PERFORMER ? pr.d : 0);
  return (2 * n * k32 * 64 + f * k64 * per_item + n * p64 * per_item) / kSmallThreads <= (two ? kSmallFmaTwo : kSmallFma);
}

template <typename T>
int launch_small_forward(const Problem& pr, const Layout& L, char* ws, const void* Q, const void* K, const void* V,
                         const void* E, const void* F, const void* W, void* out, cudaStream_t st, bool keep_status,
                         int* launches) {
  const size_t smem = small_shape(pr.N, pr.d, pr.k, pr.p()).total * 4;
  auto fn = pr.kernel == FLURKA_PERFORMER ? simt_small_forward<T, true> : simt_small_forward<T, false>;
  cudaError_t e = cudaSuccess;
  if (smem > 48 * 1024) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess)
    e = launch_after_predecessor(fn, pr.BH() * kSmallCtas, kSmallThreads, smem, st, (const T*)Q, (const T*)K, (const T*)V,
                                 (const T*)E, (const T*)F, (const T*)W, (float*)(ws + L.kpvp), (float*)(ws + L.weight),
                                 (float*)(ws + L.a32), (int*)(ws + L.status), (T*)out, pr.BH(), pr.N, pr.d, pr.k, pr.p(),
                                 pr.seq_major_heads(), pr.ef_heads(), keep_status ? 1 : 0);
  ++*launches;
  return e == cudaSuccess ? FLURKA_OK : cuda_fail(e);
}

int validate_pointers(const Problem& pr, const void* Q, const void* K, const void* V, const void* E,
                      const void* F, const void* W, const void* out) {
  if (!Q || !K || !V || !E || !F || !out) return FLURKA_ERR_NULL;
  if (pr.kernel == FLURKA_PERFORMER && !W) return FLURKA_ERR_NULL;
  const void* ptrs[7] = {Q, K, V, E, F, W, out};
  for (const void* ptr : ptrs)
    if (ptr && ((uintptr_t)ptr & 15)) return FLURKA_ERR_ALIGN;
  const size_t qb = pr.qkv_elems() * pr.esize(), eb = pr.ef_elems() * pr.esize(),
               wb = pr.w_elems() * pr.esize();
  if (overlaps(out, qb, Q, qb) || overlaps(out, qb, K, qb) || overlaps(out, qb, V, qb) ||
      overlaps(out, qb, E, eb) || overlaps(out, qb, F, eb) || (W && wb && overlaps(out, qb, W, wb)))
    return FLURKA_ERR_OVERLAP;
  return FLURKA_OK;
}

// flurka_forward proper.  `reserve` (>= the problem's own need, or 0) is the workspace size to ask
// for, so that a caller that runs several problems in a row gets one block that fits them all.
int forward_device(const void* Q, const void* K, const void* V, const void* E, const void* F, const void* W,
                   int variant, int B, int H, int N, int d, int k, int m, void* out, void* stream,
                   bool keep_status, size_t reserve, int phases = 3) {
  Problem pr;
  int rc = parse_problem(variant, B, H, N, d, k, m, &pr);
  if (rc) return rc;
  if (phases == 3) {
    rc = validate_pointers(pr, Q, K, V, E, F, W, out);
  } else if (phases == 1) {
    // first half of a sequence-sharded forward: keys, values and projections only
    if (!K || !V || !E || !F) return FLURKA_ERR_NULL;
    for (const void* ptr : {K, V, E, F})
      if ((uintptr_t)ptr & 15) return FLURKA_ERR_ALIGN;
  } else {
    // second half: queries, the random features, the output
    if (!Q || !out || (pr.kernel == FLURKA_PERFORMER && !W)) return FLURKA_ERR_NULL;
    for (const void* ptr : {Q, W, (const void*)out})
      if (ptr && ((uintptr_t)ptr & 15)) return FLURKA_ERR_ALIGN;
    if (overlaps(out, pr.qkv_elems() * pr.esize(), Q, pr.qkv_elems() * pr.esize())) return FLURKA_ERR_OVERLAP;
  }
  if (rc) return rc;
  int path = g_path;
  if (path >= FLURKA_PATH_TENSOR && !forced_tensor_ok(pr)) return FLURKA_ERR_SHAPE;
  if (path == FLURKA_PATH_AUTO) path = auto_path(pr);
  rc = check_device();
  if (rc) return rc;
  DeviceState& ds = dev_state();
  const Layout L = make_layout(pr);
  cudaStream_t st = (cudaStream_t)stream;
  char* ws = nullptr;
  if (phases == 2) {
    // the second half works on what the first half (and the caller's sum over the shards) left in the
    // workspace: same device, same head count and sizes (the slice length may differ)
    const Problem& lp = ds.last_problem;
    if (!ds.have_last || !ds.partial_pending || lp.BH() != pr.BH() || lp.d != pr.d || lp.k != pr.k || lp.m != pr.m ||
        lp.kernel != pr.kernel || lp.fp32 != pr.fp32)
      return FLURKA_ERR_WORKSPACE;
    ws = ds.last_ws;
  } else {
    if (g_path == FLURKA_PATH_AUTO && !workspace_holds(ds, std::max(L.total, reserve))) path = path_without_copies(pr, path);
    rc = get_workspace(ds, std::max(path == FLURKA_PATH_SIMT ? L.efpad : L.total, reserve), st, &ws);
    if (rc) return rc;
  }
  int launches = 0;
  ds.timer.on = g_stage_timing && phases == 3;
  StageTimer* timer = ds.timer.on ? &ds.timer : nullptr;
  if (timer) {
    rc = timer->create();
    if (rc != cudaSuccess) return cuda_fail((cudaError_t)rc);
  }
  if (path == FLURKA_PATH_SIMT && g_path == FLURKA_PATH_AUTO && phases == 3 && !timer &&
      small_forward_ok(pr)) {
    rc = pr.fp32 ? launch_small_forward<float>(pr, L, ws, Q, K, V, E, F, W, out, st, keep_status, &launches)
                 : launch_small_forward<__nv_bfloat16>(pr, L, ws, Q, K, V, E, F, W, out, st, keep_status, &launches);
  } else if (pr.fp32) {
    rc = run_pipeline<float>(pr, L, ws, Q, K, V, E, F, W, out, st, false, false, false, &ds.tc, timer, keep_status,
                             &launches, phases);
  } else {
    const bool tc1 = path == FLURKA_PATH_TENSOR || path == FLURKA_PATH_TENSOR_STAGE1;
    const bool tc2 = path == FLURKA_PATH_TENSOR || path == FLURKA_PATH_TENSOR_STAGE23 ||
                     (path == FLURKA_PATH_TENSOR_STAGE1 && ragged(pr) && tensor_stages23_ok(pr));   // (the library's own choice)
    const bool tc3 = path == FLURKA_PATH_TENSOR || path == FLURKA_PATH_TENSOR_STAGE3 || tc2;
    rc = run_pipeline<__nv_bfloat16>(pr, L, ws, Q, K, V, E, F, W, out, st, tc1, tc2, tc3, &ds.tc, timer,
                                     keep_status, &launches, phases);
  }
  if (rc) return rc;
  ds.partial_pending = phases != 3;       // K', V' of a sharded forward stay in the workspace
  ds.timer.have = ds.timer.on;
  ds.last_path = path;
  ds.last_launches = launches;
  ds.have_last = true;
  ds.last_problem = pr;
  ds.last_ws = ws;
  return FLURKA_OK;
}

}  // namespace

extern "C" {

int flurka_forward(const void* Q, const void* K, const void* V, const void* E, const void* F,
                   const void* W, int variant, int B, int H, int N, int d, int k, int m, void* out,
                   void* stream) {
  return forward_device(Q, K, V, E, F, W, variant, B, H, N, d, k, m, out, stream, /*keep_status=*/false, 0);
}

int flurka_forward_partial(const void* K, const void* V, const void* E, const void* F, int variant, int B, int H,
                           int N, int d, int k, int m, void* stream) {
  return forward_device(nullptr, K, V, E, F, nullptr, variant, B, H, N, d, k, m, nullptr, stream, false, 0, /*phases=*/1);
}

int flurka_forward_finish(const void* Q, const void* W, int variant, int B, int H, int N, int d, int k, int m,
                          void* out, void* stream) {
  return forward_device(Q, nullptr, nullptr, nullptr, nullptr, W, variant, B, H, N, d, k, m, out, stream, false, 0,
                        /*phases=*/2);
}

int flurka_partial_sums(void** dev_ptr, size_t* bytes) {
  if (!dev_ptr || !bytes) return FLURKA_ERR_NULL;
  DeviceState& ds = dev_state();
  if (!ds.have_last || !ds.partial_pending) return FLURKA_ERR_WORKSPACE;
  const Layout L = make_layout(ds.last_problem);
  *dev_ptr = ds.last_ws + L.kpvp;
  *bytes = L.kpvp_end - L.kpvp;
  return FLURKA_OK;
}

int flurka_forward_host(const void* Q, const void* K, const void* V, const void* E, const void* F,
                        const void* W, int variant, int B, int H, int N, int d, int k, int m, void* out,
                        void* stream) {
  Problem pr;
  int rc = parse_problem(variant, B, H, N, d, k, m, &pr);
  if (rc) return rc;
  if (!Q || !K || !V || !E || !F || !out) return FLURKA_ERR_NULL;
  if (pr.kernel == FLURKA_PERFORMER && !W) return FLURKA_ERR_NULL;
  rc = check_device();
  if (rc) return rc;
  DeviceState& ds = dev_state();
  const size_t qb = align256(pr.qkv_elems() * pr.esize());
  const size_t eb = align256(pr.ef_elems() * pr.esize());
  const size_t wb = align256(pr.w_elems() * pr.esize());
  const size_t need = 4 * qb + 2 * eb + wb;
  if (ds.stage_bytes < need) {
    if (ds.stage) {
      cudaError_t e = cudaDeviceSynchronize();
      if (e != cudaSuccess) return cuda_fail(e);
      cudaFree(ds.stage);
      ds.stage = nullptr;
      ds.stage_bytes = 0;
    }
    cudaError_t e = cudaMalloc(&ds.stage, need);
    if (e != cudaSuccess) { cuda_fail(e); return FLURKA_ERR_WORKSPACE; }
    ds.stage_bytes = need;
  }
  char* base = (char*)ds.stage;
  char* dQ = base;
  char* dK = dQ + qb;
  char* dV = dK + qb;
  char* dO = dV + qb;
  char* dE = dO + qb;
  char* dF = dE + eb;
  char* dW = dF + eb;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t qn = pr.qkv_elems() * pr.esize(), en = pr.ef_elems() * pr.esize(),
               wn = pr.w_elems() * pr.esize();
  cudaError_t e;
  if ((e = cudaMemcpyAsync(dE, E, en, cudaMemcpyHostToDevice, st)) != cudaSuccess) return cuda_fail(e);
  if ((e = cudaMemcpyAsync(dF, F, en, cudaMemcpyHostToDevice, st)) != cudaSuccess) return cuda_fail(e);
  if (wn && (e = cudaMemcpyAsync(dW, W, wn, cudaMemcpyHostToDevice, st)) != cudaSuccess)
    return cuda_fail(e);

  // The heads are independent, so the call works through them in up to eight groups: while the
  // inputs of one group travel to the device, the output of the group before travels back on a second
  // stream (the link is full duplex), and the compute of a group hides under the copies.
  // (units that are contiguous in memory: heads for [B,H,N,d], batches for [B,N,H,d]; whole batches
  // also when every head has its own E, F, so that a group's heads keep their numbers)
  const bool by_batch = pr.bnhd || pr.ef_per_head;
  const int heads = by_batch ? pr.B : pr.BH();
  int groups = (int)std::min<size_t>(8, qn >> 20);           // at least 1 MiB of Q per group
  groups = std::max(1, std::min(groups, heads));
  if (groups > 1 && !ds.out_stream) {
    if ((e = cudaStreamCreateWithFlags(&ds.out_stream, cudaStreamNonBlocking)) != cudaSuccess) return cuda_fail(e);
    for (int i = 0; i < 8; ++i)
      if ((e = cudaEventCreateWithFlags(&ds.group_done[i], cudaEventDisableTiming)) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaEventCreateWithFlags(&ds.out_done, cudaEventDisableTiming)) != cudaSuccess) return cuda_fail(e);
  }
  // The groups need not be equal (12 heads in 8 groups: 1, 2, 1, 2, ...).  One workspace that fits the
  // largest group is obtained before the first group runs, so it never moves between groups; the
  // status words sit at its start for every group size.
  size_t reserve = 0, without_copies = 0;
  for (int gi = 0; gi < groups; ++gi) {
    const int cnt = (int)((long long)heads * (gi + 1) / groups) - (int)((long long)heads * gi / groups);
    Problem sub = pr;
    if (by_batch) sub.B = cnt; else { sub.B = 1; sub.H = cnt; }
    const Layout L = make_layout(sub);
    reserve = std::max(reserve, L.total);
    without_copies = std::max(without_copies, L.efpad);
  }
  if (!workspace_holds(ds, reserve)) reserve = without_copies;      // (ragged lengths: see workspace_holds)
  const size_t head_bytes = (size_t)N * d * pr.esize() * (by_batch ? H : 1);
  rc = FLURKA_OK;
  for (int gi = 0; gi < groups && rc == FLURKA_OK; ++gi) {
    const int h0 = (int)((long long)heads * gi / groups), h1 = (int)((long long)heads * (gi + 1) / groups);
    const size_t off = (size_t)h0 * head_bytes, len = (size_t)(h1 - h0) * head_bytes;
    if ((e = cudaMemcpyAsync(dQ + off, (const char*)Q + off, len, cudaMemcpyHostToDevice, st)) != cudaSuccess ||
        (e = cudaMemcpyAsync(dK + off, (const char*)K + off, len, cudaMemcpyHostToDevice, st)) != cudaSuccess ||
        (e = cudaMemcpyAsync(dV + off, (const char*)V + off, len, cudaMemcpyHostToDevice, st)) != cudaSuccess) {
      rc = cuda_fail(e);
      break;
    }
    rc = forward_device(dQ + off, dK + off, dV + off, dE, dF, wn ? dW : nullptr, variant, by_batch ? h1 - h0 : 1,
                        by_batch ? H : h1 - h0, N, d, k, m, dO + off, stream, /*keep_status=*/gi > 0, reserve);
    if (rc) break;
    if (groups == 1) {
      if ((e = cudaMemcpyAsync(out, dO, qn, cudaMemcpyDeviceToHost, st)) != cudaSuccess) rc = cuda_fail(e);
    } else {
      if ((e = cudaEventRecord(ds.group_done[gi], st)) != cudaSuccess ||
          (e = cudaStreamWaitEvent(ds.out_stream, ds.group_done[gi], 0)) != cudaSuccess ||
          (e = cudaMemcpyAsync((char*)out + off, dO + off, len, cudaMemcpyDeviceToHost, ds.out_stream)) != cudaSuccess)
        rc = cuda_fail(e);
    }
  }
  if (groups > 1) {
    // the caller's stream also waits for the copies on the second stream
    if (cudaEventRecord(ds.out_done, ds.out_stream) == cudaSuccess) cudaStreamWaitEvent(st, ds.out_done, 0);
  }
  e = cudaStreamSynchronize(st);
  if (rc) return rc;
  if (e != cudaSuccess) return cuda_fail(e);
  return FLURKA_OK;
}

size_t flurka_workspace_bytes(int variant, int B, int H, int N, int d, int k, int m) {
  Problem pr;
  if (parse_problem(variant, B, H, N, d, k, m, &pr)) return 0;
  return make_layout(pr).total;
}

int flurka_set_workspace(void* dev_ptr, size_t bytes) {
  if (dev_ptr && ((uintptr_t)dev_ptr & 255)) return FLURKA_ERR_ALIGN;
  if (dev_ptr && bytes == 0) return FLURKA_ERR_WORKSPACE;
  DeviceState& ds = dev_state();
  ds.user_ws = dev_ptr;
  ds.user_ws_bytes = dev_ptr ? bytes : 0;
  ds.have_last = false;
  return FLURKA_OK;
}

int flurka_set_path(int path) {
  const int prev = g_path;
  if (path >= FLURKA_PATH_AUTO && path <= FLURKA_PATH_TENSOR_STAGE23) g_path = path;
  return prev;
}

int flurka_set_cta_limit(int max_ctas) {
  const int prev = cta_limit();
  cta_limit() = max_ctas > 0 ? max_ctas : 0;
  return prev;
}

int flurka_set_stage1_pairs(int on) {
  const int prev = stage1_pairs();
  stage1_pairs() = on != 0;
  return prev;
}

int flurka_last_path(void) { return dev_state().last_path; }
int flurka_last_launches(void) { return dev_state().last_launches; }

int flurka_debug_copy(int which, void* dev_dst, size_t bytes, void* stream) {
  if (!dev_dst) return FLURKA_ERR_NULL;
  DeviceState& ds = dev_state();
  if (!ds.have_last) return FLURKA_ERR_WORKSPACE;
  const Problem& pr = ds.last_problem;
  const Layout L = make_layout(pr);
  const size_t kd = (size_t)pr.BH() * pr.k * pr.d * 4;
  size_t off = 0, size = 0;
  switch (which) {
    case 0: off = L.kpvp; size = kd; break;
    case 1: off = L.kpvp + kd; size = kd; break;
    case 2: off = L.a32; size = (size_t)pr.BH() * pr.p() * pr.d * 4; break;
    case 3: off = L.weight; size = (size_t)pr.BH() * pr.p() * 4; break;
    case 4: off = L.status; size = 16; break;
    default: return FLURKA_ERR_VARIANT;
  }
  if (bytes != size) return FLURKA_ERR_SHAPE;
  cudaError_t e = cudaMemcpyAsync(dev_dst, ds.last_ws + off, size, cudaMemcpyDeviceToDevice,
                                  (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e);
  return FLURKA_OK;
}

int flurka_last_status(void) {
  DeviceState& ds = dev_state();
  if (!ds.have_last) return 0;
  const Layout L = make_layout(ds.last_problem);
  int words[4] = {0, 0, 0, 0};
  cudaError_t e = cudaDeviceSynchronize();
  if (e != cudaSuccess) return cuda_fail(e);
  e = cudaMemcpy(words, ds.last_ws + L.status, 16, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e);
  return words[0];
}

int flurka_last_cuda_error(void) { return g_last_cuda_error; }

int flurka_set_stage_timing(int on) {
  g_stage_timing = on != 0;
  for (int i = 0; i < kMaxDevices; ++i) g_dev[i].timer.have = false;
  return FLURKA_OK;
}

int flurka_last_stage_ms(float* ms3) {
  if (!ms3) return FLURKA_ERR_NULL;
  DeviceState& ds = dev_state();
  if (!ds.timer.have) return FLURKA_ERR_WORKSPACE;
  cudaError_t e = cudaEventSynchronize(ds.timer.ev[3]);
  if (e != cudaSuccess) return cuda_fail(e);
  for (int i = 0; i < 3; ++i) {
    e = cudaEventElapsedTime(&ms3[i], ds.timer.ev[i], ds.timer.ev[i + 1]);
    if (e != cudaSuccess) return cuda_fail(e);
  }
  return FLURKA_OK;
}

const char* flurka_strerror(int code) {
  switch (code) {
    case FLURKA_OK: return "ok";
    case FLURKA_ERR_NULL: return "a required pointer is NULL";
    case FLURKA_ERR_VARIANT: return "unknown kernel variant, element type or selector";
    case FLURKA_ERR_SHAPE: return "unsupported shape";
    case FLURKA_ERR_ALIGN: return "pointer not sufficiently aligned";
    case FLURKA_ERR_WORKSPACE: return "workspace missing, too small or not allocatable";
    case FLURKA_ERR_CUDA: return "a CUDA call failed (see flurka_last_cuda_error)";
    case FLURKA_ERR_DEVICE: return "no sm_100 device is current";
    case FLURKA_ERR_OVERLAP: return "out overlaps an input";
    case FLURKA_ERR_TOO_LARGE: return "problem needs more scratch than the built-in array holds";
    default: return "unknown flurka status";
  }
}

int flurka_version(void) { return FLURKA_VERSION; }

}  // extern "C"

namespace {

// Scratch of the entry point with un-projected inputs, after the inner problem's own layout:
//   kt    fp32 E Xk[b], F Xv[b]: tensor path [2][B][dm/64][k][64] (64-wide column blocks), else [2][B][k][dm]
//   a3    bf16 [2B][k][3 dm]: three-term split of kt (tensor path only)
//   qp    Xq W^Q as [B,N,H,d] in the I/O type
struct FusedLayout {
  Layout L;
  size_t kt, kt_bytes, a3, qp, total;
};

FusedLayout make_fused_layout(const Problem& pr, int dm, bool copies = true) {
  FusedLayout f;
  f.L = make_layout(pr);
  size_t off = copies ? f.L.total : f.L.efpad;             // (room for copies of E, F: ragged lengths on tensor cores)
  f.kt_bytes = (size_t)2 * pr.B * pr.k * dm * 4;
  f.kt = off; off = align256(off + f.kt_bytes);
  f.a3 = off; off = align256(off + (pr.fp32 ? 0 : (size_t)2 * pr.B * pr.k * 3 * dm * 2));
  f.qp = off; off = align256(off + pr.qkv_elems() * pr.esize());
  f.total = off;
  return f;
}

bool fused_tensor_ok(const Problem& pr, int dm) { return tensor_path_ok(pr) && dm % 64 == 0 && dm >= 64; }

template <typename T>
int simt_map(const void* A, const void* Bm, void* C, bool a_f32, bool c_f32, int M, int K, int ncols, int Z,
             size_t a_stride, size_t b_stride, int head_d, int z0, cudaStream_t st, int* launches) {
  dim3 grid((ncols + 31) / 32, (M + 31) / 32, Z);
  if (a_f32)
    simt_linear_map<float, T, float><<<grid, 256, 0, st>>>((const float*)A, (const T*)Bm, (float*)C, M, K, ncols,
                                                           a_stride, b_stride, head_d, z0);
  else if (c_f32)
    simt_linear_map<T, T, float><<<grid, 256, 0, st>>>((const T*)A, (const T*)Bm, (float*)C, M, K, ncols, a_stride,
                                                       b_stride, head_d, z0);
  else
    simt_linear_map<T, T, T><<<grid, 256, 0, st>>>((const T*)A, (const T*)Bm, (T*)C, M, K, ncols, a_stride, b_stride,
                                                   head_d, z0);
  ++*launches;
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? FLURKA_OK : cuda_fail(e);
}

template <typename T>
int fused_pipeline(const Problem& pr, int dm, const FusedLayout& FL, char* ws, const void* Xq, const void* Xk,
                   const void* Xv, const void* E, const void* F, const void* Wq, const void* Wk, const void* Wv,
                   const void* W, void* out, cudaStream_t st, bool tensor, TensorContext* tc, StageTimer* timer,
                   int* launches) {
  float* kt = (float*)(ws + FL.kt);
  void* qp = ws + FL.qp;
  auto stage1 = [&](float* kpvp, int* status, int* n) -> int {
    int cuda_err = 0, rc;
    if (tensor) {
      // Q = Xq W^Q first (the long one), then the contraction of the un-projected keys and values as
      // dm/64 pseudo-heads of width 64, then W^K, W^V on the k contracted rows
      rc = launch_k0_query_map(*tc, Xq, Wq, qp, pr.B, pr.N, pr.H, dm, pr.d, status, st, &cuda_err);
      if (rc) { g_last_cuda_error = cuda_err; return rc; }
      const void *Ep = E, *Fp = F;
      rc = pad_projections(pr, ws + FL.L.efpad, &Ep, &Fp, st, n);
      if (rc) return rc;
      rc = launch_k1(*tc, Xk, Xv, Ep, Fp, kt, pr.B * (dm / 64), dm / 64, pr.N, 64, pr.k, status, st, &cuda_err, 0,
                     ef_pitch(pr));
      if (rc) { g_last_cuda_error = cuda_err; return rc; }
      rc = launch_k0_key_value_maps(*tc, kt, (__nv_bfloat16*)(ws + FL.a3), Wk, Wv, kpvp, pr.B, pr.H, dm, pr.d, pr.k,
                                    status, st, &cuda_err);
      if (rc) { g_last_cuda_error = cuda_err; return rc; }
      *n += 4;
      return FLURKA_OK;
    }
    const size_t xb = (size_t)pr.N * dm, ktb = (size_t)pr.k * dm;
    // kt[t][b] = (E | F) X[b];  K', V' = kt W^K, kt W^V (head-split);  Q = Xq W^Q
    if ((rc = simt_map<T>(E, Xk, kt, false, true, pr.k, pr.N, dm, pr.B, 0, xb, 0, 0, st, n))) return rc;
    if ((rc = simt_map<T>(F, Xv, kt + (size_t)pr.B * ktb, false, true, pr.k, pr.N, dm, pr.B, 0, xb, 0, 0, st, n))) return rc;
    if ((rc = simt_map<T>(kt, Wk, kpvp, true, true, pr.k, dm, pr.H * pr.d, pr.B, ktb, 0, pr.d, 0, st, n))) return rc;
    if ((rc = simt_map<T>(kt + (size_t)pr.B * ktb, Wv, kpvp, true, true, pr.k, dm, pr.H * pr.d, pr.B, ktb, 0, pr.d, pr.B,
                          st, n))) return rc;
    return simt_map<T>(Xq, Wq, qp, false, sizeof(T) == 4, pr.B * pr.N, dm, pr.H * pr.d, 1, 0, 0, 0, 0, st, n);
  };
  const bool tensor23 = tensor && tensor_stages23_ok(pr);
  return run_pipeline_with<T>(pr, FL.L, ws, qp, W, out, st, tensor23, tensor23, tc, timer, /*keep_status=*/false, launches,
                              stage1, 3, tensor ? kt : nullptr, tensor ? FL.kt_bytes : 0, /*own_queries=*/!tensor);
}

}  // namespace

extern "C" {

size_t flurka_fused_workspace_bytes(int variant, int B, int H, int N, int dm, int d, int k, int m) {
  Problem pr;
  if (parse_problem(variant | FLURKA_LAYOUT_BNHD, B, H, N, d, k, m, &pr) || dm <= 0) return 0;
  return make_fused_layout(pr, dm).total;
}

int flurka_forward_fused(const void* Xq, const void* Xk, const void* Xv, const void* E, const void* F,
                         const void* Wq, const void* Wk, const void* Wv, const void* W, int variant, int B, int H,
                         int N, int dm, int d, int k, int m, void* out, void* stream) {
  Problem pr;
  // the layout is fixed (out is [B,N,H,d]); the contraction is shared by all heads, so E, F cannot be per head
  if (variant & (FLURKA_LAYOUT_BNHD | FLURKA_EF_PER_HEAD)) return FLURKA_ERR_VARIANT;
  int rc = parse_problem(variant | FLURKA_LAYOUT_BNHD, B, H, N, d, k, m, &pr);
  if (rc) return rc;
  if (dm <= 0 || dm > 16384) return FLURKA_ERR_SHAPE;
  if (!Xq || !Xk || !Xv || !E || !F || !Wq || !Wk || !Wv || !out) return FLURKA_ERR_NULL;
  if (pr.kernel == FLURKA_PERFORMER && !W) return FLURKA_ERR_NULL;
  const void* ptrs[10] = {Xq, Xk, Xv, E, F, Wq, Wk, Wv, W, out};
  for (const void* ptr : ptrs)
    if (ptr && ((uintptr_t)ptr & 15)) return FLURKA_ERR_ALIGN;
  const size_t xb = (size_t)B * N * dm * pr.esize(), ob = pr.qkv_elems() * pr.esize(),
               eb = pr.ef_elems() * pr.esize(), mb = (size_t)dm * H * d * pr.esize(), wb = pr.w_elems() * pr.esize();
  if (overlaps(out, ob, Xq, xb) || overlaps(out, ob, Xk, xb) || overlaps(out, ob, Xv, xb) || overlaps(out, ob, E, eb) ||
      overlaps(out, ob, F, eb) || overlaps(out, ob, Wq, mb) || overlaps(out, ob, Wk, mb) || overlaps(out, ob, Wv, mb) ||
      (W && wb && overlaps(out, ob, W, wb)))
    return FLURKA_ERR_OVERLAP;
  int path = g_path;
  const bool tensor_ok = fused_tensor_ok(pr, dm);
  if (path >= FLURKA_PATH_TENSOR && !(tensor_ok && forced_tensor_ok(pr))) return FLURKA_ERR_SHAPE;
  if (path == FLURKA_PATH_AUTO) path = tensor_ok ? FLURKA_PATH_TENSOR : FLURKA_PATH_SIMT;
  if (path != FLURKA_PATH_TENSOR && path != FLURKA_PATH_SIMT) return FLURKA_ERR_VARIANT;   // no bisecting paths here
  rc = check_device();
  if (rc) return rc;
  DeviceState& ds = dev_state();
  if (g_path == FLURKA_PATH_AUTO && !workspace_holds(ds, make_fused_layout(pr, dm).total)) path = path_without_copies(pr, path);
  const FusedLayout FL = make_fused_layout(pr, dm, /*copies=*/path != FLURKA_PATH_SIMT);
  cudaStream_t st = (cudaStream_t)stream;
  char* ws = nullptr;
  rc = get_workspace(ds, FL.total, st, &ws);
  if (rc) return rc;
  int launches = 0;
  ds.timer.on = g_stage_timing;
  StageTimer* timer = g_stage_timing ? &ds.timer : nullptr;
  if (timer) {
    rc = timer->create();
    if (rc != cudaSuccess) return cuda_fail((cudaError_t)rc);
  }
  if (pr.fp32)
    rc = fused_pipeline<float>(pr, dm, FL, ws, Xq, Xk, Xv, E, F, Wq, Wk, Wv, W, out, st, false, &ds.tc, timer, &launches);
  else
    rc = fused_pipeline<__nv_bfloat16>(pr, dm, FL, ws, Xq, Xk, Xv, E, F, Wq, Wk, Wv, W, out, st,
                                       path == FLURKA_PATH_TENSOR, &ds.tc, timer, &launches);
  if (rc) return rc;
  ds.timer.have = g_stage_timing;
  ds.partial_pending = false;
  ds.last_path = path == FLURKA_PATH_TENSOR ? tensor_path_name(pr) : path;
  ds.last_launches = launches;
  ds.have_last = true;
  ds.last_problem = pr;
  ds.last_ws = ws;
  return FLURKA_OK;
}

}  // extern "C"

namespace {

// Scratch of the backward pass, after the forward layout: da [BH][p][d], e [BH][p] (adjacent: one
// range to clear), then dK', dV' [2][BH][k][d]; all fp32.
struct BackwardLayout {
  Layout L;
  size_t da, dae_bytes, ei, dkpvp, abf, split, efpad, total;
};

// Shapes of which a forced tensor-core path takes the backward (and which report that path): d = 64, and PERFORMER with
// d = 128, at lengths that are multiples of 8.
bool backward_tensor_ok(const Problem& pr) {
  return tensor_path_ok(pr) && !ragged(pr) && (pr.d == 64 || pr.kernel == FLURKA_PERFORMER);
}
// Shapes whose query side has a tensor-core kernel.  Beyond those above: RNN with d = 128 and ragged lengths, whose weights
// are held in 16 to 17 bits (P, c as two bf16 terms); those terms do not fit beside d = 128 and W.
bool backward_query_tensor_ok(const Problem& pr) {
  return tensor_path_ok(pr) && !(ragged(pr) && pr.d == 128 && pr.kernel == FLURKA_PERFORMER);
}

// Whether a ragged backward pass takes the tensor-core kernels for its products with E, F, K, V (and the copies of E, F and of
// dE, dF): from about 2^22 multiply-adds per product on.  us per call, tensor cores / CUDA cores: 2.6 M (one head, N = 643,
// k = 64, PERFORMER d = 64) 76 / 72, 5.3 M (two heads) 76 / 76, 4.2 M (one head, N = 257, k = 256) 97 / 105, RNN 66 / 74,
// 10.5 M (two heads, N = 1283, k = 64) 76 / 82, RNN 49 / 53; 16 heads, N = 257, k = 64: 84 / 123.
bool ragged_backward_pays(const Problem& pr) { return projection_fmas(pr) >= (double)(1 << 22); }

BackwardLayout make_backward_layout(const Problem& pr) {
  BackwardLayout b;
  b.L = make_layout(pr, /*with_split_scratch=*/false);
  size_t off = b.L.total;
  const size_t da_bytes = (size_t)pr.BH() * pr.p() * pr.d * 4;
  b.da = off;
  b.ei = off + da_bytes;
  b.dae_bytes = da_bytes + (size_t)pr.BH() * pr.p() * 4;
  off = align256(off + b.dae_bytes);
  b.dkpvp = off; off = align256(off + (size_t)2 * pr.BH() * pr.k * pr.d * 4);
  b.split = off;
  if (tensor_path_ok(pr)) off = align256(off + (size_t)2 * pr.k * 2 * pr.BH() * pr.d * 2);      // dK', dV' as two bf16 terms
  b.efpad = off;
  off = align256(off + efpad_bytes(pr));
  b.abf = off;
  if (backward_query_tensor_ok(pr))                                       // a as two or three bf16 terms
    off = align256(off + (size_t)bwd_query_a_terms(pr.kernel == FLURKA_PERFORMER, ragged(pr)) * pr.BH() * pr.p() * pr.d * 2);
  b.total = off;
  return b;
}

template <typename T, bool P, int R, int NB, int kD>
int launch_simt_bwd_key_side_at(const Problem& pr, const float* kpvp, const void* W, const float* weight, const float* da,
                                const float* ei, float* dkpvp, __nv_bfloat16* split, cudaStream_t st) {
  const size_t smem = simt_bwd_key_side_smem(R, pr.d);
  auto fn = simt_bwd_key_side<T, P, R, NB, kD>;
  cudaError_t e = cudaSuccess;
  if (smem > 48 * 1024) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess)
    e = launch_after_predecessor(fn, dim3((pr.k + 16 * R - 1) / (16 * R), pr.BH()), kSimtThreads, smem, st, kpvp,
                                 (const T*)W, weight, da, ei, dkpvp, split, pr.BH(), pr.d, pr.k, pr.p());
  return e == cudaSuccess ? FLURKA_OK : cuda_fail(e);
}

template <typename T, bool P, int R, int NB>
int launch_simt_bwd_key_side_as(const Problem& pr, const float* kpvp, const void* W, const float* weight, const float* da,
                                const float* ei, float* dkpvp, __nv_bfloat16* split, cudaStream_t st) {
  return pr.d == 64 * NB ? launch_simt_bwd_key_side_at<T, P, R, NB, 64 * NB>(pr, kpvp, W, weight, da, ei, dkpvp, split, st)
                         : launch_simt_bwd_key_side_at<T, P, R, NB, 0>(pr, kpvp, W, weight, da, ei, dkpvp, split, st);
}

template <typename T, bool P>
int launch_simt_bwd_key_side(const Problem& pr, const float* kpvp, const void* W, const float* weight, const float* da,
                             const float* ei, float* dkpvp, __nv_bfloat16* split, cudaStream_t st) {
  // 64 keys per block where that still gives every SM a block, else 32
  const bool big = (long long)((pr.k + 63) / 64) * pr.BH() >= device_sms();
  if (pr.d > 64) return big ? launch_simt_bwd_key_side_as<T, P, 4, 2>(pr, kpvp, W, weight, da, ei, dkpvp, split, st)
                            : launch_simt_bwd_key_side_as<T, P, 2, 2>(pr, kpvp, W, weight, da, ei, dkpvp, split, st);
  return big ? launch_simt_bwd_key_side_as<T, P, 4, 1>(pr, kpvp, W, weight, da, ei, dkpvp, split, st)
             : launch_simt_bwd_key_side_as<T, P, 2, 1>(pr, kpvp, W, weight, da, ei, dkpvp, split, st);
}

template <typename T, bool P>
int backward_pipeline(const Problem& pr, const BackwardLayout& BL, char* ws, const void* Q, const void* K,
                      const void* V, const void* E, const void* F, const void* W, const void* dO, void* dQ, void* dK,
                      void* dV, void* dE, void* dF, cudaStream_t st, int* launches, TensorContext* tc, bool tcq) {
  // tc != NULL: stage 1 and the gradients that are products with E, F, K, V run on the tensor-core kernels (exact
  // products of bf16 inputs, fp32 sums; dK', dV' as two bf16 terms), and but for ragged lengths the key side's forward
  // half does; tcq: so do the query side and both halves of the key side at any length (but for few
  // keys, below)
  const Layout& L = BL.L;
  float* kpvp = (float*)(ws + L.kpvp);
  float* weight = (float*)(ws + L.weight);
  float* a32 = (float*)(ws + L.a32);
  float* da = (float*)(ws + BL.da);
  float* ei = (float*)(ws + BL.ei);
  float* dkpvp = (float*)(ws + BL.dkpvp);
  const int smh = pr.seq_major_heads(), efh = pr.ef_heads();
  cudaError_t e = launch_clear(ws + L.status, L.kpvp_end - L.status, da, BL.dae_bytes, device_sms(), st);
  if (e != cudaSuccess) return cuda_fail(e);
  // the forward's stages 1 and 2 again: K', V', a_i, b_i (or z_i)
  int rc = FLURKA_OK;
  int cuda_err = 0;
  const void *Ep = E, *Fp = F;           // what the tensor-core kernels read: E, F, or copies with padded rows
  if (tc) {
    rc = pad_projections(pr, ws + BL.efpad, &Ep, &Fp, st, launches);
    if (rc) return rc;
    rc = launch_k1(*tc, K, V, Ep, Fp, kpvp, pr.BH(), smh, pr.N, pr.d, pr.k, (int*)(ws + L.status), st, &cuda_err, efh,
                   ef_pitch(pr));
    if (rc) { g_last_cuda_error = cuda_err; return rc; }
    ++*launches;
  } else {
    rc = launch_simt_down_project<T>(pr, K, V, E, F, kpvp, st, launches);
    if (rc) return rc;
  }
  if (tcq || (tc && !ragged(pr))) {
    // the key side on its tensor-core kernel, with a in fp32 or as two bf16 terms as well.  Split over the keys, its partial
    // results lie where dK', dV' are written later, its arrival counters behind the status words (cleared with them), of which
    // there is room for 60: more (head, feature tile) pairs, up to the half of the SMs, stay undivided.  One CTA per pair / split: the
    // kernel 44 / 31 us at 8 heads, d = 128, k = 512, m = 256; the call 144 / 132.5 at 16 heads of N = 2048.
    const size_t pairs = (size_t)pr.BH() * ((pr.p() + 127) / 128);
    const bool room = k2_part_floats(P, pr.BH(), pr.d, pr.k, pr.p()) * 4 <= BL.efpad - BL.dkpvp &&
                      16 + pairs * 4 <= L.kpvp - L.status;
    rc = launch_k2(*tc, P, kpvp, W, weight, nullptr, room ? (float*)(ws + BL.dkpvp) : nullptr,
                   room ? (int*)(ws + L.status) + 4 : nullptr, pr.BH(), pr.d, pr.k, pr.p(), (int*)(ws + L.status), st,
                   &cuda_err, tcq ? nullptr : a32, tcq ? (__nv_bfloat16*)(ws + BL.abf) : nullptr,
                   ragged(pr) ? bwd_query_a_terms(P, true) : 0);
    if (rc) { g_last_cuda_error = cuda_err; return rc; }
    ++*launches;
  } else {
    rc = launch_simt_key_side<T, P>(pr, kpvp, W, weight, a32, nullptr, st, launches);
    if (rc) return rc;
  }
  if (tcq) {
    const __nv_bfloat16* abf = (const __nv_bfloat16*)(ws + BL.abf);
    rc = launch_bwd_query(*tc, P, ragged(pr), Q, dO, W, weight, abf, dQ, da, ei, pr.BH(), smh, pr.N, pr.d, pr.p(),
                          (int*)(ws + L.status), st, &cuda_err);
    if (rc) { g_last_cuda_error = cuda_err; return rc; }
    ++*launches;
  } else {
    // tiles of 64 rows where they are at least as many as SMs, else of 32
    const bool big = (long long)((pr.N + 63) / 64) * pr.BH() >= device_sms();
    auto fn = pr.d > 64 ? (big ? simt_bwd_query_side<T, P, 4, 2> : simt_bwd_query_side<T, P, 2, 2>)
                        : (big ? simt_bwd_query_side<T, P, 4, 1> : simt_bwd_query_side<T, P, 2, 1>);
    const int rows = big ? 64 : 32;
    const size_t smem = simt_bwd_query_floats(pr.d, rows / 16, P) * 4;
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
      return cuda_fail(e);
    fn<<<dim3((pr.N + rows - 1) / rows, pr.BH()), kSimtThreads, smem, st>>>((const T*)Q, (const T*)W, (const T*)dO, weight, a32,
                                                                           (T*)dQ, da, ei, pr.N, pr.d, pr.p(), smh);
    ++*launches;
  }
  __nv_bfloat16* split = tc ? (__nv_bfloat16*)(ws + BL.split) : nullptr;
  // One block of features (RNN with d = 64, PERFORMER with d = 128 and m = 64) and few keys: the CUDA-core kernel's CTAs of 32 keys are one
  // wave, and its chain is shorter.  (Four of them stand for one of k9's or k10's: with k = 64, half a block of keys, that is half a wave.)
  // us per launch, CUDA cores / k9: 8 heads, k = 512 7.1 / 9.9; two waves, 16 heads, k = 512 10.3 / 9.8; the call with k = 64, N = 376: 32
  // heads 41.5 / 42.7, 64 heads 53.6 / 51.0.  CUDA cores / k10, d = 128: 8 heads, k = 128 15.6 / 22.5, k = 64 15.5 / 16.4; two
  // waves, 16 heads, k = 512 30.6 / 22.6; two blocks, m = 128, 8 heads, k = 64 27.7 / 21.0, k = 256 28.0 / 27.6.  (The RNN with d = 128 has
  // two blocks: 16.6 / 17.7 at 8 heads, k = 256, but 16.4 / 14.1 with k = 64.)  PERFORMER with d = 64 and a ragged length wants its other half
  // on tensor cores too: b_i has the rounding of L as they form it.
  const bool few_keys = pr.d == (P ? 128 : 64) && pr.p() <= 64 && pr.BH() * ((pr.k + 127) / 128) * 4 <= device_sms();
  if (tcq && P && pr.d == 64 && !ragged(pr)) {
    rc = launch_k6(*tc, W, kpvp, weight, da, ei, split, pr.BH(), pr.k, pr.p(), (int*)(ws + L.status), st, &cuda_err);
    if (rc) { g_last_cuda_error = cuda_err; return rc; }
    ++*launches;
  } else if (tcq && P && !few_keys) {
    rc = launch_k10(*tc, W, kpvp, weight, da, ei, split, pr.BH(), pr.d, pr.k, pr.p(), (int*)(ws + L.status), st, &cuda_err);
    if (rc) { g_last_cuda_error = cuda_err; return rc; }
    ++*launches;
  } else if (tcq && !P && !few_keys) {
    rc = launch_k9(*tc, kpvp, weight, da, ei, split, pr.BH(), pr.d, pr.k, (int*)(ws + L.status), st, &cuda_err);
    if (rc) { g_last_cuda_error = cuda_err; return rc; }
    ++*launches;
  } else {
    rc = launch_simt_bwd_key_side<T, P>(pr, kpvp, W, weight, da, ei, dkpvp, split, st);
    if (rc) return rc;
    ++*launches;
  }
  if (tc) {
    const bool padded = Ep != E;
    void *dEp = padded ? (void*)Ep : dE, *dFp = padded ? (void*)Fp : dF;   // the copies are not read again after this
    rc = launch_k5(*tc, Ep, Fp, K, V, split, dK, dV, dEp, dFp, pr.BH(), smh, pr.N, pr.d, pr.k, efh, ef_pitch(pr),
                   (int*)(ws + L.status), st, &cuda_err);
    if (rc) { g_last_cuda_error = cuda_err; return rc; }
    *launches += 2;
    if (padded) {
      rc = launch_unpad_rows(dEp, dFp, dE, dF, pr.k * (efh > 0 ? efh : 1), pr.N, ef_pitch(pr), st, &cuda_err);
      if (rc) { g_last_cuda_error = cuda_err; return rc; }
      ++*launches;
    }
  } else {
    // tiles of 128 rows where they are at least as many as SMs, else of 32
    const int zi = 2 * ((pr.d + 63) / 64), zp = 2 * (efh > 0 ? efh : 1);
    auto blocks = [](int n, int per) { return (n + per - 1) / per; };
    const int sms = device_sms();
    if ((long long)blocks(pr.N, 128) * pr.BH() * zi >= sms)
      simt_bwd_inputs<T, 8><<<dim3(blocks(pr.N, 128), pr.BH(), zi), kSimtThreads, 0, st>>>(
          (const T*)E, (const T*)F, dkpvp, (T*)dK, (T*)dV, pr.BH(), pr.N, pr.d, pr.k, smh, efh);
    else
      simt_bwd_inputs<T, 2><<<dim3(blocks(pr.N, 32), pr.BH(), zi), kSimtThreads, 0, st>>>(
          (const T*)E, (const T*)F, dkpvp, (T*)dK, (T*)dV, pr.BH(), pr.N, pr.d, pr.k, smh, efh);
    ++*launches;
    if ((long long)blocks(pr.N, 64) * blocks(pr.k, 128) * zp >= sms)
      simt_bwd_projections<T, 8><<<dim3(blocks(pr.N, 64), blocks(pr.k, 128), zp), kSimtThreads, 0, st>>>(
          (const T*)K, (const T*)V, dkpvp, (T*)dE, (T*)dF, pr.BH(), pr.N, pr.d, pr.k, smh, efh);
    else
      simt_bwd_projections<T, 2><<<dim3(blocks(pr.N, 64), blocks(pr.k, 32), zp), kSimtThreads, 0, st>>>(
          (const T*)K, (const T*)V, dkpvp, (T*)dE, (T*)dF, pr.BH(), pr.N, pr.d, pr.k, smh, efh);
    ++*launches;
  }
  e = cudaGetLastError();
  return e == cudaSuccess ? FLURKA_OK : cuda_fail(e);
}

}  // namespace

extern "C" {

size_t flurka_backward_workspace_bytes(int variant, int B, int H, int N, int d, int k, int m) {
  Problem pr;
  if (parse_problem(variant, B, H, N, d, k, m, &pr)) return 0;
  return make_backward_layout(pr).total;
}

int flurka_backward(const void* Q, const void* K, const void* V, const void* E, const void* F, const void* W,
                    const void* dO, int variant, int B, int H, int N, int d, int k, int m, void* dQ, void* dK,
                    void* dV, void* dE, void* dF, void* stream) {
  Problem pr;
  int rc = parse_problem(variant, B, H, N, d, k, m, &pr);
  if (rc) return rc;
  if (!Q || !K || !V || !E || !F || !dO || !dQ || !dK || !dV || !dE || !dF) return FLURKA_ERR_NULL;
  if (pr.kernel == FLURKA_PERFORMER && !W) return FLURKA_ERR_NULL;
  const void* ins[7] = {Q, K, V, E, F, W, dO};
  void* outs[5] = {dQ, dK, dV, dE, dF};
  const size_t qb = pr.qkv_elems() * pr.esize(), eb = pr.ef_elems() * pr.esize(), wb = pr.w_elems() * pr.esize();
  const size_t in_bytes[7] = {qb, qb, qb, eb, eb, wb, qb}, out_bytes[5] = {qb, qb, qb, eb, eb};
  for (const void* ptr : ins)
    if (ptr && ((uintptr_t)ptr & 15)) return FLURKA_ERR_ALIGN;
  for (int o = 0; o < 5; ++o) {
    if ((uintptr_t)outs[o] & 15) return FLURKA_ERR_ALIGN;
    for (int i = 0; i < 7; ++i)
      if (ins[i] && in_bytes[i] && overlaps(outs[o], out_bytes[o], ins[i], in_bytes[i])) return FLURKA_ERR_OVERLAP;
    for (int o2 = 0; o2 < o; ++o2)
      if (overlaps(outs[o], out_bytes[o], outs[o2], out_bytes[o2])) return FLURKA_ERR_OVERLAP;
  }
  rc = check_device();
  if (rc) return rc;
  DeviceState& ds = dev_state();
  const BackwardLayout BL = make_backward_layout(pr);
  cudaStream_t st = (cudaStream_t)stream;
  char* ws = nullptr;
  // tensor-core kernels where the shape allows (and the path knob does not force the CUDA-core kernels); a forced tensor
  // path with another shape is refused
  const bool tensor_ok = backward_tensor_ok(pr);
  if (g_path >= FLURKA_PATH_TENSOR && !(tensor_ok && forced_tensor_ok(pr))) return FLURKA_ERR_SHAPE;
  const bool use_tc = tensor_path_ok(pr) && g_path != FLURKA_PATH_SIMT &&
                      (!ragged(pr) || (ragged_backward_pays(pr) && workspace_holds(ds, BL.abf)));
  TensorContext* tc = use_tc ? &ds.tc : nullptr;
  // (a caller's workspace may have been sized without the two terms of a, which the query side on CUDA cores does not need)
  const bool tcq = tc && backward_query_tensor_ok(pr) && (tensor_ok || workspace_holds(ds, BL.total));
  // (a ragged length on CUDA cores: neither copies nor the two-term gradients)
  rc = get_workspace(ds, use_tc ? (tcq ? BL.total : BL.abf) : (ragged(pr) ? BL.split : BL.efpad), st, &ws);
  if (rc) return rc;
  int launches = 0;
  const bool perf = pr.kernel == FLURKA_PERFORMER;
  if (pr.fp32)
    rc = perf ? backward_pipeline<float, true>(pr, BL, ws, Q, K, V, E, F, W, dO, dQ, dK, dV, dE, dF, st, &launches, nullptr, false)
              : backward_pipeline<float, false>(pr, BL, ws, Q, K, V, E, F, W, dO, dQ, dK, dV, dE, dF, st, &launches,
                                                nullptr, false);
  else
    rc = perf ? backward_pipeline<__nv_bfloat16, true>(pr, BL, ws, Q, K, V, E, F, W, dO, dQ, dK, dV, dE, dF, st, &launches, tc, tcq)
              : backward_pipeline<__nv_bfloat16, false>(pr, BL, ws, Q, K, V, E, F, W, dO, dQ, dK, dV, dE, dF, st,
                                                        &launches, tc, tcq);
  if (rc) return rc;
  ds.partial_pending = false;
  ds.timer.have = false;
  // (TENSOR_STAGE1 wherever weights have more than 8 bits, whichever kernels the key and the query side run on)
  ds.last_path = tc && tensor_ok ? FLURKA_PATH_TENSOR : (tc ? FLURKA_PATH_TENSOR_STAGE1 : FLURKA_PATH_SIMT);
  ds.last_launches = launches;
  ds.have_last = true;
  ds.last_problem = pr;
  ds.last_ws = ws;
  return FLURKA_OK;
}

// A loop of nothing but exponentials: eight independent ex2.approx chains per thread, every SM full.
namespace {
__global__ void ex2_rate_kernel(int iters, float* sink) {
  float x[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) x[c] = -0.001f * (float)(threadIdx.x + c + 1);
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int c = 0; c < 8; ++c) asm volatile("ex2.approx.ftz.f32 %0, %0;" : "+f"(x[c]));
  }
  float acc = 0.f;
#pragma unroll
  for (int c = 0; c < 8; ++c) acc += x[c];
  if (acc == -1.f) sink[0] = acc;       // never true (2^x > 0): keeps the chains alive
}
}  // namespace

int flurka_measure_ex2_rate(double* gexp_per_s) {
  if (!gexp_per_s) return FLURKA_ERR_NULL;
  int rc = check_device();
  if (rc) return rc;
  DeviceState& ds = dev_state();
  const int blocks = ds.tc.sm_total() * 8, threads = 256, iters = 4096;
  float* sink = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t e = cudaMalloc(&sink, sizeof(float));
  if (e != cudaSuccess) return cuda_fail(e);
  if ((e = cudaEventCreate(&e0)) != cudaSuccess || (e = cudaEventCreate(&e1)) != cudaSuccess) {
    cudaFree(sink);
    if (e0) cudaEventDestroy(e0);
    return cuda_fail(e);
  }
  float best_ms = 0.f;
  for (int rep = 0; rep < 4; ++rep) {               // the first launch warms up
    cudaEventRecord(e0, 0);
    ex2_rate_kernel<<<blocks, threads>>>(iters, sink);
    cudaEventRecord(e1, 0);
    e = cudaEventSynchronize(e1);
    if (e != cudaSuccess) break;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (rep > 0 && (best_ms == 0.f || ms < best_ms)) best_ms = ms;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(sink);
  if (e != cudaSuccess) return cuda_fail(e);
  if (best_ms <= 0.f) return FLURKA_ERR_CUDA;
  *gexp_per_s = (double)blocks * threads * 8.0 * iters / (best_ms * 1e-3) / 1e9;
  return FLURKA_OK;
}

size_t flurka_static_scratch_need(int variant, int B, int H, int N, int d, int k, int m) {
  Problem pr;
  if (parse_problem(variant, B, H, N, d, k, m, &pr)) return 0;
  return make_layout(pr, /*with_split_scratch=*/false).total;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------
// Forward pass for callers that must not allocate: all scratch lives in a fixed device array that
// is part of the library image.  In host code `g_static_scratch` is only a handle for the symbol,
// never a device address; the address kernels may use comes from cudaGetSymbolAddress, looked up
// once per device with that device current.
// ---------------------------------------------------------------------------------------------
namespace {

static __device__ __align__(256) unsigned char g_static_scratch[FLURKA_STATIC_SCRATCH_BYTES];

char* g_static_scratch_addr[kMaxDevices] = {};

int static_scratch_address(char** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) { (void)cudaGetLastError(); return FLURKA_ERR_DEVICE; }
  if (dev < 0 || dev >= kMaxDevices) return FLURKA_ERR_DEVICE;
  if (!g_static_scratch_addr[dev]) {
    void* ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_static_scratch);
    if (e != cudaSuccess) return cuda_fail(e);
    if (!ptr) return FLURKA_ERR_WORKSPACE;
    g_static_scratch_addr[dev] = (char*)ptr;
  }
  *out = g_static_scratch_addr[dev];
  return FLURKA_OK;
}

}  // namespace

extern "C" int flurka_forward_static_scratch(const void* Q, const void* K, const void* V, const void* E,
                                             const void* F, const void* W, int variant, int B, int H,
                                             int N, int d, int k, int m, void* out, void* stream) {
  Problem pr;
  int rc = parse_problem(variant, B, H, N, d, k, m, &pr);
  if (rc) return rc;
  rc = validate_pointers(pr, Q, K, V, E, F, W, out);
  if (rc) return rc;
  // the CUDA-core kernels' scratch: no partial results of a split key side
  const Layout L = make_layout(pr, /*with_split_scratch=*/false);
  if (L.total > (size_t)FLURKA_STATIC_SCRATCH_BYTES) return FLURKA_ERR_TOO_LARGE;
  rc = check_device();
  if (rc) return rc;
  char* ws = nullptr;
  rc = static_scratch_address(&ws);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  // The array still holds the previous call's contents: the pipeline zeroes the status words and the
  // K', V' accumulators before the kernels add into them.  No stage timing and no record of the call
  // is kept: flurka_last_stage_ms and the other flurka_last_* queries keep describing flurka_forward.
  int launches = 0;
  if (pr.fp32)
    return run_pipeline<float>(pr, L, ws, Q, K, V, E, F, W, out, st, false, false, false, nullptr, nullptr, false,
                               &launches);
  return run_pipeline<__nv_bfloat16>(pr, L, ws, Q, K, V, E, F, W, out, st, false, false, false, nullptr, nullptr,
                                     false, &launches);
}
