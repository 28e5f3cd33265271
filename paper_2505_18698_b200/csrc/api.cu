// C-ABI boundary of libmonarch_attn: argument validation, workspace layout, path selection and
// kernel launches.  No torch types; plain device/host pointers and sizes only.
#include "../../include/monarch_attn.h"
#include "../../include/monarch_attn_test.h"

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "generic_kernels.cuh"
#include "tensor_path.cuh"
#include "tensor_persistent.cuh"
#include "tensor_decoupled.cuh"
#include "fused_small.cuh"
#include "fused_head.cuh"
#include "fused_f32.cuh"
#include "fused_jsplit.cuh"
#include "tile_mma.cuh"
#include "tile_tc.cuh"
#include "host_call.h"
#include "status_word.cuh"
#include "internal_api.h"

namespace ma {

static thread_local int g_last_launches = 0;
static thread_local const char* g_last_kernels = "";     // which set of kernels served the last call (test hook)

static inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
static inline int esize(int dtype) { return dtype == MA_F32 ? 4 : 2; }

struct Problem {
  int batch, heads, N, d, b, T, dtype, m, BH;
  int n_valid;   // keys b k + i >= n_valid are masked out (App. C.3); N when there is no padding
  int H;         // 0: [batch][heads][N][d]; heads: [batch][N][heads][d]
  float* lse;    // optional output [batch*heads][N]: row log-sum-exp of the final L half-step
  const int* seq_len;   // optional DEVICE array [batch]: valid length of every sequence (App. C.3)
  int whole;     // heads whose number chooses between kernels that round differently: BH, or those of the call that this is a part of
};

static int validate_shape(int batch, int heads, int N, int d, int b, int T, int dtype, Problem* p) {
  if (dtype != MA_F32 && dtype != MA_F16 && dtype != MA_BF16) return MA_ERR_DTYPE;
  if (batch <= 0 || heads <= 0 || N <= 0 || d <= 0 || b <= 0 || T < 1) return MA_ERR_SHAPE;
  if (N % b != 0) return MA_ERR_SHAPE;
  if ((long long)batch * heads > 0x7fffffffLL / 2) return MA_ERR_SHAPE;
  *p = Problem{batch, heads, N, d, b, T, dtype, N / b, batch * heads, N, 0, nullptr, nullptr, batch * heads};
  return MA_OK;
}

// ------------------------------------------------------------------ generic path
constexpr size_t kStatusBytes = 256;
constexpr size_t kMaxSmem = 227 * 1024;
constexpr int kSmsB200 = 148;     // (path choice needs no device: the workspace query runs without one)

static bool generic_supported(const Problem& p) {
  if (p.BH > 65535) return false;   // gridDim.y
  size_t r = generic::r_step_smem_floats(p.b, p.d, true) * 4;
  size_t l = generic::l_step_smem_floats(p.m, p.d, false) * 4;
  size_t lf = generic::l_step_smem_floats(p.m, p.d, true) * 4;
  return r <= kMaxSmem && l <= kMaxSmem && lf <= kMaxSmem;
}

struct GenericWs {
  int* status;
  float *aL, *aR, *y, *cL, *cR;
  size_t bytes;
};

static GenericWs generic_layout(const Problem& p, void* base) {
  GenericWs w;
  char* c = (char*)base;
  size_t off = 0;
  size_t big = align_up((size_t)p.BH * p.N * p.d * 4, 256);
  size_t small = align_up((size_t)p.BH * p.N * 4, 256);
  w.status = (int*)(c + off); off += kStatusBytes;
  w.aL = (float*)(c + off); off += big;
  w.aR = (float*)(c + off); off += big;
  w.y = (float*)(c + off); off += big;
  w.cL = (float*)(c + off); off += small;
  w.cR = (float*)(c + off); off += small;
  w.bytes = off;
  return w;
}

// Launch with programmatic stream serialisation (the kernels wait for the launch before them
// themselves: generic::grid_dependency_sync).
template <typename... KArgs, typename... Args>
static cudaError_t launch_serialised(void (*kern)(KArgs...), dim3 grid, int threads, size_t smem,
                                     cudaStream_t st, Args... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
}

template <typename TIn>
static int launch_generic_t(const Problem& p, const TIn* Q, const TIn* K, const TIn* V, TIn* Y,
                            float scale, const GenericWs& w, cudaStream_t st) {
  using namespace generic;
  int launches = 0;
  dim3 gr(p.m, p.BH), gl(p.b, p.BH);
  auto set_smem = [](const void* f, size_t bytes) {
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  if (cudaMemsetAsync(w.status, 0, kStatusBytes, st) != cudaSuccess) return MA_ERR_CUDA;
  for (int t = 1; t <= p.T; ++t) {
    const bool first = (t == 1), last = (t == p.T);
    size_t rs = r_step_smem_floats(p.b, p.d, last) * 4;
#define MA_LAUNCH_R(FIRST, WITHV)                                                              \
  do {                                                                                         \
    if (set_smem((const void*)r_step_kernel<TIn, FIRST, WITHV>, rs) != cudaSuccess)            \
      return MA_ERR_CUDA;                                                                      \
    if (launch_serialised(r_step_kernel<TIn, FIRST, WITHV>, gr, kThreads, rs, st, Q, K, V, w.aR, \
                          w.cR, w.aL, w.cL, w.y, p.N, p.d, p.b, p.m, scale, p.n_valid,          \
                          p.H, p.seq_len, p.heads) != cudaSuccess)                              \
      return MA_ERR_CUDA;                                                                       \
  } while (0)
    if (first && last) MA_LAUNCH_R(true, true);
    else if (first) MA_LAUNCH_R(true, false);
    else if (last) MA_LAUNCH_R(false, true);
    else MA_LAUNCH_R(false, false);
#undef MA_LAUNCH_R
    ++launches;
    size_t ls = l_step_smem_floats(p.m, p.d, last) * 4;
    if (last) {
      if (set_smem((const void*)l_step_kernel<TIn, true>, ls) != cudaSuccess) return MA_ERR_CUDA;
      if (launch_serialised(l_step_kernel<TIn, true>, gl, kThreads, ls, st, Q, w.aL, w.cL, w.y, w.aR, w.cR, Y,
                            p.N, p.d, p.b, p.m, scale, p.H, p.lse, p.seq_len, p.heads) != cudaSuccess)
        return MA_ERR_CUDA;
    } else {
      if (set_smem((const void*)l_step_kernel<TIn, false>, ls) != cudaSuccess) return MA_ERR_CUDA;
      if (launch_serialised(l_step_kernel<TIn, false>, gl, kThreads, ls, st, Q, w.aL, w.cL, w.y, w.aR, w.cR, Y,
                            p.N, p.d, p.b, p.m, scale, p.H, (float*)nullptr, p.seq_len, p.heads) != cudaSuccess)
        return MA_ERR_CUDA;
    }
    ++launches;
  }
  if (cudaGetLastError() != cudaSuccess) return MA_ERR_CUDA;
  g_last_launches = launches;
  g_last_kernels = "generic";
  return MA_OK;
}

static int launch_generic(const Problem& p, const void* Q, const void* K, const void* V, void* Y,
                          float scale, void* ws, cudaStream_t st) {
  GenericWs w = generic_layout(p, ws);
  switch (p.dtype) {
    case MA_F32:
      return launch_generic_t<float>(p, (const float*)Q, (const float*)K, (const float*)V,
                                     (float*)Y, scale, w, st);
    case MA_F16:
      return launch_generic_t<__half>(p, (const __half*)Q, (const __half*)K, (const __half*)V,
                                      (__half*)Y, scale, w, st);
    default:
      return launch_generic_t<__nv_bfloat16>(p, (const __nv_bfloat16*)Q, (const __nv_bfloat16*)K,
                                             (const __nv_bfloat16*)V, (__nv_bfloat16*)Y, scale, w,
                                             st);
  }
}

// ------------------------------------------------------------------ path selection
// fp32 inputs that only the fused fp32 kernel can take: it is not the faster one by ffused::chosen, but a block's K and V
// do not fit the generic kernels (d = 64, 800 rows in one block).
static bool f32_in_one_launch(const Problem& p) {
  return p.dtype == MA_F32 && p.BH <= 65535 && ffused::supported(p.N, p.d, p.b, p.m);
}

// `plain`: the call has no mask and no row_lse output (the kernel split by in-block position
// serves nothing else; the entry point for the other layout selects it itself).
static int resolve_path(const Problem& p, int path, bool plain = true) {
  if (path == MA_PATH_AUTO) {
    // From the third round on, plain 16-bit states are too coarse on peaky logits (they are fed
    // back round after round: about one head in 300 of the N = 256 recipe exceeds 1e-2 at T = 3).
    // The fused per-head kernel and the tcgen05 kernels keep such states; the tile kernels switch to
    // hi + lo pairs from T = 3 on, so they take every 16-bit shape they support then.
    // (short sequences with small blocks: the fused per-head kernel with hi + lo states, one launch)
    if (p.T >= 3 && fsmall::supported_hilo(p.N, p.d, p.b, p.m, p.dtype, p.T)) return MA_PATH_FUSED_SMALL;
    if (p.T >= 3 && tile::supported(p.N, p.d, p.b, p.m, p.dtype, p.BH)) return MA_PATH_TILE_MMA;
    // N = 1024 as 32 x 32: one launch, a head split over four CTAs by in-block position
    if (plain && p.T <= 2 && jsplit::supported(p.N, p.d, p.b, p.m, p.dtype, p.BH)) return MA_PATH_FUSED_JSPLIT;
    // Short sequences with small blocks: one CTA per head, states in shared memory.
    if (p.b <= 16 && p.m <= 16 && fsmall::supported(p.N, p.d, p.b, p.m, p.dtype, p.T))
      return MA_PATH_FUSED_SMALL;
    if (tp::supported(p.N, p.d, p.b, p.m, p.dtype, p.BH)) return MA_PATH_TENSOR;
    // (blocks of more than 32 rows: the tile kernels' two launches are as fast or faster with inputs
    // in HBM, measured; the fused kernel takes them when asked for by name, and for the mask entries)
    if (p.b <= 32 && fsmall::supported(p.N, p.d, p.b, p.m, p.dtype, p.T)) return MA_PATH_FUSED_SMALL;
    if (tile::supported(p.N, p.d, p.b, p.m, p.dtype, p.BH)) return MA_PATH_TILE_MMA;
    // fp32 inputs: short sequences in one launch with the states in shared memory
    if (p.dtype == MA_F32 && p.BH <= 65535 && ffused::chosen(p.N, p.d, p.b, p.m, p.whole, kSmsB200)) return MA_PATH_FUSED_F32;
    if (generic_supported(p)) return MA_PATH_GENERIC;
    return f32_in_one_launch(p) ? MA_PATH_FUSED_F32 : -1;
  }
  if (path == MA_PATH_GENERIC) return generic_supported(p) ? path : -1;
  if (path == MA_PATH_FUSED_F32) {
    if (p.BH <= 65535 && ffused::supported(p.N, p.d, p.b, p.m)) return path;
    // (heads one column wide: a row takes 16 bytes here whatever its width, and from N = 11600 on K leaves no room; the same
    // arithmetic in 2T launches)
    return p.d == 1 && generic_supported(p) ? MA_PATH_GENERIC : -1;
  }
  if (path == MA_PATH_FUSED_JSPLIT)
    return (plain && jsplit::supported(p.N, p.d, p.b, p.m, p.dtype, p.BH)) ? path : -1;
  if (path == MA_PATH_TILE_MMA) return tile::supported(p.N, p.d, p.b, p.m, p.dtype, p.BH) ? path : -1;
  if (path == MA_PATH_FUSED_SMALL)
    return fsmall::supported(p.N, p.d, p.b, p.m, p.dtype, p.T) ? path : -1;
  if (path == MA_PATH_TENSOR) return tp::supported(p.N, p.d, p.b, p.m, p.dtype, p.BH) ? path : -1;
  if (path == MA_PATH_TENSOR_TMEM)
    return (tp::supported(p.N, p.d, p.b, p.m, p.dtype, p.BH) &&
            tp::tmem_kernel_supported(p.b, p.H, p.lse, p.n_valid < p.N ? p.n_valid : 0))
               ? path
               : -1;
  if (path == MA_PATH_TENSOR_BASIC)
    return tensor::supported(p.N, p.d, p.b, p.m, p.dtype, p.BH) ? path : -1;
  return -1;
}

// Path choice of the entry points with a row_lse output or the other layout, which the second-generation tensor kernel,
// the per-head kernels, the tile kernels and the fp32 kernels serve; -1 if none applies.
static int resolve_not_plain(const Problem& p, int path) {
  return path == MA_PATH_TENSOR_TMEM || path == MA_PATH_TENSOR_BASIC ? -1 : resolve_path(p, path, false);
}

static size_t workspace_bytes_for(const Problem& p, int resolved) {
  if (resolved == MA_PATH_GENERIC) return generic_layout(p, nullptr).bytes;
  if (resolved == MA_PATH_FUSED_SMALL || resolved == MA_PATH_FUSED_F32 || resolved == MA_PATH_FUSED_JSPLIT)
    return kStatusBytes;   // no states leave the chip
  if (resolved == MA_PATH_TILE_MMA) return tile::workspace_bytes(p.BH, p.N, p.d, p.b, p.T);
  if (resolved == MA_PATH_TENSOR_BASIC) return tensor::workspace_bytes(p.BH, p.N, p.d, p.b, p.T);
  if (resolved == MA_PATH_TENSOR || resolved == MA_PATH_TENSOR_TMEM)
    return tp::workspace_bytes(p.BH, p.N, p.T, tp::uses_hilo(p.dtype, p.b));
  return 0;
}

// ------------------------------------------------------------------ library-owned buffers
constexpr int kMaxDevices = 64;
struct DeviceBuffers {
  void* ws = nullptr;
  size_t ws_bytes = 0;
  long long armed_key = -1;   // problem whose status block / counters the workspace is armed for
  bool captured = false;   // a graph holds calls that use the workspace: replays write it unseen, and it is never freed
  void* stage = nullptr;   // Q, K, V, Y staging for the host entry point
  size_t stage_bytes = 0;
  // host entry point: kernels and the copy back run on streams of their own, so that the compute
  // and the device-to-host copy of one chunk of heads overlap the host-to-device copies of the
  // next (PCIe is full duplex)
  cudaStream_t compute = nullptr, d2h = nullptr;
  cudaEvent_t chunk_in[8] = {}, chunk_done[8] = {};
  cudaEvent_t all_back = nullptr;
};
constexpr int kHostChunks = 8;
static int g_host_chunks = 0;   // chunks a host call is cut into (<= kHostChunks); 0: by size
static DeviceBuffers g_dev[kMaxDevices];

// `keep`: what there was stays allocated (a graph may still use it).
static int grow(void** ptr, size_t* have, size_t need, bool keep = false) {
  if (*have >= need) return MA_OK;
  if (*ptr) {
    if (!keep) {
      if (cudaDeviceSynchronize() != cudaSuccess) return MA_ERR_CUDA;
      cudaFree(*ptr);
    }
    *ptr = nullptr;
    *have = 0;
  }
  size_t sz = align_up(need, (size_t)1 << 20);
  if (cudaMalloc(ptr, sz) != cudaSuccess) {
    cudaGetLastError();
    *ptr = nullptr;
    return MA_ERR_CUDA;
  }
  *have = sz;
  return MA_OK;
}

// Whether the kernels of a path keep anything in the workspace (beside a caller's status word).
static bool touches_workspace(int resolved) {
  return resolved != MA_PATH_FUSED_SMALL && resolved != MA_PATH_FUSED_F32 && resolved != MA_PATH_FUSED_JSPLIT;
}

// MA_PATH_TILE_MMA has two sets of kernels: tcgen05 tiles (tile_tc.cuh: f16 states, up to two rounds,
// d <= 64) and warp-MMA tiles (tile_mma.cuh: hi + lo states for three or more rounds, wider heads,
// negative scales).  Where both apply, two figures of a call decide:
//   * the tiles that its two half-steps launch on tcgen05, times b + m.  The chain of a tcgen05 tile takes the same time for any block, that of
//     a warp-MMA tile grows with its block (of b rows, then of m), and the first sort needs some tiles to be worth its set-up;
//   * the share of those tiles that rows fill.  They hold whole blocks rounded up to 32, 64 or 128 rows, and what is empty takes the same time;
//     a warp-MMA tile is as wide as its block.
// Both have to be larger where the groups go over a tile before its MMA (bf16 inputs, lengths), above all for one round, which has the least
// other work.  us per call in graphs, warp-MMA / tcgen05 tiles, of some of the 868 sizes measured (3 to 128 rows and blocks, d = 8 to 64, 6 to
// 4000 full tiles, masked and not; the lines depend on neither d nor masks):
//   two rounds   6000: 3 heads of 46 x 50 30.3 / 21.9, 1 of 33 x 128 32.0 / 20.5, 1 of 72 x 62 33.0 / 23.6; below it 1 of 61 x 32 17.5 / 18.6
//                8000: 1 of 66 x 64 35.5 / 23.6, 4 of 40 x 57 33.1 / 24.4, 2 of 57 x 46 23.1 / 23.5; below it 1 of 61 x 62 21.9 / 23.1
//                shares: 0.54 in 34 of 86 x 15 48.4 / 38.4, 0.23 in 1544 of 39 x 5 237 / 267; bf16 0.56 in 42 of 80 x 16 53.9 / 57.9, 0.41 in 182 of
//                10 x 39 55.9 / 62.1; f16 with blocks of more than 64 0.21 in 874 of 4 x 105 444 / 357, 0.17 in 72 of 3 x 120 44.2 / 47.1
//   one round   15000: 2 of 65 x 57 15.1 / 11.8, 1 of 124 x 64 14.1 / 10.5, 14 of 118 x 32 21.0 / 15.1; below it 3 of 61 x 29 8.2 / 10.0
//               16000: 1 of 48 x 128 14.9 / 11.5, 8 of 57 x 64 16.4 / 14.4; below it 4 of 54 x 29 11.0 / 12.1
//               shares: 0.57 in 124 of 126 x 13 66.0 / 56.1, 0.30 in 102 of 38 x 7 14.2 / 17.7; bf16 0.78 in 19 of 102 x 25 24.9 / 19.9, 0.68 in 60 of
//               34 x 32 25.5 / 23.0, 0.69 in 24 of 53 x 20 13.2 / 14.2, 0.57 in 12 of 72 x 37 17.2 / 20.6
// On average the sort that is taken is 0.8 % off the better one; the tcgen05 tiles are taken where they are up to 15 % slower (1 of 87 x 111, masked,
// one round 11.8 / 13.6), the warp-MMA tiles where they are up to 27 % slower (1 of 43 x 128 in bf16, one round 14.8 / 11.7).
static bool tiles_on_tensor_cores(const Problem& p, float scale) {
  if (p.T > 2 || !(scale >= 0.f) || !ttc::supported(p.N, p.d, p.b, p.m, p.dtype, p.BH)) return false;
  auto tiles_of = [](int blocks, int rows) {
    const int per_tile = rows <= 32 ? 4 : (rows <= 64 ? 2 : 1);
    return (blocks + per_tile - 1) / per_tile;
  };
  const long long tiles = (long long)p.whole * (tiles_of(p.m, p.b) + tiles_of(p.b, p.m)), size = tiles * (p.b + p.m);
  const double share = 2. * p.whole * p.N / (128. * tiles);
  const bool prepared = p.dtype != MA_F16 || p.seq_len != nullptr;
  const bool two = p.T == 2;
  if (share < (prepared ? (two ? 0.55 : 0.6) : (two && p.b > 64 ? 0. : 0.4))) return false;
  if (two) return size >= (prepared ? 8000 : 6000);
  if (!prepared) return size >= 15000;
  return size >= (share >= 0.85 ? 16000 : (share >= 0.7 ? 30000 : 90000));
}

// Where a call's waits report to, and the status word it clears first (a caller's workspace; nullptr: none).
struct Status {
  int *report, *clear;
};

static int launch_resolved(const void* Q, const void* K, const void* V, void* Y, const Problem& p,
                           float scale, int resolved, void* ws, const Status& status, cudaStream_t st, bool ws_armed) {
  int rc, launches = 1;
  const char* kernels = "";
  if (resolved == MA_PATH_GENERIC) {
    kernels = "generic";
    rc = launch_generic(p, Q, K, V, Y, scale, ws, st);
    launches = 2 * p.T;
  } else if (resolved == MA_PATH_FUSED_SMALL && scale > 1e-30f && fhead::supported(p.N, p.d, p.b, p.m, p.dtype, p.T) &&
             !fsmall::supported_hilo(p.N, p.d, p.b, p.m, p.dtype, p.T)) {
    // MA_PATH_FUSED_SMALL has two kernels: fused_head.cuh for 9 .. 32 rows and blocks with d <= 64, and the
    // general one (narrower and wider blocks, wider heads, hi + lo states for three or more rounds).
    kernels = "fused_head";
    rc = fhead::launch({Q, K, V, Y, p.BH, p.N, p.d, p.b, p.m, p.T, p.dtype, p.H, p.heads, p.n_valid, scale, p.lse,
                        p.seq_len, status.report, status.clear, tp::knobs().waits()}, st);
  } else if (resolved == MA_PATH_FUSED_SMALL) {
    kernels = "fused_small";
    rc = fsmall::launch(Q, K, V, Y, p.BH, p.N, p.d, p.b, p.m, p.T, p.dtype, scale, p.n_valid, p.H, p.lse, st,
                        p.seq_len, p.heads, status.clear);
  } else if (resolved == MA_PATH_FUSED_F32) {
    kernels = "fused_f32";
    rc = ffused::launch(Q, K, V, Y, p.BH, p.N, p.d, p.b, p.m, p.T, p.dtype, scale, p.n_valid, p.H, p.lse, status.clear, st);
  } else if (resolved == MA_PATH_FUSED_JSPLIT) {
    kernels = "jsplit";
    rc = jsplit::launch(Q, K, V, Y, p.BH, p.T, p.dtype, scale, status.report, status.clear, tp::knobs().waits(), st, p.H);
  } else if (resolved == MA_PATH_TILE_MMA && tiles_on_tensor_cores(p, scale)) {
    kernels = "tile_tc";
    const tile::Ws w = tile::ws_layout(ws, p.BH, p.N, p.d, p.b, false);
    rc = ttc::launch({Q, K, V, Y, p.BH, p.N, p.d, p.b, p.m, p.T, p.dtype, p.H, p.heads, p.n_valid, scale, p.lse, p.seq_len,
                      tp::knobs().waits()},
                     {w.aL, w.aR, w.y, w.cL, status.report, status.clear}, st);
    launches = 2 * p.T;
  } else if (resolved == MA_PATH_TILE_MMA) {
    kernels = "tile_mma";
    tile::Args a{Q, K, V, Y, p.lse, p.BH, p.N, p.d, p.b, p.m, p.T, p.n_valid, p.H, scale, p.seq_len, p.heads, status.clear};
    rc = tile::launch(a, p.dtype, ws, st, &launches);
  } else if (resolved == MA_PATH_TENSOR_BASIC) {
    kernels = "tensor_basic";
    rc = tensor::launch(Q, K, V, Y, p.BH, p.N, p.d, p.b, p.T, p.dtype, scale, ws, status.report, st, &launches);
  } else {
    rc = tp::launch(Q, K, V, Y, p.BH, p.N, p.b, p.T, p.dtype, scale, ws, st, &launches,
                    resolved == MA_PATH_TENSOR_TMEM ? 1 : 0,
                    ws_armed, status.report, &kernels, p.H, p.lse, p.n_valid < p.N ? p.n_valid : 0, p.whole);
  }
  if (rc == MA_OK) {
    g_last_launches = launches;
    g_last_kernels = kernels;
  }
  return rc;
}

static int fwd_ex(const void* Q, const void* K, const void* V, void* Y, const Problem& p,
                  float scale, int resolved, void* ws, size_t ws_bytes, const Status& status, cudaStream_t st,
                  bool ws_armed = false) {
  if (!ws || ws_bytes < workspace_bytes_for(p, resolved)) return MA_ERR_WORKSPACE;
  if (((uintptr_t)ws & 255) != 0) return MA_ERR_ALIGN;
  return launch_resolved(Q, K, V, Y, p, scale, resolved, ws, status, st, ws_armed);
}

static int check_ptrs(const void* Q, const void* K, const void* V, void* Y, const Problem& p) {
  if (!Q || !K || !V || !Y) return MA_ERR_NULL;
  if ((((uintptr_t)Q | (uintptr_t)K | (uintptr_t)V | (uintptr_t)Y) & 15) != 0) return MA_ERR_ALIGN;
  size_t bytes = (size_t)p.BH * p.N * p.d * esize(p.dtype);
  const char* y0 = (const char*)Y;
  const void* in[3] = {Q, K, V};
  for (int i = 0; i < 3; ++i) {
    const char* a = (const char*)in[i];
    if (y0 < a + bytes && a < y0 + bytes) return MA_ERR_ALIGN;
  }
  return MA_OK;
}

// Which kernels serve a call; -1 if none.
static int resolve_call(const Call& c, const Problem& p) {
  switch (c.entry) {
    case Entry::kFwd: return resolve_path(p, MA_PATH_AUTO);
    case Entry::kEx: return resolve_path(p, c.path);
    case Entry::kObjective: return resolve_not_plain(p, c.path);
    case Entry::kBshd:
      // (the kernel split by in-block position takes this layout too: a head is a column offset of
      // its tensor maps)
      if (((c.path == MA_PATH_AUTO && p.T <= 2) || c.path == MA_PATH_FUSED_JSPLIT) &&
          jsplit::supported(p.N, p.d, p.b, p.m, p.dtype, p.BH))
        return MA_PATH_FUSED_JSPLIT;
      return resolve_not_plain(p, c.path);
    case Entry::kPadded:
    case Entry::kVarlen: break;
  }
  // The mask entries.  Short 16-bit sequences (up to two rounds, or where the hi + lo instantiation
  // applies): the fused per-head kernel (one launch).  `padded` then has the second-generation
  // tensor kernel where a tile row owns a whole key block (b = 64, 128: the mask touches the last
  // block's tiles only).  Other 16-bit shapes: the tile kernels (hi + lo states from the
  // third round on); else the fp32 kernels.
  if ((p.T <= 2 && fsmall::supported(p.N, p.d, p.b, p.m, p.dtype, p.T)) ||
      fsmall::supported_hilo(p.N, p.d, p.b, p.m, p.dtype, p.T))
    return MA_PATH_FUSED_SMALL;
  if (c.entry == Entry::kPadded && resolve_path(p, MA_PATH_AUTO, false) == MA_PATH_TENSOR && p.b != 32)
    return MA_PATH_TENSOR;
  if (tile::supported(p.N, p.d, p.b, p.m, p.dtype, p.BH)) return MA_PATH_TILE_MMA;
  if (c.entry == Entry::kPadded && p.dtype == MA_F32 && p.BH <= 65535 && ffused::chosen(p.N, p.d, p.b, p.m, p.BH, kSmsB200))
    return MA_PATH_FUSED_F32;
  if (generic_supported(p)) return MA_PATH_GENERIC;
  return c.entry == Entry::kPadded && f32_in_one_launch(p) ? MA_PATH_FUSED_F32 : -1;
}

static int run_call(const Call& c) {
  Problem p;
  int rc = validate_shape(c.batch, c.heads, c.N, c.d, c.b, c.T, c.dtype, &p);
  if (rc != MA_OK) return rc;
  if (c.whole > 0) p.whole = c.whole;
  // less than one block of padding: every key block keeps at least one valid key
  if (c.entry == Entry::kPadded && (c.n_valid > c.N || c.n_valid <= c.N - c.b)) return MA_ERR_SHAPE;
  rc = check_ptrs(c.Q, c.K, c.V, c.Y, p);
  if (rc != MA_OK) return rc;
  if (c.entry == Entry::kVarlen) {
    if (!c.seq_len) return MA_ERR_NULL;
    if (((uintptr_t)c.seq_len & 3) != 0) return MA_ERR_ALIGN;
  }
  if (c.entry == Entry::kObjective) {
    if (!c.lse) return MA_ERR_NULL;
    if (((uintptr_t)c.lse & 3) != 0) return MA_ERR_ALIGN;
  }
  if (c.entry != Entry::kFwd && (!(c.scale == c.scale) || isinf(c.scale))) return MA_ERR_SHAPE;
  const int r = resolve_call(c, p);
  if (r < 0) return MA_ERR_UNSUPPORTED;
  cudaStream_t st = (cudaStream_t)c.stream;
  if (c.entry == Entry::kPadded) p.n_valid = c.n_valid;
  if (c.entry == Entry::kVarlen) p.seq_len = c.seq_len;
  if (c.entry == Entry::kObjective) p.lse = c.lse;
  if (c.entry == Entry::kBshd) p.H = c.heads;
  if (c.entry != Entry::kFwd && (c.ws || !c.alloc))
    return fwd_ex(c.Q, c.K, c.V, c.Y, p, c.scale, r, c.ws, c.ws_bytes, Status{(int*)c.ws, (int*)c.ws}, st);
  const Status status{status_word(), nullptr};
  if (!status.report) return MA_ERR_CUDA;
  if (c.entry != Entry::kFwd) {
    // the fused kernels touch no scratch: nothing is allocated for them
    if (!touches_workspace(r)) return launch_resolved(c.Q, c.K, c.V, c.Y, p, c.scale, r, nullptr, status, st, false);
    const size_t bytes = workspace_bytes_for(p, r);
    void* ws = c.alloc(c.ctx, bytes);
    return ws ? fwd_ex(c.Q, c.K, c.V, c.Y, p, c.scale, r, ws, bytes, status, st) : MA_ERR_CUDA;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return MA_ERR_CUDA;
  DeviceBuffers& B = g_dev[dev];
  const size_t had = B.ws_bytes;
  rc = grow(&B.ws, &B.ws_bytes, workspace_bytes_for(p, r), B.captured);
  if (rc != MA_OK) return rc;
  if (touches_workspace(r) && !B.captured) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &capture) != cudaSuccess) return MA_ERR_CUDA;
    B.captured = capture != cudaStreamCaptureStatusNone;
  }
  // The persistent kernel leaves its status block and counters zeroed, so the library's own
  // workspace is cleared only when the problem (hence the layout) changes; or each time, once a graph may write it in between.
  const long long key = ((long long)r << 56) ^ ((long long)p.T << 48) ^ ((long long)p.BH << 24) ^ p.N;
  const bool armed = (r == MA_PATH_TENSOR) && !B.captured && had == B.ws_bytes && B.armed_key == key;
  rc = fwd_ex(c.Q, c.K, c.V, c.Y, p, 1.0f / sqrtf((float)c.d), r, B.ws, B.ws_bytes, status, st, armed);
  B.armed_key = (rc == MA_OK && r == MA_PATH_TENSOR) ? key : -1;
  return rc;
}

// The pinned host range that `host` lies in; false for pageable and for managed memory.
static bool pinned_range(const void* host, hostcall::Pinned* r) {
  typedef CUresult (*Fn)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);
  static Fn fn = nullptr;
  if (!fn) {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &f, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return false;
    fn = (Fn)f;
  }
  unsigned long long type = 0, address = 0, managed = 0, start = 0, size = 0;
  CUpointer_attribute what[5] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                 CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                 CU_POINTER_ATTRIBUTE_RANGE_SIZE};
  void* to[5] = {&type, &address, &managed, &start, &size};
  if (fn(5, what, to, (CUdeviceptr)host) != CUDA_SUCCESS || type != CU_MEMORYTYPE_HOST || managed != 0) return false;
  *r = hostcall::Pinned{(size_t)address, (size_t)start, (size_t)size};
  return true;
}

// Stream operations of a host call (host_call.h).
struct HostOps {
  DeviceBuffers& B;
  cudaStream_t caller, compute, back;
  int N, d, b, T, dtype, heads;
  int launches;
  static int status(cudaError_t e) { return e == cudaSuccess ? MA_OK : MA_ERR_CUDA; }
  static int order(cudaStream_t later, cudaStream_t earlier, cudaEvent_t ev) {
    const int rc = status(cudaEventRecord(ev, earlier));
    return rc != MA_OK ? rc : status(cudaStreamWaitEvent(later, ev, 0));
  }
  int h2d(void* dst, const void* src, size_t n) { return status(cudaMemcpyAsync(dst, src, n, cudaMemcpyHostToDevice, caller)); }
  int d2h(void* dst, const void* src, size_t n) { return status(cudaMemcpyAsync(dst, src, n, cudaMemcpyDeviceToHost, back)); }
  int fork(int c) { return order(compute, caller, B.chunk_in[c]); }
  int after(int c) { return order(back, compute, B.chunk_done[c]); }
  int join_compute() { return order(caller, compute, B.all_back); }
  int join_back() { return order(caller, back, B.all_back); }
  int forward(const void* Q, const void* K, const void* V, void* Y, int units) {
    const int rc = run_call(Call{Entry::kFwd, Q, K, V, Y, 1, units, N, d, b, T, dtype, 0.f, MA_PATH_AUTO, 0, nullptr, nullptr,
                                 nullptr, 0, compute, nullptr, nullptr, heads});
    launches += rc == MA_OK ? g_last_launches : 0;
    return rc;
  }
};

}  // namespace ma

using namespace ma;

extern "C" {

size_t monarch_attn_workspace_bytes(int batch, int heads, int N, int d, int b, int T, int dtype,
                                    int path) {
  Problem p;
  if (validate_shape(batch, heads, N, d, b, T, dtype, &p) != MA_OK) return 0;
  int r = resolve_path(p, path);
  if (r < 0) return 0;
  return workspace_bytes_for(p, r);
}

int monarch_attn_internal_run(const Call* c) { return run_call(*c); }

int monarch_attn_fwd_ex(const void* Q, const void* K, const void* V, void* Y, int batch, int heads,
                        int N, int d, int b, int T, int dtype, float softmax_scale, int path,
                        void* workspace, size_t workspace_bytes, void* stream) {
  return run_call(Call{Entry::kEx, Q, K, V, Y, batch, heads, N, d, b, T, dtype, softmax_scale, path, 0, nullptr,
                       nullptr, workspace, workspace_bytes, stream, nullptr, nullptr, 0});
}

int monarch_attn_fwd_padded(const void* Q, const void* K, const void* V, void* Y, int batch,
                            int heads, int N, int d, int b, int T, int dtype, float softmax_scale,
                            int n_valid, void* workspace, size_t workspace_bytes, void* stream) {
  return run_call(Call{Entry::kPadded, Q, K, V, Y, batch, heads, N, d, b, T, dtype, softmax_scale, MA_PATH_AUTO,
                       n_valid, nullptr, nullptr, workspace, workspace_bytes, stream, nullptr, nullptr, 0});
}

int monarch_attn_fwd_varlen(const void* Q, const void* K, const void* V, void* Y, int batch,
                            int heads, int N, int d, int b, int T, int dtype, float softmax_scale,
                            const int* seq_len, void* workspace, size_t workspace_bytes,
                            void* stream) {
  return run_call(Call{Entry::kVarlen, Q, K, V, Y, batch, heads, N, d, b, T, dtype, softmax_scale, MA_PATH_AUTO, 0,
                       seq_len, nullptr, workspace, workspace_bytes, stream, nullptr, nullptr, 0});
}

int monarch_attn_fwd_objective(const void* Q, const void* K, const void* V, void* Y, int batch,
                               int heads, int N, int d, int b, int T, int dtype,
                               float softmax_scale, int path, float* row_lse, void* workspace,
                               size_t workspace_bytes, void* stream) {
  return run_call(Call{Entry::kObjective, Q, K, V, Y, batch, heads, N, d, b, T, dtype, softmax_scale, path, 0,
                       nullptr, row_lse, workspace, workspace_bytes, stream, nullptr, nullptr, 0});
}

int monarch_attn_fwd_bshd(const void* Q, const void* K, const void* V, void* Y, int batch, int N,
                          int heads, int d, int b, int T, int dtype, float softmax_scale, int path,
                          void* workspace, size_t workspace_bytes, void* stream) {
  return run_call(Call{Entry::kBshd, Q, K, V, Y, batch, heads, N, d, b, T, dtype, softmax_scale, path, 0, nullptr,
                       nullptr, workspace, workspace_bytes, stream, nullptr, nullptr, 0});
}

int monarch_attn_fwd(const void* Q, const void* K, const void* V, void* Y, int batch, int heads,
                     int N, int d, int b, int T, int dtype, void* stream) {
  return run_call(Call{Entry::kFwd, Q, K, V, Y, batch, heads, N, d, b, T, dtype, 0.f, MA_PATH_AUTO, 0, nullptr,
                       nullptr, nullptr, 0, stream, nullptr, nullptr, 0});
}

int monarch_attn_fwd_host(const void* Qh, const void* Kh, const void* Vh, void* Yh, int batch,
                          int heads, int N, int d, int b, int T, int dtype, void* stream) {
  Problem p;
  int rc = validate_shape(batch, heads, N, d, b, T, dtype, &p);
  if (rc != MA_OK) return rc;
  if (!Qh || !Kh || !Vh || !Yh) return MA_ERR_NULL;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return MA_ERR_CUDA;
  DeviceBuffers& B = g_dev[dev];
  size_t one = align_up((size_t)p.BH * p.N * p.d * esize(p.dtype), 256);
  rc = grow(&B.stage, &B.stage_bytes, 4 * one);
  if (rc != MA_OK) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if (!B.all_back) {
    if (cudaStreamCreateWithFlags(&B.compute, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&B.d2h, cudaStreamNonBlocking) != cudaSuccess)
      return MA_ERR_CUDA;
    for (int c = 0; c < kHostChunks; ++c)
      if (cudaEventCreateWithFlags(&B.chunk_in[c], cudaEventDisableTiming) != cudaSuccess ||
          cudaEventCreateWithFlags(&B.chunk_done[c], cudaEventDisableTiming) != cudaSuccess)
        return MA_ERR_CUDA;
    if (cudaEventCreateWithFlags(&B.all_back, cudaEventDisableTiming) != cudaSuccess) return MA_ERR_CUDA;
  }
  // (batch, head) units are independent (Sec. 3: every equation is per head), so the call is cut
  // into chunks of units: copy in on `stream`, compute on the library's compute stream, copy back
  // on its copy-back stream, chained by events.
  const size_t unit = (size_t)p.N * p.d * esize(p.dtype);
  // The per-head kernels write each row of Y once, in whole lines: to pinned memory they write it
  // directly, and the copy back is gone.
  char* direct = nullptr;
  const int r = resolve_path(p, MA_PATH_AUTO);
  if (r == MA_PATH_FUSED_SMALL || r == MA_PATH_FUSED_F32) {
    hostcall::Pinned at;
    if (pinned_range(Yh, &at)) direct = (char*)hostcall::writable(at, (size_t)p.BH * unit);
  }
  // Every copy costs 3-4 us beyond its bytes, and copies in slow down while others go back; the copies
  // and kernels of a chunk overlap the copies of the next.  Measured with 1, 2, 3, 4 and 6 chunks (us): 0.2 MB
  // a tensor 46, 52, 62, 75, 98; 2.4 MB 220, 227, 235, 249, 268; 9.4 MB 717, 661, 661, 664, 692; 20 MB 1521, 1388,
  // 1345, 1346, 1354; 25 MB 1866, 1684, 1633, 1645, 1662.  Without the direct
  // writes: three.
  const size_t bytes = (size_t)p.BH * unit;
  const int want = g_host_chunks > 0 ? g_host_chunks : (direct && bytes < ((size_t)4 << 20) ? 1 : (direct && bytes < ((size_t)14 << 20) ? 2 : 3));
  const int chunks = (unit % 16 == 0 && p.BH >= want) ? want : 1;
  HostOps ops{B, st, chunks > 1 ? B.compute : st, chunks > 1 ? B.d2h : st, N, d, b, T, dtype, p.BH, 0};
  rc = hostcall::run({(const char*)Qh, (const char*)Kh, (const char*)Vh, (char*)Yh, (char*)B.stage, direct, one, unit}, p.BH,
                     chunks, ops);
  if (rc == MA_OK) g_last_launches = ops.launches;
  return rc;
}

int monarch_attn_device_status(const void* workspace, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  int* own = workspace ? nullptr : status_word();
  if (!workspace && !own) return MA_ERR_CUDA;
  int word = 0;
  if (cudaMemcpyAsync(&word, workspace ? workspace : own, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return MA_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return MA_ERR_CUDA;
  if (word != 0 && own) {          // reported once; an aborted run leaves counters behind: clear on the next call
    if (cudaMemsetAsync(own, 0, sizeof(int), st) != cudaSuccess) return MA_ERR_CUDA;
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevices) g_dev[dev].armed_key = -1;
  }
  return word == 0 ? MA_OK : MA_ERR_TIMEOUT;
}

int monarch_attn_last_launch_count(void) { return g_last_launches; }

const char* monarch_attn_last_kernels(void) { return g_last_kernels; }

}  // extern "C"

// ------------------------------------------------------------------ no-allocation entry point
// Scratch for monarch_attn_fwd_noalloc lives in the library image.  In host code the name of a
// __device__ array is only a handle for the runtime, never a device address: the address is
// looked up once per device with cudaGetSymbolAddress and that pointer is what kernels receive.
static __device__ __align__(256) unsigned char g_noalloc_scratch[MONARCH_ATTN_NOALLOC_SCRATCH_BYTES];
static void* g_noalloc_ptr[ma::kMaxDevices] = {nullptr};

extern "C" {

int monarch_attn_fwd_noalloc(const void* Q, const void* K, const void* V, void* Y, int batch,
                             int heads, int N, int d, int b, int T, int dtype, void* stream) {
  Problem p;
  int rc = validate_shape(batch, heads, N, d, b, T, dtype, &p);
  if (rc != MA_OK) return rc;
  rc = check_ptrs(Q, K, V, Y, p);
  if (rc != MA_OK) return rc;
  if (!generic_supported(p)) return MA_ERR_UNSUPPORTED;
  if (generic_layout(p, nullptr).bytes > (size_t)MONARCH_ATTN_NOALLOC_SCRATCH_BYTES)
    return MA_ERR_TOO_LARGE;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return MA_ERR_CUDA;
  if (!g_noalloc_ptr[dev]) {   // set-up, once per device, with that device current
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) {
      cudaGetLastError();
      return MA_ERR_CUDA;
    }
    g_noalloc_ptr[dev] = ptr;
  }
  return launch_generic(p, Q, K, V, Y, 1.0f / sqrtf((float)d), g_noalloc_ptr[dev],
                        (cudaStream_t)stream);
}

int monarch_attn_debug_knob(int knob, long long value) {
  if (knob == 1) {
    tp::knobs().wait_cycles = value > 0 ? value : tensor::kWaitCycles;
  } else if (knob == 2) {
    tp::knobs().skip_first_half_step = value != 0;
  } else if (knob == 3) {
    g_host_chunks = value < 1 ? 0 : (value > kHostChunks ? kHostChunks : (int)value);
  } else {
    return MA_ERR_SHAPE;
  }
  for (int d = 0; d < kMaxDevices; ++d) g_dev[d].armed_key = -1;
  return MA_OK;
}

int monarch_attn_set_trace_buffer(void* device_buffer, size_t bytes) {
  if (device_buffer != nullptr && bytes < (size_t)4 * 64 * 8 * sizeof(long long)) return MA_ERR_WORKSPACE;
  tp::trace_buffer() = (long long*)device_buffer;
  return MA_OK;
}

const char* monarch_attn_status_string(int status) {
  switch (status) {
    case MA_OK: return "ok";
    case MA_ERR_NULL: return "a required pointer is NULL";
    case MA_ERR_SHAPE: return "invalid shape: need batch, heads, N, d, b > 0, N % b == 0, T >= 1";
    case MA_ERR_DTYPE: return "unknown dtype";
    case MA_ERR_UNSUPPORTED: return "no kernel on the requested path for this (b, m, d, dtype)";
    case MA_ERR_ALIGN: return "pointer not aligned, or output aliases an input";
    case MA_ERR_WORKSPACE: return "workspace missing or too small";
    case MA_ERR_CUDA: return "a CUDA call failed";
    case MA_ERR_TIMEOUT: return "a bounded device-side wait ran out";
    case MA_ERR_TOO_LARGE: return "problem exceeds the scratch built into monarch_attn_fwd_noalloc";
    default: return "unknown status";
  }
}

}  // extern "C"
