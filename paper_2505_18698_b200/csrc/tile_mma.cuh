// Warp-MMA kernels for 16-bit inputs of any block shape: m, b <= 128 (m need not equal b),
// d <= 128 (a multiple of 8), f16/bf16, key padding mask (App. C.3), either layout.
//
// One launch per half-step, one CTA per tile, one warp per 16 score rows.  This is the path of the
// shapes that neither the tcgen05 kernel (d = 64, m = b in {32, 64, 128}) nor the fused per-head
// kernel (states of a head in shared memory) takes: e.g. (b, m) = (32, 64) or (64, 128) at
// N = 2048 / 8192, d = 72, d = 48 with N = 7680 = 60 blocks of 128.  The states alpha_L, alpha_R, y
// (Sec. 3 'Implementation') are f16 arrays in the workspace, c_L is fp32.
//
// Every array (Q, K, V, the states) is stored in the SAME row order, row n = k*b + i of a head, so
// alpha_R of the first round is Q itself and the permutation between the half-steps (Eq. 9, 10) is
// the choice of rows a tile gathers: an R tile copies the b consecutive rows of block k, an L tile
// the m rows (l, j) that sit b rows apart, into shared memory (rows padded by 16 bytes, so 8-row
// fragment loads are conflict-free).  Arithmetic is f16 x f16 -> fp32 (mma.sync m16n8k16; bf16
// inputs are converted on the way in), alpha_R is stored divided by c_R with the weights' columns
// rescaled by powers of two first, as in the fused kernels.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "shared_align.cuh"
#include "status_word.cuh"
#include "warp_mma.cuh"
#include "fused_small.cuh"

namespace ma {
namespace tile {

using warpmma::Mma;
using warpmma::col_sum;
using warpmma::ex2;
using warpmma::kLn2;
using warpmma::kLog2e;
using warpmma::ldsm_x4;
using warpmma::ldsm_x4_trans;
using warpmma::lg2;
using warpmma::quad_max;
using warpmma::quad_sum;
using fsmall::stsm_x4;

typedef __half T;
constexpr int kMaxSmem = 227 * 1024;
constexpr float kMasked = -1e30f;   // logit of a masked column: exp2(kMasked - max) == 0

// Shared-memory row pitch for DT 16-column steps: the 16 bytes of padding put 8 consecutive rows
// in 8 different 16-byte bank groups.
__host__ __device__ constexpr int pitch_of(int dt) { return dt * 32 + 16; }

// The half-step kernels of a call are launched with programmatic stream serialisation: the next
// launch's CTAs may take SM slots as this launch's last CTAs drain, but they touch no memory before
// every CTA of the launch before them has finished (wait), so the stream order of the data holds.
__device__ __forceinline__ void grid_dependency_sync() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Rows of head h in Q, K, V, Y: element offset of row 0 and the stride between rows.
struct HeadRows {
  size_t base, stride;
};
__device__ __forceinline__ HeadRows head_rows(int h, int N, int d, int H) {
  HeadRows r;
  r.base = H == 0 ? (size_t)h * N * d : ((size_t)(h / H) * N * H + (h % H)) * d;
  r.stride = H == 0 ? (size_t)d : (size_t)H * d;
  return r;
}

// Starts the copy of `rows` rows of d 16-bit elements (row r at src + r * stride) into a shared
// tile (asynchronous 16-byte copies of the raw values; columns d .. 16*DT - 1 are zero-filled).
// After gather_wait(), convert_rows() turns bf16 tiles into f16 in place: every thread converts
// exactly the chunks it copied, so no barrier is needed in between.
template <typename TSrc, int DT>
__device__ __forceinline__ void gather_rows(uint8_t* dst, const TSrc* __restrict__ src, size_t stride,
                                            int rows, int d) {
  constexpr int kChunks = DT * 2;
  // a thread keeps its 16-byte column and walks down the rows (blockDim.x is a multiple of 32)
  const int ch = threadIdx.x % kChunks, rstep = blockDim.x / kChunks;
  uint32_t dst_u = (uint32_t)__cvta_generic_to_shared(dst) + (threadIdx.x / kChunks) * pitch_of(DT) + ch * 16;
  if (ch * 8 < d) {
    const TSrc* p = src + (size_t)(threadIdx.x / kChunks) * stride + ch * 8;
    for (int r = threadIdx.x / kChunks; r < rows; r += rstep, p += (size_t)rstep * stride, dst_u += rstep * pitch_of(DT))
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst_u), "l"(p) : "memory");
  } else {
    for (int r = threadIdx.x / kChunks; r < rows; r += rstep)
      *reinterpret_cast<uint4*>(dst + r * pitch_of(DT) + ch * 16) = make_uint4(0u, 0u, 0u, 0u);
  }
}
__device__ __forceinline__ void gather_wait() {
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}
template <typename TSrc, int DT>
__device__ __forceinline__ void convert_rows(uint8_t* dst, int rows, int d) {
  if (!Mma<TSrc>::is_f16) {
    constexpr int kChunks = DT * 2;
    const int ch = threadIdx.x % kChunks, rstep = blockDim.x / kChunks;
    if (ch * 8 < d)
      for (int r = threadIdx.x / kChunks; r < rows; r += rstep) {
        uint4* p = reinterpret_cast<uint4*>(dst + r * pitch_of(DT) + ch * 16);
        *p = warpmma::to_f16x8(*p, (const TSrc*)nullptr);
      }
  }
}

__device__ __forceinline__ uint4 store16_from_f16(uint4 v, __half*) { return v; }
__device__ __forceinline__ uint4 store16_from_f16(uint4 v, __nv_bfloat16* p) { return warpmma::from_f16x8(v, p); }

// One warp copies its 16 staged rows (first `rows` of them valid) out: row r to dst + r * stride.
template <typename TDst, int DT>
__device__ __forceinline__ void scatter_rows16(TDst* __restrict__ dst, size_t stride, const uint8_t* src,
                                               int rows, int d, int lane) {
  constexpr int kChunks = DT * 2;              // a lane keeps its 16-byte column and walks down the rows
  const int ch = lane % kChunks;
  if (ch * 8 >= d) return;
  for (int r = lane / kChunks; r < rows; r += 32 / kChunks) {
    const uint4 v = *reinterpret_cast<const uint4*>(src + r * pitch_of(DT) + ch * 16);
    TDst* gp = dst + (size_t)r * stride + ch * 8;
    *reinterpret_cast<uint4*>(gp) = store16_from_f16(v, gp);
  }
}

// Tiles are allocated with their row count rounded up to 16: a warp stores whole 16-row fragments,
// and the rows past the block land in that padding.
__host__ __device__ constexpr int round16(int x) { return (x + 15) & ~15; }
// `hilo`: the states alpha_L and alpha_R are kept as a hi + lo pair of f16 arrays (one more tile).
// x rounded to f16 (hi) and the f16 rounding of what is left (lo): hi + lo carries 22 bits of x.
template <bool HILO>
__device__ __forceinline__ void split_hilo(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  hi = Mma<T>::pack(x0, x1);
  lo = 0u;
  if (HILO) {
    const float2 h = Mma<T>::unpack(hi);
    lo = Mma<T>::pack(x0 - h.x, x1 - h.y);
  }
}

inline size_t r_smem_bytes(int b, int dt, bool hilo) { return (size_t)(hilo ? 5 : 4) * round16(b) * pitch_of(dt); }
inline size_t l_smem_bytes(int m, int cm, int dt, bool hilo) {
  const size_t tiles = (size_t)(hilo ? 4 : 3) * round16(m) * pitch_of(dt);  // Q(l,j), alpha_L(k,j) (+ lo), y(k,j)
  const size_t p_tile = (size_t)(hilo ? 2 : 1) * round16(m) * (cm * 2 + 16);   // weights for the transposed product (+ lo)
  const size_t stats = (size_t)(2 * 8 * cm + cm) * 4;          // column max / sum per warp, c_L
  return tiles + p_tile + stats;
}

// ---------------------------------------------------------------------------------------------
// R half-step for key block k of head h (Eq. 7, 9 -> Eq. 10):
//   Z_R[j,i] = scale * <aR(k,j), K(k,i)>  (alpha_R arrives divided by c_R), R = softmax_i Z_R,
//   aL(k,j) = sum_i R[j,i] K(k,i), cL(k,j) = sum_i R log R, (last round) y(k,j) = sum_i R[j,i] V(k,i)
// CB: b rounded up to 32, 64 or 128; DT: 16-column steps over d (4 or 8).
template <typename TIn, int CB, int DT, bool HILO>
__global__ void __launch_bounds__(256)
r_tile_kernel(const TIn* __restrict__ Q, const TIn* __restrict__ K, const TIn* __restrict__ V,
              const __half* __restrict__ aR, __half* __restrict__ aL, __half* __restrict__ y,
              const __half* __restrict__ aR_lo, __half* __restrict__ aL_lo,
              float* __restrict__ cL, int N, int d, int b, float scale, int n_valid, int H, int first,
              int last, const int* __restrict__ seq_len, int heads, int* clear) {
  extern __shared__ __align__(128) uint8_t smem[];
  constexpr int kPitch = pitch_of(DT);
  grid_dependency_sync();
  clear_status(clear);
  const int k = blockIdx.x, h = blockIdx.y;
  // Batched sequences of different lengths (App. C.3): a key block that lies wholly in this
  // sequence's padding is absent from its problem (the L half-step never reads its rows of the
  // states); the last block that is present gets the appendix's mask.
  if (seq_len != nullptr) {
    n_valid = min(max(seq_len[h / heads], 1), N);
    if (k * b >= n_valid) return;
  }
  const int warp = warp_of_cta(), lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int rb = round16(b);
  uint8_t* sA = smem;
  uint8_t* sK = sA + (size_t)rb * kPitch;
  uint8_t* sV = sK + (size_t)rb * kPitch;
  uint8_t* sY = sV + (size_t)rb * kPitch;      // staging of y rows on the last round
  uint8_t* sAlo = sY + (size_t)rb * kPitch;    // low halves of alpha_R in, of alpha_L out (hi + lo states)
  constexpr bool hilo = HILO;
  const HeadRows hr = head_rows(h, N, d, H);
  const size_t st_rows = ((size_t)h * N + (size_t)k * b) * d;    // block k of the state arrays

  if (first) gather_rows<TIn, DT>(sA, Q + hr.base + (size_t)k * b * hr.stride, hr.stride, b, d);
  else gather_rows<__half, DT>(sA, aR + st_rows, (size_t)d, b, d);
  if (!first && hilo) gather_rows<__half, DT>(sAlo, aR_lo + st_rows, (size_t)d, b, d);
  gather_rows<TIn, DT>(sK, K + hr.base + (size_t)k * b * hr.stride, hr.stride, b, d);
  if (last) gather_rows<TIn, DT>(sV, V + hr.base + (size_t)k * b * hr.stride, hr.stride, b, d);
  gather_wait();
  if (first) convert_rows<TIn, DT>(sA, b, d);
  convert_rows<TIn, DT>(sK, b, d);
  if (last) convert_rows<TIn, DT>(sV, b, d);
  __syncthreads();

  const int j0 = 16 * warp;
  if (j0 >= b) return;
  const uint32_t sA_u = (uint32_t)__cvta_generic_to_shared(sA), sK_u = (uint32_t)__cvta_generic_to_shared(sK);
  const uint32_t sV_u = (uint32_t)__cvta_generic_to_shared(sV), sY_u = (uint32_t)__cvta_generic_to_shared(sY);
  const float fl = scale * kLog2e;
  const int ilim = min(b, n_valid - k * b);          // valid key columns of this block

  float s[CB / 8][4];
#pragma unroll
  for (int nt = 0; nt < CB / 8; ++nt)
#pragma unroll
    for (int e = 0; e < 4; ++e) s[nt][e] = 0.f;
  {
    const uint32_t a_u = sA_u + min(j0 + (lane & 7) + ((lane >> 3) & 1) * 8, b - 1) * kPitch + (lane >> 4) * 16;
    uint32_t b_u[CB / 16];
#pragma unroll
    for (int cp = 0; cp < CB / 16; ++cp)
      b_u[cp] = sK_u + min(16 * cp + (lane & 7) + (lane >> 4) * 8, b - 1) * kPitch + ((lane >> 3) & 1) * 16;
#pragma unroll
    for (int ks = 0; ks < DT; ++ks) {
      uint32_t a[4];
      ldsm_x4(a, a_u + ks * 32);
#pragma unroll
      for (int cp = 0; cp < CB / 16; ++cp) {
        if (16 * cp >= b) continue;
        uint32_t bf[4];
        ldsm_x4(bf, b_u[cp] + ks * 32);
        Mma<T>::run(s[2 * cp], a, bf);
        Mma<T>::run(s[2 * cp + 1], a, bf + 2);
      }
    }
    if (!first && hilo) {      // + <alpha_R lo, K>
      const uint32_t alo_u = a_u - sA_u + (uint32_t)__cvta_generic_to_shared(sAlo);
#pragma unroll
      for (int ks = 0; ks < DT; ++ks) {
        uint32_t a[4];
        ldsm_x4(a, alo_u + ks * 32);
#pragma unroll
        for (int cp = 0; cp < CB / 16; ++cp) {
          if (16 * cp >= b) continue;
          uint32_t bf[4];
          ldsm_x4(bf, b_u[cp] + ks * 32);
          Mma<T>::run(s[2 * cp], a, bf);
          Mma<T>::run(s[2 * cp + 1], a, bf + 2);
        }
      }
    }
  }
  // rows j = j0 + g (c0, c1) and j0 + g + 8 (c2, c3); columns i = 8 nt + 2t, +1
  float inv_s[2];
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    const int j = j0 + g + 8 * hh;
    // masked columns (past the block, or past n_valid: App. C.3) get a huge negative FINITE
    // logit: their weight is exactly 0 and 0 * z stays 0 in the entropy sum (0 log 0 = 0)
    float mx = kMasked;
#pragma unroll
    for (int nt = 0; nt < CB / 8; ++nt)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float z = (8 * nt + 2 * t + e < ilim) ? s[nt][2 * hh + e] * fl : kMasked;
        s[nt][2 * hh + e] = z;
        mx = fmaxf(mx, z);
      }
    mx = quad_max(mx);
    float sum = 0.f, sz = 0.f;
#pragma unroll
    for (int nt = 0; nt < CB / 8; ++nt)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float z = s[nt][2 * hh + e];
        const float p = ex2(z - mx);                 // 0 for masked columns
        s[nt][2 * hh + e] = p;
        sum += p;
        sz = fmaf(p, z, sz);
      }
    sum = quad_sum(sum);
    sz = quad_sum(sz);
    inv_s[hh] = 1.f / sum;
    // c_L = sum R log R (natural log): ln2 * (sum p z / sum - max - log2 sum)
    if (t == 0 && j < b) cL[(size_t)h * N + (size_t)k * b + j] = kLn2 * (sz * inv_s[hh] - mx - lg2(sum));
  }
  // Weights as A fragments.  With hi + lo states (HILO) the weights are a hi + lo pair as well:
  // alpha_L feeds logits of size ~100, so the 2^-12 relative rounding of a dominant weight is a
  // logit error of a few hundredths, and from the third round on that alone costs more than 1e-2
  // on the worst head of a peaky recipe (measured 2.7e-2; 2e-4 with the pair).
  uint32_t pa[CB / 16][4], pal[HILO ? CB / 16 : 1][4];
#pragma unroll
  for (int kk = 0; kk < CB / 16; ++kk) {
    pa[kk][0] = Mma<T>::pack(s[2 * kk][0], s[2 * kk][1]);
    pa[kk][1] = Mma<T>::pack(s[2 * kk][2], s[2 * kk][3]);
    pa[kk][2] = Mma<T>::pack(s[2 * kk + 1][0], s[2 * kk + 1][1]);
    pa[kk][3] = Mma<T>::pack(s[2 * kk + 1][2], s[2 * kk + 1][3]);
    if (HILO) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2 hi = Mma<T>::unpack(pa[kk][q]);
        const int nt = 2 * kk + (q >> 1), e0 = 2 * (q & 1);
        pal[kk][q] = Mma<T>::pack(s[nt][e0] - hi.x, s[nt][e0 + 1] - hi.y);
      }
    }
  }
  // second products, two 8-column tiles of v at a time; results staged in this warp's own 16 rows
  // of the alpha_R tile (dead: only this warp read them) and of the y staging tile
  const int st_row = (lane & 7) + ((lane >> 3) & 1) * 8, st_nt = (lane >> 4) & 1;
  const uint32_t stA_u = sA_u + (j0 + st_row) * kPitch + st_nt * 16;
  const uint32_t stY_u = sY_u + (j0 + st_row) * kPitch + st_nt * 16;
  const uint32_t stLo_u = (uint32_t)__cvta_generic_to_shared(sAlo) + (j0 + st_row) * kPitch + st_nt * 16;
  __syncwarp();
  uint32_t v_off[CB / 16];
#pragma unroll
  for (int kk = 0; kk < CB / 16; ++kk) v_off[kk] = min(16 * kk + (lane & 15), b - 1) * kPitch + (lane >> 4) * 16;
#pragma unroll
  for (int np = 0; np < DT; ++np) {
    float o[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    float yv[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int kk = 0; kk < CB / 16; ++kk) {
      if (16 * kk >= b) continue;
      uint32_t bf[4];
      const uint32_t off = v_off[kk] + np * 32;
      ldsm_x4_trans(bf, sK_u + off);
      Mma<T>::run(o[0], pa[kk], bf);
      Mma<T>::run(o[1], pa[kk], bf + 2);
      if (HILO) {
        Mma<T>::run(o[0], pal[kk], bf);
        Mma<T>::run(o[1], pal[kk], bf + 2);
      }
      if (last) {
        ldsm_x4_trans(bf, sV_u + off);
        Mma<T>::run(yv[0], pa[kk], bf);
        Mma<T>::run(yv[1], pa[kk], bf + 2);
      }
    }
    uint32_t hi[4], lo[4];
    split_hilo<HILO>(o[0][0] * inv_s[0], o[0][1] * inv_s[0], hi[0], lo[0]);
    split_hilo<HILO>(o[0][2] * inv_s[1], o[0][3] * inv_s[1], hi[1], lo[1]);
    split_hilo<HILO>(o[1][0] * inv_s[0], o[1][1] * inv_s[0], hi[2], lo[2]);
    split_hilo<HILO>(o[1][2] * inv_s[1], o[1][3] * inv_s[1], hi[3], lo[3]);
    stsm_x4(stA_u + np * 32, hi[0], hi[1], hi[2], hi[3]);
    if (hilo) stsm_x4(stLo_u + np * 32, lo[0], lo[1], lo[2], lo[3]);
    if (last)
      stsm_x4(stY_u + np * 32, Mma<T>::pack(yv[0][0] * inv_s[0], yv[0][1] * inv_s[0]),
              Mma<T>::pack(yv[0][2] * inv_s[1], yv[0][3] * inv_s[1]),
              Mma<T>::pack(yv[1][0] * inv_s[0], yv[1][1] * inv_s[0]),
              Mma<T>::pack(yv[1][2] * inv_s[1], yv[1][3] * inv_s[1]));
  }
  __syncwarp();
  const int rows = min(16, b - j0);
  scatter_rows16<__half, DT>(aL + st_rows + (size_t)j0 * d, (size_t)d, sA + (size_t)j0 * kPitch, rows, d, lane);
  if (hilo)
    scatter_rows16<__half, DT>(aL_lo + st_rows + (size_t)j0 * d, (size_t)d, sAlo + (size_t)j0 * kPitch, rows, d, lane);
  if (last)
    scatter_rows16<__half, DT>(y + st_rows + (size_t)j0 * d, (size_t)d, sY + (size_t)j0 * kPitch, rows, d, lane);
}

// ---------------------------------------------------------------------------------------------
// L half-step for in-block position j of head h (Eq. 8, 10 -> Eq. 9 or Eq. 4):
//   Z_L[l,k] = scale * <Q(l,j), aL(k,j)> - cL(k,j), L = softmax_k Z_L
//   not final: aR(k,j) = sum_l L[l,k] Q(l,j) / cR(k,j), cR(k,j) = sum_l L[l,k]
//   final:     Y(l,j) = sum_k L[l,k] y(k,j); optionally the row's log-sum-exp (Eq. 6)
// CM: m rounded up to 32, 64 or 128.
template <typename TIn, int CM, int DT, bool HILO>
__global__ void __launch_bounds__(256)
l_tile_kernel(const TIn* __restrict__ Q, const __half* __restrict__ aL, const float* __restrict__ cL,
              const __half* __restrict__ y, __half* __restrict__ aR, const __half* __restrict__ aL_lo,
              __half* __restrict__ aR_lo, TIn* __restrict__ Y, float* __restrict__ lse, int N, int d, int b,
              int m, float scale, int H, int last, const int* __restrict__ seq_len, int heads) {
  extern __shared__ __align__(128) uint8_t smem[];
  constexpr int kPitch = pitch_of(DT), kPPitch = CM * 2 + 16;
  grid_dependency_sync();
  const int j = blockIdx.x, h = blockIdx.y;
  // Batched sequences of different lengths (App. C.3): this sequence's problem has the blocks
  // 0 .. ceil(length / b) - 1 only; rows of Y in blocks past them are written as zeros.
  const int m_alloc = m;
  if (seq_len != nullptr) m = (min(max(seq_len[h / heads], 1), N) + b - 1) / b;
  const int warp = warp_of_cta(), lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int rm = round16(m);
  uint8_t* sQ = smem;
  uint8_t* sL = sQ + (size_t)rm * kPitch;
  uint8_t* sYt = sL + (size_t)rm * kPitch;
  constexpr bool hilo = HILO;
  uint8_t* sLlo = sYt + (size_t)rm * kPitch;   // low halves of alpha_L in, of alpha_R out (hi + lo states)
  uint8_t* sP = sLlo + (hilo ? (size_t)rm * kPitch : 0);
  uint8_t* sPlo = sP + (size_t)rm * kPPitch;   // low halves of the non-final weights (hi + lo states)
  float* sColMax = reinterpret_cast<float*>(sPlo + (hilo ? (size_t)rm * kPPitch : 0));
  float* sColSum = sColMax + 8 * CM;
  float* sC = sColSum + 8 * CM;
  const HeadRows hr = head_rows(h, N, d, H);
  const size_t st_rows = ((size_t)h * N + j) * d;              // row (0, j) of the state arrays
  const size_t st_stride = (size_t)b * d;                      // rows (k, j), (k+1, j) are b rows apart

  gather_rows<TIn, DT>(sQ, Q + hr.base + (size_t)j * hr.stride, (size_t)b * hr.stride, m, d);
  gather_rows<__half, DT>(sL, aL + st_rows, st_stride, m, d);
  if (hilo) gather_rows<__half, DT>(sLlo, aL_lo + st_rows, st_stride, m, d);
  if (last) gather_rows<__half, DT>(sYt, y + st_rows, st_stride, m, d);
  for (int kq = threadIdx.x; kq < m; kq += blockDim.x) sC[kq] = cL[(size_t)h * N + (size_t)kq * b + j] * kLog2e;
  gather_wait();
  convert_rows<TIn, DT>(sQ, m, d);
  __syncthreads();

  const int l0 = 16 * warp;
  const bool active = l0 < m;
  const uint32_t sQ_u = (uint32_t)__cvta_generic_to_shared(sQ), sL_u = (uint32_t)__cvta_generic_to_shared(sL);
  const uint32_t sY_u = (uint32_t)__cvta_generic_to_shared(sYt), sP_u = (uint32_t)__cvta_generic_to_shared(sP);
  const float fl = scale * kLog2e;
  const int st_row = (lane & 7) + ((lane >> 3) & 1) * 8, st_nt = (lane >> 4) & 1;

  float s[CM / 8][4];
  float inv_s[2] = {0.f, 0.f};
  if (active) {
#pragma unroll
    for (int nt = 0; nt < CM / 8; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) s[nt][e] = 0.f;
    const uint32_t a_u = sQ_u + min(l0 + (lane & 7) + ((lane >> 3) & 1) * 8, m - 1) * kPitch + (lane >> 4) * 16;
    uint32_t b_u[CM / 16];
#pragma unroll
    for (int cp = 0; cp < CM / 16; ++cp)
      b_u[cp] = sL_u + min(16 * cp + (lane & 7) + (lane >> 4) * 8, m - 1) * kPitch + ((lane >> 3) & 1) * 16;
#pragma unroll
    for (int ks = 0; ks < DT; ++ks) {
      uint32_t a[4];
      ldsm_x4(a, a_u + ks * 32);
#pragma unroll
      for (int cp = 0; cp < CM / 16; ++cp) {
        if (16 * cp >= m) continue;
        uint32_t bf[4];
        ldsm_x4(bf, b_u[cp] + ks * 32);
        Mma<T>::run(s[2 * cp], a, bf);
        Mma<T>::run(s[2 * cp + 1], a, bf + 2);
        if (hilo) {      // + <Q, alpha_L lo>
          ldsm_x4(bf, b_u[cp] - sL_u + (uint32_t)__cvta_generic_to_shared(sLlo) + ks * 32);
          Mma<T>::run(s[2 * cp], a, bf);
          Mma<T>::run(s[2 * cp + 1], a, bf + 2);
        }
      }
    }
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      float mx = kMasked;
#pragma unroll
      for (int nt = 0; nt < CM / 8; ++nt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int kc = 8 * nt + 2 * t + e;
          const float z = kc < m ? fmaf(s[nt][2 * hh + e], fl, -sC[kc]) : kMasked;
          s[nt][2 * hh + e] = z;
          mx = fmaxf(mx, z);
        }
      mx = quad_max(mx);
      float sum = 0.f;
#pragma unroll
      for (int nt = 0; nt < CM / 8; ++nt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float p = ex2(s[nt][2 * hh + e] - mx);
          s[nt][2 * hh + e] = p;
          sum += p;
        }
      sum = quad_sum(sum);
      inv_s[hh] = 1.f / sum;
      const int l = l0 + g + 8 * hh;
      if (last && lse != nullptr && t == 0 && l < m)
        lse[(size_t)h * N + (size_t)l * b + j] = (mx + log2f(sum)) * kLn2;
    }
  }

  if (last) {
    if (m < m_alloc) {
      const HeadRows hz = head_rows(h, N, d, H);
      const int cpr = d / 8;                       // 16-byte chunks per row
      for (int idx = threadIdx.x; idx < (m_alloc - m) * cpr; idx += blockDim.x) {
        const int l = m + idx / cpr, ch = idx - (idx / cpr) * cpr;
        *reinterpret_cast<uint4*>(Y + hz.base + ((size_t)l * b + j) * hz.stride + ch * 8) = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    if (!active) return;
    // Y(l,j) = sum_k L[l,k] y(k,j): A = weights rows l, B = y rows (k,j) read transposed
    uint32_t pa[CM / 16][4];
#pragma unroll
    for (int kk = 0; kk < CM / 16; ++kk) {
      pa[kk][0] = Mma<T>::pack(s[2 * kk][0], s[2 * kk][1]);
      pa[kk][1] = Mma<T>::pack(s[2 * kk][2], s[2 * kk][3]);
      pa[kk][2] = Mma<T>::pack(s[2 * kk + 1][0], s[2 * kk + 1][1]);
      pa[kk][3] = Mma<T>::pack(s[2 * kk + 1][2], s[2 * kk + 1][3]);
    }
    // staged in this warp's own rows of the Q tile (only this warp read them)
    const uint32_t st_u = sQ_u + (l0 + st_row) * kPitch + st_nt * 16;
    __syncwarp();
#pragma unroll
    for (int np = 0; np < DT; ++np) {
      float o[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
      for (int kk = 0; kk < CM / 16; ++kk) {
        if (16 * kk >= m) continue;
        uint32_t bf[4];
        ldsm_x4_trans(bf, sY_u + min(16 * kk + (lane & 15), m - 1) * kPitch + (lane >> 4) * 16 + np * 32);
        Mma<T>::run(o[0], pa[kk], bf);
        Mma<T>::run(o[1], pa[kk], bf + 2);
      }
      stsm_x4(st_u + np * 32, Mma<T>::pack(o[0][0] * inv_s[0], o[0][1] * inv_s[0]),
              Mma<T>::pack(o[0][2] * inv_s[1], o[0][3] * inv_s[1]),
              Mma<T>::pack(o[1][0] * inv_s[0], o[1][1] * inv_s[0]),
              Mma<T>::pack(o[1][2] * inv_s[1], o[1][3] * inv_s[1]));
    }
    __syncwarp();
    scatter_rows16<TIn, DT>(Y + hr.base + ((size_t)l0 * b + j) * hr.stride, (size_t)b * hr.stride,
                            sQ + (size_t)l0 * kPitch, min(16, m - l0), d, lane);
    return;
  }

  // ---- not final: alpha_R(k,j) = sum_l L[l,k] Q(l,j) / c_R(k,j).  The contraction runs over the
  // rows of the weights, which are spread over the warps: the normalised weights go through a
  // shared tile.  Before rounding to 16 bits every column k is multiplied by a power of two g_k
  // (the result is invariant) so that its largest weight is near 1 however small c_R is, and c_R
  // is summed over the weights AS ROUNDED, so that numerator and denominator see the same numbers.
  if (active) {
#pragma unroll
    for (int nt = 0; nt < CM / 8; ++nt)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float p0 = (l0 + g < m) ? s[nt][e] * inv_s[0] : 0.f;          // rows past the block: 0
        const float p1 = (l0 + g + 8 < m) ? s[nt][2 + e] * inv_s[1] : 0.f;
        s[nt][e] = p0;
        s[nt][2 + e] = p1;
        float cm = fmaxf(p0, p1);
        cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, 4));
        cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, 8));
        cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, 16));
        if (g == 0) sColMax[warp * CM + 8 * nt + 2 * t + e] = cm;
      }
  }
  __syncthreads();
  const int row_warps = (m + 15) >> 4;       // warps that hold weight rows
  if (active) {
    const uint32_t st_u = sP_u + (l0 + st_row) * kPPitch + st_nt * 16;
#pragma unroll
    for (int np = 0; np < CM / 16; ++np) {
      uint32_t u[2][2], ul[2][2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int nt = 2 * np + q;
        float gk[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float cm = 0.f;
          for (int w = 0; w < row_warps; ++w) cm = fmaxf(cm, sColMax[w * CM + 8 * nt + 2 * t + e]);
          gk[e] = cm > 0.f ? __uint_as_float((253u << 23) - (__float_as_uint(cm) & 0x7f800000u)) : 0.f;
        }
        const float w00 = s[nt][0] * gk[0], w01 = s[nt][1] * gk[1];
        const float w10 = s[nt][2] * gk[0], w11 = s[nt][3] * gk[1];
        u[q][0] = Mma<T>::pack(w00, w01);
        u[q][1] = Mma<T>::pack(w10, w11);
        float2 f0 = Mma<T>::unpack(u[q][0]), f1 = Mma<T>::unpack(u[q][1]);
        if (hilo) {      // weights as a hi + lo pair (see r_tile_kernel); c_R sums both halves
          ul[q][0] = Mma<T>::pack(w00 - f0.x, w01 - f0.y);
          ul[q][1] = Mma<T>::pack(w10 - f1.x, w11 - f1.y);
          const float2 g0 = Mma<T>::unpack(ul[q][0]), g1 = Mma<T>::unpack(ul[q][1]);
          f0.x += g0.x; f0.y += g0.y; f1.x += g1.x; f1.y += g1.y;
        }
        const float c0 = col_sum(f0.x + f1.x), c1 = col_sum(f0.y + f1.y);
        if (g == 0) {
          sColSum[warp * CM + 8 * nt + 2 * t] = c0;
          sColSum[warp * CM + 8 * nt + 2 * t + 1] = c1;
        }
      }
      stsm_x4(st_u + np * 32, u[0][0], u[0][1], u[1][0], u[1][1]);
      if (hilo)
        stsm_x4(st_u - sP_u + (uint32_t)__cvta_generic_to_shared(sPlo) + np * 32, ul[0][0], ul[0][1], ul[1][0],
                ul[1][1]);
    }
  }
  __syncthreads();
  // warp kt forms rows k = 16 kt .. 16 kt + 15 of alpha_R
  const int k0 = 16 * warp;
  if (k0 >= m) return;
  float ic[2];
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    const int kq = min(k0 + g + 8 * hh, CM - 1);
    float cr = 0.f;
    for (int w = 0; w < row_warps; ++w) cr += sColSum[w * CM + kq];
    ic[hh] = cr > 1e-30f ? 1.f / cr : 0.f;     // c_R underflow: alpha_R = 0, a uniform row next
  }
  // staged in this warp's rows k of the alpha_L tile (every warp is done reading it)
  const uint32_t st_u = sL_u + (k0 + st_row) * kPitch + st_nt * 16;
  // A = weights transposed: element (k, l) from the tile stored [l][k] (its rows l >= m are the
  // zero rows the owning warp stored, so a partly filled 16-row step contributes nothing)
  const uint32_t pt_u = sP_u + ((lane & 7) + ((lane >> 4) & 1) * 8) * kPPitch + (k0 + ((lane >> 3) & 1) * 8) * 2;
#pragma unroll
  for (int np = 0; np < DT; ++np) {
    float o[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int ls = 0; ls < CM / 16; ++ls) {
      if (16 * ls >= m) continue;
      uint32_t a[4], bf[4];
      ldsm_x4_trans(a, pt_u + 16 * ls * kPPitch);
      ldsm_x4_trans(bf, sQ_u + min(16 * ls + (lane & 15), m - 1) * kPitch + (lane >> 4) * 16 + np * 32);
      Mma<T>::run(o[0], a, bf);
      Mma<T>::run(o[1], a, bf + 2);
      if (hilo) {
        ldsm_x4_trans(a, pt_u - sP_u + (uint32_t)__cvta_generic_to_shared(sPlo) + 16 * ls * kPPitch);
        Mma<T>::run(o[0], a, bf);
        Mma<T>::run(o[1], a, bf + 2);
      }
    }
    uint32_t hi[4], lo[4];
    split_hilo<HILO>(o[0][0] * ic[0], o[0][1] * ic[0], hi[0], lo[0]);
    split_hilo<HILO>(o[0][2] * ic[1], o[0][3] * ic[1], hi[1], lo[1]);
    split_hilo<HILO>(o[1][0] * ic[0], o[1][1] * ic[0], hi[2], lo[2]);
    split_hilo<HILO>(o[1][2] * ic[1], o[1][3] * ic[1], hi[3], lo[3]);
    stsm_x4(st_u + np * 32, hi[0], hi[1], hi[2], hi[3]);
    if (hilo) stsm_x4(st_u - sL_u + (uint32_t)__cvta_generic_to_shared(sLlo) + np * 32, lo[0], lo[1], lo[2], lo[3]);
  }
  __syncwarp();
  scatter_rows16<__half, DT>(aR + st_rows + (size_t)k0 * st_stride, st_stride, sL + (size_t)k0 * kPitch,
                             min(16, m - k0), d, lane);
  if (hilo)
    scatter_rows16<__half, DT>(aR_lo + st_rows + (size_t)k0 * st_stride, st_stride, sLlo + (size_t)k0 * kPitch,
                               min(16, m - k0), d, lane);
}

// ---------------------------------------------------------------------------------------------
// Host side: workspace layout and launches.
inline bool supported(int N, int d, int b, int m, int dtype, int BH) {
  (void)N;
  if (dtype != 1 && dtype != 2) return false;
  if (d % 8 != 0 || d > 128 || b > 128 || m > 128 || BH > 65535) return false;
  const int dt = d <= 64 ? 4 : 8, cm = m <= 32 ? 32 : (m <= 64 ? 64 : 128);
  return r_smem_bytes(b, dt, true) <= (size_t)kMaxSmem && l_smem_bytes(m, cm, dt, true) <= (size_t)kMaxSmem;
}
// From the third round on the states alpha_L and alpha_R are hi + lo pairs of f16 arrays: they feed
// logits of size ~100, and with peaky logits their 2^-11 rounding, fed back round after round,
// costs more than 1e-2 on the worst head from T = 3 on (measured; 2 rounds stay at 3e-3).
inline bool uses_hilo(int T) { return T >= 3; }

struct Ws {
  __half *aL, *aR, *y, *aL_lo, *aR_lo;
  float* cL;
  size_t bytes;
};
inline Ws ws_layout(void* base, int BH, int N, int d, int b, bool hilo) {
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  Ws w;
  char* c = (char*)base;
  size_t off = 256;                                   // status word, which the waits of the tcgen05 tiles set
  const size_t big = up((size_t)BH * N * d * 2);
  w.aL = (__half*)(c + off); off += big;
  w.aR = (__half*)(c + off); off += big;
  w.y = (__half*)(c + off); off += big;
  // (rows of m floats; the tcgen05 tiles, which serve the calls with plain states, want them 16-byte aligned)
  w.cL = (float*)(c + off); off += up((size_t)BH * b * (hilo ? N / b : (N / b + 3) / 4 * 4) * 4);
  w.aL_lo = w.aR_lo = nullptr;
  if (hilo) {
    w.aL_lo = (__half*)(c + off); off += big;
    w.aR_lo = (__half*)(c + off); off += big;
  }
  w.bytes = off;
  return w;
}
inline size_t workspace_bytes(int BH, int N, int d, int b, int T) { return ws_layout(nullptr, BH, N, d, b, uses_hilo(T)).bytes; }

// Launch configuration with programmatic stream serialisation (see grid_dependency_sync).
inline cudaLaunchConfig_t serialised_config(dim3 grid, int threads, size_t smem, cudaStream_t st) {
  static cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cfg;
}

struct Args {
  const void *Q, *K, *V;
  void* Y;
  float* lse;
  int BH, N, d, b, m, T, n_valid, H;
  float scale;
  const int* seq_len = nullptr;   // optional DEVICE array [BH / heads]: valid length of every sequence
  int heads = 1;
  int* clear = nullptr;           // status word of a caller's workspace
};

int launch(const Args& a, int dtype, void* ws, cudaStream_t st, int* launches);

#ifdef MA_TU_TILE_MMA
template <typename TIn, int CB, int DT, bool HILO>
inline int launch_r(const Args& a, const Ws& w, bool first, bool last, cudaStream_t st) {
  auto kern = r_tile_kernel<TIn, CB, DT, HILO>;
  const size_t smem = r_smem_bytes(a.b, DT, HILO);
  static warpmma::SmemOptIn opt_in;
  if (!opt_in.done((const void*)kern, kMaxSmem)) return 7;
  cudaLaunchConfig_t cfg = serialised_config(dim3(a.m, a.BH), 32 * ((a.b + 15) / 16), smem, st);
  return cudaLaunchKernelEx(&cfg, kern, (const TIn*)a.Q, (const TIn*)a.K, (const TIn*)a.V, (const __half*)w.aR,
                            w.aL, w.y, (const __half*)w.aR_lo, w.aL_lo, w.cL, a.N, a.d, a.b, a.scale, a.n_valid,
                            a.H, first ? 1 : 0, last ? 1 : 0, a.seq_len, a.heads, first ? a.clear : nullptr) == cudaSuccess
             ? 0
             : 7;
}
template <typename TIn, int CM, int DT, bool HILO>
inline int launch_l(const Args& a, const Ws& w, bool last, cudaStream_t st) {
  auto kern = l_tile_kernel<TIn, CM, DT, HILO>;
  const size_t smem = l_smem_bytes(a.m, CM, DT, HILO);
  static warpmma::SmemOptIn opt_in;
  if (!opt_in.done((const void*)kern, kMaxSmem)) return 7;
  cudaLaunchConfig_t cfg = serialised_config(dim3(a.b, a.BH), 32 * ((a.m + 15) / 16), smem, st);
  return cudaLaunchKernelEx(&cfg, kern, (const TIn*)a.Q, (const __half*)w.aL, (const float*)w.cL,
                            (const __half*)w.y, w.aR, (const __half*)w.aL_lo, w.aR_lo, (TIn*)a.Y,
                            last ? a.lse : (float*)nullptr, a.N, a.d, a.b, a.m, a.scale, a.H, last ? 1 : 0, a.seq_len,
                            a.heads) == cudaSuccess
             ? 0
             : 7;
}

template <typename TIn, int DT, bool HILO>
inline int launch_td(const Args& a, void* ws, cudaStream_t st, int* launches) {
  const Ws w = ws_layout(ws, a.BH, a.N, a.d, a.b, HILO);
  int n = 0;
  for (int t = 1; t <= a.T; ++t) {
    const bool first = t == 1, last = t == a.T;
    int rc;
    if (a.b <= 32) rc = launch_r<TIn, 32, DT, HILO>(a, w, first, last, st);
    else if (a.b <= 64) rc = launch_r<TIn, 64, DT, HILO>(a, w, first, last, st);
    else rc = launch_r<TIn, 128, DT, HILO>(a, w, first, last, st);
    if (rc != 0) return rc;
    if (a.m <= 32) rc = launch_l<TIn, 32, DT, HILO>(a, w, last, st);
    else if (a.m <= 64) rc = launch_l<TIn, 64, DT, HILO>(a, w, last, st);
    else rc = launch_l<TIn, 128, DT, HILO>(a, w, last, st);
    if (rc != 0) return rc;
    n += 2;
  }
  if (cudaGetLastError() != cudaSuccess) return 7;
  *launches = n;
  return 0;
}

template <typename TIn, bool HILO>
inline int launch_h(const Args& a, void* ws, cudaStream_t st, int* launches) {
  return a.d <= 64 ? launch_td<TIn, 4, HILO>(a, ws, st, launches) : launch_td<TIn, 8, HILO>(a, ws, st, launches);
}
int launch(const Args& a, int dtype, void* ws, cudaStream_t st, int* launches) {
  if (dtype == 1)
    return uses_hilo(a.T) ? launch_h<__half, true>(a, ws, st, launches) : launch_h<__half, false>(a, ws, st, launches);
  return uses_hilo(a.T) ? launch_h<__nv_bfloat16, true>(a, ws, st, launches)
                        : launch_h<__nv_bfloat16, false>(a, ws, st, launches);
}

#endif  // MA_TU_TILE_MMA

}  // namespace tile
}  // namespace ma
