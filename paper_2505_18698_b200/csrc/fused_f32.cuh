// Fused fp32 kernel for short sequences: all T rounds of Eq. 7-10 and the Monarch multiply of Eq. 4
// in ONE launch, fp32 arithmetic and fp32 states in shared memory (the accuracy of the generic
// kernels without their 2T launches and their round trips through the workspace).
//
// Within a head the whole recursion is independent across the in-block position j: row (l, j) of
// the Monarch matrix is L[j,:,l] (x) R[:,j,:], and R[k,j,:], c_L[j,k], alpha_L[j,k,:], L[j,:,:],
// alpha_R[k,j,:], c_R[k,j], y[j,k,:] only ever read quantities with the SAME j, plus K, V and the m
// rows (l, j) of Q (Eq. 7-10: the softmax over i and the sum over i couple a key block, the softmax
// over k and the sum over l couple a position).  A CTA therefore owns JT positions of one head, keeps
// all of K and its own rows of Q on chip, and runs every half-step for its positions with no exchange
// with other CTAs; `positions_per_cta` trades CTAs in flight against the copies of K.
//
// What bounds it: FFMA issue and the shared-memory reads that feed it.  Every product of a half-step
// is a batch of small matrix products, so a thread forms a register tile (4 positions x 2 keys of the
// scores, 4 rows x 4 columns of the second products) from 16-byte loads: 1 to 1.5 shared-memory
// wavefronts per clock of FMA work at JT = 4, where one lane per output needed 8.  A group of 8 or 16
// lanes (32 for one position) holds whole score rows, so scores and softmax are one step.  Rows are an
// odd number of 16-byte units apart, and so are blocks, so that the eight rows a load touches are
// conflict-free along a block (R) and across blocks (L).  alpha_R and alpha_L replace each other in place,
// V is read once, from global memory (requested into L2 at the start), and y takes rows of K.
//
// Measured (B200, us per call, against one lane per output): 96 heads of 256 = 16 x 16, three rounds 44 /
// 224; 96 of 384 = 16 x 24, one round 39 / 193; 12 of 256, two rounds 13.4 / 30; one head, one round 7.7 /
// 10.3.  Index arithmetic without integer division, ragged reads out of the way (code 126 -> 41 KB and 140 ->
// 64 KB: instruction fetch was the first stall) and weights stored normalised took 8 to 20 % off.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "generic_kernels.cuh"
#include "status_word.cuh"
#include "tensor_path.cuh"

namespace ma {
namespace ffused {

using generic::ld_as_float;
using generic::st_from_float;

constexpr int kThreads = 256, kMaxSmem = 227 * 1024;

// Shared memory in 16-byte units: K [k][i], then for the CTA's JT positions Q and alpha_R / alpha_L
// [k or l][jj], the weights of a half-step [row][column], and c_L, c_R per row.
struct Layout {
  int d4, pu, bu, ju, su;      // units of a row, row pitch, block pitch of K, of Q and alpha, pitch of a row of weights
  int Q, A, S, C, total;
};
__host__ __device__ inline Layout layout(int d, int b, int m, int JT) {
  Layout y;
  y.d4 = (d + 3) / 4;
  y.pu = y.d4 | 1;
  y.bu = (b * y.pu) | 1;
  y.ju = (JT * y.pu) | 1;
  y.su = (((b > m ? b : m) + 3) / 4) | 1;
  y.Q = m * y.bu;
  y.A = y.Q + m * y.ju;
  y.S = y.A + m * y.ju;
  y.C = y.S + JT * m * y.su;
  y.total = y.C + 2 * ((JT * m + 3) / 4);
  return y;
}
inline size_t smem_bytes(int d, int b, int m, int JT) { return (size_t)layout(d, b, m, JT).total * 16; }

// Positions per CTA: the number for which the fullest SM has the least to do, a CTA costing its
// positions and about three more for its copy of K and its start (measured: 1 to 3 agree on most shapes;
// 32 heads of 384 = 16 x 24, two rounds: 42 us with 1, 33 with 3); a third more where no second CTA fits
// beside it (96 heads of 256 = 16 x 16, three rounds: 43 us with 4 positions, 64 with the 16 that just fit;
// 36 heads of 238 = 14 x 17, two rounds: 22 with 4, 27.5 with 8).
inline int positions_per_cta(int d, int b, int m, int BH, int num_sms) {
  int best = 0;
  long long least = 0;
  for (int jt = 1; jt <= b; jt = jt < 4 ? 2 * jt : jt + 4) {
    if (smem_bytes(d, b, m, jt) > (size_t)kMaxSmem) break;
    const long long ctas = (long long)BH * ((b + jt - 1) / jt);
    const bool two = 2 * (smem_bytes(d, b, m, jt) + 1024) <= (size_t)228 * 1024;
    const long long cost = (ctas + num_sms - 1) / num_sms * (jt + 3) * (two ? 3 : 4);
    if (best == 0 || cost < least) {
      best = jt;
      least = cost;
    }
  }
  return best;
}
inline bool supported(int N, int d, int b, int m) {
  (void)N;
  return b <= 1024 && m <= 1024 && (size_t)m * ((size_t)b * (((d + 3) / 4) | 1)) <= (size_t)kMaxSmem / 16 &&
         smem_bytes(d, b, m, 1) <= (size_t)kMaxSmem;
}
// Whether AUTO takes this kernel.  Long heads leave room for a position or two beside K, and every CTA
// loads all of K: with many heads and many CTAs a head the generic kernels are faster then (96 heads of 768 = 32 x 24,
// two rounds: 355 against 473 us; 17 CTAs a head, 96 of 731 = 43 x 17, one round: 1.4 x), with few heads this one is (2 heads of
// 600 = 25 x 24: 28 against 67 us), and with up to six CTAs a head (192 of 225 = 75 x 3, one round: 133 against 221 us; 96 of
// 396 = 33 x 12 in six: 0.80 of the generic kernels' time; seven and eight CTAs a head: 0.83 to 1.12).
inline bool chosen(int N, int d, int b, int m, int BH, int num_sms) {
  if (!supported(N, d, b, m)) return false;
  const int jt = positions_per_cta(d, b, m, BH, num_sms), ctas = (b + jt - 1) / jt;
  return smem_bytes(d, b, m, b < 4 ? b : 4) <= (size_t)kMaxSmem || ctas <= 6 || (long long)BH * ctas <= 2LL * num_sms;
}

__device__ __forceinline__ void fma4(float4& acc, float p, const float4& x) {
  const float2 p2 = make_float2(p, p);
  const float2 lo = ffma2(p2, make_float2(x.x, x.y), make_float2(acc.x, acc.y));
  const float2 hi = ffma2(p2, make_float2(x.z, x.w), make_float2(acc.z, acc.w));
  acc = make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ void dot4(float2& acc, const float4& a, const float4& x) {
  acc = ffma2(make_float2(a.x, a.y), make_float2(x.x, x.y), acc);
  acc = ffma2(make_float2(a.z, a.w), make_float2(x.z, x.w), acc);
}
__device__ __forceinline__ float elem(const float4& v, int i) { return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w)); }
// Four elements from column `col` of a row of d (zeros past its end).  Rows that are no whole number of
// 16-byte units are read element by element, out of line.
template <typename TIn>
__device__ __noinline__ float4 load4_ragged(const TIn* p, int left) {
  return make_float4(ld_as_float(p), left > 1 ? ld_as_float(p + 1) : 0.f, left > 2 ? ld_as_float(p + 2) : 0.f,
                     left > 3 ? ld_as_float(p + 3) : 0.f);
}
template <bool WHOLE, typename TIn>
__device__ __forceinline__ float4 load4(const TIn* p, int col, int d) {
  if (!WHOLE && d % 4 != 0) return load4_ragged(p + col, d - col);
  if constexpr (sizeof(TIn) == 4) {
    return *reinterpret_cast<const float4*>(p + col);
  } else {
    const uint2 u = *reinterpret_cast<const uint2*>(p + col);
    const TIn* e = reinterpret_cast<const TIn*>(&u);
    return make_float4(ld_as_float(e), ld_as_float(e + 1), ld_as_float(e + 2), ld_as_float(e + 3));
  }
}
// Four elements to shared memory: asynchronously where rows are whole 16-byte units of fp32 (nothing waits in registers, and all of a
// thread's copies are in flight at once: 12 heads of 384 = 16 x 24 8.4 -> 8.1 us, 8 of 200 = 10 x 20, two rounds 13.5 -> 12.9, 96 of 256, three 45.1 -> 43.9).
template <bool WHOLE, typename TIn>
__device__ __forceinline__ void copy4(float4* to, const TIn* p, int col, int d) {
  if constexpr (WHOLE && sizeof(TIn) == 4) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(p + col) : "memory");
  } else {
    *to = load4<WHOLE>(p, col, d);
  }
}
template <typename TIn>
__device__ __noinline__ void store4_ragged(TIn* p, int left, float4 v) {
#pragma unroll
  for (int c = 0; c < 4; ++c)
    if (c < left) st_from_float(p + c, elem(v, c));
}
template <bool WHOLE, typename TIn>
__device__ __forceinline__ void store4(TIn* p, int col, int d, const float4& v) {
  if (WHOLE || (d % 4 == 0 && sizeof(TIn) == 4)) *reinterpret_cast<float4*>(p + col) = v;
  else store4_ragged(p + col, d - col, v);
}
// Over the eight lanes that share a row.
__device__ __forceinline__ float row_max(float v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float row_sum(float v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// x / n for 0 <= x < 2^22, inv = 1.f / n.
__device__ __forceinline__ int divide(int x, float inv) { return __float2int_rd(((float)x + 0.5f) * inv); }

// Scores and softmax of R rows against up to 8 TC columns by a group of 8 DS lanes: a lane has TC columns
// (c, c + 8, ..) and a DS-th of the depth; the depth is summed over the group, which then splits the
// rows.  rows[r], cols[c]: addresses; logit(r, column, dot) scales and masks; the weights of the first n_rows
// rows go to w + r * wp, and done(r, max, sum of exp(z - max), sum of weight * logit) keeps the rest.
template <int R, int DS, int TC, typename Logit, typename Done>
__device__ __forceinline__ void score_rows(const float4* (&rows)[R], const float4* (&cols)[TC], int d4, int lane, int n_cols,
                                           float* w, int wp, Logit logit, Done done, int n_rows) {
  static_assert(R == 1 || R == DS || R == 2 * DS, "rows are split over the depth parts");
  const int c0 = lane & 7, part = (lane >> 3) & (DS - 1);
  float2 acc[R][TC];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < TC; ++c) acc[r][c] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int u = part; u < d4; u += DS) {
    float4 x[TC];
#pragma unroll
    for (int c = 0; c < TC; ++c) x[c] = cols[c][u];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float4 v = rows[r][u];
#pragma unroll
      for (int c = 0; c < TC; ++c) dot4(acc[r][c], v, x[c]);
    }
  }
  constexpr int RL = R >= DS ? R / DS : 1;      // rows a lane keeps
  float z[RL][TC];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < TC; ++c) {
      float v = acc[r][c].x + acc[r][c].y;
#pragma unroll
      for (int o = 8; o < 8 * DS; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (R == 1 || r / RL == part) z[r % RL][c] = v;
    }
#pragma unroll
  for (int q = 0; q < RL; ++q) {
    const int r = R == 1 ? 0 : part * RL + q;
    float zmax = -INFINITY;
#pragma unroll
    for (int c = 0; c < TC; ++c) {
      z[q][c] = c0 + 8 * c < n_cols ? logit(r, c0 + 8 * c, z[q][c]) : -INFINITY;
      zmax = fmaxf(zmax, z[q][c]);
    }
    zmax = row_max(zmax);
    float s = 0.f, sz = 0.f;
#pragma unroll
    for (int c = 0; c < TC; ++c) {
      const bool valid = z[q][c] > -INFINITY;
      const float p = valid ? expf(z[q][c] - zmax) : 0.f;
      s += p;
      if (valid) sz = fmaf(p, z[q][c], sz);          // 0 log 0 = 0 for masked keys
      z[q][c] = p;
    }
    s = row_sum(s);
    sz = row_sum(sz);
    const float inv = 1.f / s;
    if (R > 1 || part == 0) {
#pragma unroll
      for (int c = 0; c < TC; ++c)
        if (r < n_rows && c0 + 8 * c < n_cols) w[r * wp + c0 + 8 * c] = z[q][c] * inv;
      if (c0 == 0) done(r, zmax, s, sz * inv);
    }
  }
}

// TR: positions of a register tile (1, 2 or 4).  CB, CM: up to 8 CB keys and 8 CM blocks; 0: any numbers.
// WHOLE: rows are whole 16-byte units.
template <typename TIn, int TR, int CB, int CM, bool WHOLE>
__global__ void __launch_bounds__(kThreads, 2)
monarch_fused_f32(const TIn* __restrict__ Q, const TIn* __restrict__ K, const TIn* __restrict__ V,
                  TIn* __restrict__ Y, int N, int d, int b, int m, int T_steps, float scale,
                  int n_valid, int H, int JT, float* __restrict__ row_lse, int* clear) {
  constexpr int TC = TR == 1 ? 1 : 2;        // (any sizes) keys of a score tile (R), rows and blocks of one (L)
  constexpr int TL = TR == 1 ? 1 : 4;        // rows of a second product's tile in the L half-step
  constexpr int DS = TR == 1 ? 4 : 2, kGroups = kThreads / (8 * DS);      // lanes of a score group: 8 DS
  extern __shared__ __align__(16) float4 sm[];
  generic::grid_dependency_sync();
  clear_status(clear);
  const int h = blockIdx.y, j0 = blockIdx.x * JT, nj = min(JT, b - j0);
  const int tid = threadIdx.x;
  const Layout ly = layout(d, b, m, JT);
  const int d4 = ly.d4, pu = ly.pu, bu = ly.bu, ju = ly.ju, su = ly.su;
  float4 *sK = sm, *sQ = sm + ly.Q, *sA = sm + ly.A;
  float* cL = reinterpret_cast<float*>(sm + ly.C);          // [k * JT + jj]
  float* cR = cL + (JT * m + 3) / 4 * 4;                    // [k * JT + jj]
  float* sW = reinterpret_cast<float*>(sm + ly.S);          // weights, row pitch 4 su
  const int wp = 4 * su;

  // the head's first row, and from row to row
  const size_t base = H == 0 ? (size_t)h * N * d : ((size_t)(h / H) * N * H + h % H) * d;
  const int rs = H == 0 ? d : H * d;
  Q += base;
  K += base;
  V += base;
  Y += base;
  if (row_lse != nullptr) row_lse += (size_t)h * N;
  const float inv_d4 = 1.f / d4;

  // ---- loads; V is asked for into L2
  const float inv_b = 1.f / b, inv_nj = 1.f / nj;
#pragma unroll 8
  for (int e = tid; e < N * d4; e += kThreads) {
    const int n = divide(e, inv_d4), u = e - n * d4, k = divide(n, inv_b), i = n - k * b;
    copy4<WHOLE>(&sK[k * bu + i * pu + u], K + (size_t)n * rs, 4 * u, d);
  }
#pragma unroll 4
  for (int e = tid; e < nj * m * d4; e += kThreads) {
    const int r = divide(e, inv_d4), u = e - r * d4, l = divide(r, inv_nj), jj = r - l * nj;
    copy4<WHOLE>(&sQ[l * ju + jj * pu + u], Q + (size_t)(l * b + j0 + jj) * rs, 4 * u, d);
  }
  for (int n = tid; n < N; n += kThreads) {
    const char* p = reinterpret_cast<const char*>(V + (size_t)n * rs);
    for (int o = 0; o < d * (int)sizeof(TIn); o += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + o));
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();

  // Softmax over the first `cols` of `rows` rows of logits, eight lanes a row: to weights;
  // done(row, max, sum of exp(z - max), sum of weight * logit).
  auto softmax = [&](int rows, int cols, auto done) {
    for (int r0 = 0; r0 < rows; r0 += kThreads / 8) {
      const int r = r0 + (tid >> 3), g = tid & 7;
      const bool on = r < rows;
      float* w = sW + (on ? r : 0) * wp;
      float zmax = -INFINITY;
      if (on)
        for (int i = g; i < cols; i += 8) zmax = fmaxf(zmax, w[i]);
      zmax = row_max(zmax);
      float s = 0.f, sz = 0.f;
      if (on)
        for (int i = g; i < cols; i += 8) {
          const float z = w[i];
          const bool valid = z > -INFINITY;
          const float p = valid ? expf(z - zmax) : 0.f;
          w[i] = p;
          s += p;
          if (valid) sz = fmaf(p, z, sz);
        }
      s = row_sum(s);
      sz = row_sum(sz);
      const float inv = 1.f / s;
      if (on)
        for (int i = g; i < cols; i += 8) w[i] *= inv;
      if (on && g == 0) done(r, zmax, s, sz * inv);
    }
  };

  const int JG = (nj + TR - 1) / TR, LG = (m + TL - 1) / TL;
  const float inv_JG = 1.f / JG, inv_LG = 1.f / LG, inv_m = 1.f / m;
  for (int step = 1; step <= T_steps; ++step) {
    const bool first = step == 1, last = step == T_steps;
    // ---------------------------------------------------------------- R half-step (Eq. 7, 9, 10)
    // Z_R[i] = scale * <alpha_R(k,j), K(k,i)> / c_R(k,j); R = softmax_i Z_R;
    // alpha_L(j,k) = sum_i R[i] K(k,i); c_L(j,k) = sum_i R log R; (last) y(j,k) = sum_i R[i] V(k,i)
    const float4* a = first ? sQ : sA;         // L^(0) = identity: alpha_R = the Q row (k, j), c_R = 1
    auto r_scale = [&](int r) {
      if (first) return scale;
      const float c = cR[r];
      return scale * (c > 1e-30f ? 1.f / c : 0.f);         // c_R underflow: uniform row (Z_R = 0)
    };
    if constexpr (CB > 0) {
      const int groups = m * JG;
      for (int g0 = 0; g0 < groups; g0 += kGroups) {
        const bool on = g0 + tid / (8 * DS) < groups;
        const int gi = on ? g0 + tid / (8 * DS) : groups - 1;      // (every lane takes part in the shuffles)
        const int k = divide(gi, inv_JG), jr = (gi - k * JG) * TR;
        const float4 *rows[TR], *cols[CB];
        float f[TR];
#pragma unroll
        for (int r = 0; r < TR; ++r) {
          rows[r] = a + k * ju + min(jr + r, nj - 1) * pu;
          f[r] = r_scale(k * JT + min(jr + r, nj - 1));
        }
#pragma unroll
        for (int c = 0; c < CB; ++c) cols[c] = sK + k * bu + min((tid & 7) + 8 * c, b - 1) * pu;
        score_rows<TR, DS, CB>(
            rows, cols, d4, tid, on ? b : 0, sW + (k * JT + jr) * wp, wp,
            [&](int r, int i, float dot) {
              float fr = f[0];
#pragma unroll
              for (int e = 1; e < TR; ++e) fr = r == e ? f[e] : fr;
              // padding mask (App. C.3, post-padding): key columns b k + i >= n_valid get -inf
              return k * b + i < n_valid ? dot * fr : -INFINITY;
            },
            [&](int r, float zmax, float sum, float sz) {
              if (!on || jr + r >= nj) return;
              cL[k * JT + jr + r] = sz - (zmax + logf(sum));
            },
            nj - jr);
      }
      __syncthreads();
    } else {
      const int IG = (b + TC - 1) / TC, items = m * JG * IG;
      for (int it = tid; it < items; it += kThreads) {
        const int q = it / IG, i0 = (it - q * IG) * TC, k = q / JG, jr = (q - k * JG) * TR;
        const float4 *ap[TR], *kp[TC];
        float2 acc[TR][TC];
#pragma unroll
        for (int r = 0; r < TR; ++r) ap[r] = a + k * ju + min(jr + r, nj - 1) * pu;
#pragma unroll
        for (int c = 0; c < TC; ++c) kp[c] = sK + k * bu + min(i0 + c, b - 1) * pu;
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
          for (int c = 0; c < TC; ++c) acc[r][c] = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int u = 0; u < d4; ++u) {
          float4 x[TC];
#pragma unroll
          for (int c = 0; c < TC; ++c) x[c] = kp[c][u];
#pragma unroll
          for (int r = 0; r < TR; ++r) {
            const float4 v = ap[r][u];
#pragma unroll
            for (int c = 0; c < TC; ++c) dot4(acc[r][c], v, x[c]);
          }
        }
#pragma unroll
        for (int r = 0; r < TR; ++r) {
          if (jr + r >= nj) continue;
          const float f = r_scale(k * JT + jr + r);
#pragma unroll
          for (int c = 0; c < TC; ++c)
            if (i0 + c < b)
              sW[(k * JT + jr + r) * wp + i0 + c] = k * b + i0 + c < n_valid ? (acc[r][c].x + acc[r][c].y) * f : -INFINITY;
        }
      }
      __syncthreads();
      softmax(m * JT, b, [&](int r, float zmax, float s, float sz) { cL[r] = sz - (zmax + logf(s)); });
      __syncthreads();
    }
    // second products: TR positions x 4 columns; row(k, i, u): four columns from 4 u of row (k, i) of K or V
    auto apply = [&](auto row, auto put) {
      const int items = m * JG * d4;
      for (int it = tid; it < items; it += kThreads) {
        const int q = divide(it, inv_d4), u = it - q * d4, k = divide(q, inv_JG), jr = (q - k * JG) * TR;
        const float* w[TR];
        float4 acc[TR];
#pragma unroll
        for (int r = 0; r < TR; ++r) {
          w[r] = sW + (k * JT + min(jr + r, nj - 1)) * wp;
          acc[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        int i = 0;
#pragma unroll 2
        for (; i + 4 <= b; i += 4) {
          float4 x[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) x[e] = row(k, i + e, u);
#pragma unroll
          for (int r = 0; r < TR; ++r) {
            const float4 p = *reinterpret_cast<const float4*>(w[r] + i);
            fma4(acc[r], p.x, x[0]);
            fma4(acc[r], p.y, x[1]);
            fma4(acc[r], p.z, x[2]);
            fma4(acc[r], p.w, x[3]);
          }
        }
        for (; i < b; ++i) {
          const float4 x = row(k, i, u);
#pragma unroll
          for (int r = 0; r < TR; ++r) fma4(acc[r], w[r][i], x);
        }
#pragma unroll
        for (int r = 0; r < TR; ++r)
          if (jr + r < nj) put(k, jr + r, u, acc[r]);
      }
    };
    apply([&](int k, int i, int u) { return sK[k * bu + i * pu + u]; },
          [&](int k, int jj, int u, const float4& v) { sA[k * ju + jj * pu + u] = v; });
    __syncthreads();
    if (last) {      // y over the rows of K
      apply([&](int k, int i, int u) { return load4<WHOLE>(V + (size_t)(k * b + i) * rs, 4 * u, d); },
            [&](int k, int jj, int u, const float4& v) { sK[k * bu + jj * pu + u] = v; });
      __syncthreads();
    }

    // ---------------------------------------------------------------- L half-step (Eq. 8, 9 / Eq. 4)
    // Z_L[k] = scale * <Q(l,j), alpha_L(j,k)> - c_L(j,k); L = softmax_k Z_L
    auto row_done = [&](int r, float zmax, float s) {
      // log-sum-exp of row b l + j: summed over a head's rows it is the objective (Eq. 6)
      const int jj = r / m, l = r - jj * m;
      if (last && row_lse != nullptr) row_lse[l * b + j0 + jj] = zmax + logf(s);
    };
    if constexpr (CM > 0) {
      const int RG = (m + TR - 1) / TR, groups = nj * RG;
      const float inv_RG = 1.f / RG;
      for (int g0 = 0; g0 < groups; g0 += kGroups) {
        const bool on = g0 + tid / (8 * DS) < groups;
        const int gi = on ? g0 + tid / (8 * DS) : groups - 1;
        const int jj = divide(gi, inv_RG), l0 = (gi - jj * RG) * TR;
        const float4 *rows[TR], *cols[CM];
#pragma unroll
        for (int r = 0; r < TR; ++r) rows[r] = sQ + min(l0 + r, m - 1) * ju + jj * pu;
#pragma unroll
        for (int c = 0; c < CM; ++c) cols[c] = sA + min((tid & 7) + 8 * c, m - 1) * ju + jj * pu;
        score_rows<TR, DS, CM>(
            rows, cols, d4, tid, on ? m : 0, sW + (jj * m + l0) * wp, wp,
            [&](int, int k, float dot) { return dot * scale - cL[k * JT + jj]; },
            [&](int r, float zmax, float sum, float) {
              if (!on || l0 + r >= m) return;
              row_done(jj * m + l0 + r, zmax, sum);
            },
            m - l0);
      }
      __syncthreads();
    } else {
      const int G = (m + TC - 1) / TC, items = nj * G * G;
      for (int it = tid; it < items; it += kThreads) {
        const int q = it / G, k0 = (it - q * G) * TC, jj = q / G, l0 = (q - jj * G) * TC;
        const float4 *qp[TC], *ap[TC];
        float2 acc[TC][TC];
#pragma unroll
        for (int r = 0; r < TC; ++r) {
          qp[r] = sQ + min(l0 + r, m - 1) * ju + jj * pu;
          ap[r] = sA + min(k0 + r, m - 1) * ju + jj * pu;
#pragma unroll
          for (int c = 0; c < TC; ++c) acc[r][c] = make_float2(0.f, 0.f);
        }
#pragma unroll 4
        for (int u = 0; u < d4; ++u) {
          float4 x[TC];
#pragma unroll
          for (int c = 0; c < TC; ++c) x[c] = ap[c][u];
#pragma unroll
          for (int r = 0; r < TC; ++r) {
            const float4 v = qp[r][u];
#pragma unroll
            for (int c = 0; c < TC; ++c) dot4(acc[r][c], v, x[c]);
          }
        }
#pragma unroll
        for (int r = 0; r < TC; ++r)
#pragma unroll
          for (int c = 0; c < TC; ++c)
            if (l0 + r < m && k0 + c < m)
              sW[(jj * m + l0 + r) * wp + k0 + c] = (acc[r][c].x + acc[r][c].y) * scale - cL[(k0 + c) * JT + jj];
      }
      __syncthreads();
      softmax(nj * m, m, [&](int r, float zmax, float s, float) { row_done(r, zmax, s); });
      __syncthreads();
    }
    const int items = nj * LG * d4;
    for (int it = tid; it < items; it += kThreads) {
      const int q = divide(it, inv_d4), u = it - q * d4, jj = divide(q, inv_LG), r0 = (q - jj * LG) * TL;
      const float* w = sW + jj * m * wp;
      float4 acc[TL];
#pragma unroll
      for (int r = 0; r < TL; ++r) acc[r] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (last) {
        // Y(l,j) = sum_k L[l,k] y(k,j), rows l = r0 ..
        const float4* y = sK + jj * pu + u;
        int k = 0;
#pragma unroll 2
        for (; k + 4 <= m; k += 4) {
          float4 x[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) x[e] = y[(k + e) * bu];
#pragma unroll
          for (int r = 0; r < TL; ++r) {
            const float4 p = *reinterpret_cast<const float4*>(w + min(r0 + r, m - 1) * wp + k);
            fma4(acc[r], p.x, x[0]);
            fma4(acc[r], p.y, x[1]);
            fma4(acc[r], p.z, x[2]);
            fma4(acc[r], p.w, x[3]);
          }
        }
        for (; k < m; ++k) {
          const float4 x = y[k * bu];
#pragma unroll
          for (int r = 0; r < TL; ++r) fma4(acc[r], w[min(r0 + r, m - 1) * wp + k], x);
        }
#pragma unroll
        for (int r = 0; r < TL; ++r)
          if (r0 + r < m) store4<WHOLE>(Y + (size_t)((r0 + r) * b + j0 + jj) * rs, 4 * u, d, acc[r]);
      } else {
        // alpha_R(k,j) = sum_l L[l,k] Q(l,j), c_R(k,j) = sum_l L[l,k], blocks k = r0 ..
        const float4* x = sQ + jj * pu + u;
#pragma unroll 4
        for (int l = 0; l < m; ++l) {
          const float4 v = x[l * ju];
          if constexpr (TL == 4) {
            const float4 p = *reinterpret_cast<const float4*>(w + l * wp + r0);
            fma4(acc[0], p.x, v);
            fma4(acc[1], p.y, v);
            fma4(acc[2], p.z, v);
            fma4(acc[3], p.w, v);
          } else {
            fma4(acc[0], w[l * wp + r0], v);
          }
        }
#pragma unroll
        for (int r = 0; r < TL; ++r)
          if (r0 + r < m) sA[(r0 + r) * ju + jj * pu + u] = acc[r];
      }
    }
    if (!last) {
      // c_R, four lanes a column
      for (int c0 = 0; c0 < nj * m; c0 += kThreads / 4) {
        const int c = c0 + (tid >> 2), jj = divide(min(c, nj * m - 1), inv_m), k = min(c, nj * m - 1) - jj * m;
        float sum = 0.f;
        for (int l = tid & 3; l < m; l += 4) sum += sW[(jj * m + l) * wp + k];
        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
        sum += __shfl_xor_sync(0xffffffffu, sum, 2);
        if (c < nj * m && (tid & 3) == 0) cR[k * JT + jj] = sum;
      }
      __syncthreads();
    }
  }
}

int launch(const void* Q, const void* K, const void* V, void* Y, int BH, int N, int d, int b, int m,
           int T, int dtype, float scale, int n_valid, int H, float* lse, int* clear, cudaStream_t st);

#ifdef MA_TU_FUSED_F32
template <typename TIn>
inline int launch_t(const void* Q, const void* K, const void* V, void* Y, int BH, int N, int d, int b,
                    int m, int T, float scale, int n_valid, int H, float* lse, int* clear, cudaStream_t st) {
  static int sms[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 7;
  if (sms[dev] == 0 && cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 7;
  const int JT = positions_per_cta(d, b, m, BH, sms[dev]);
  if (JT < 1 || BH > 65535) return 4;
  // (the kernels with whole score rows in a group of lanes are for fp32 inputs, the only ones this path
  // is chosen for, up to 32 keys and blocks, with the
  // reads of ragged rows left out where there are none: instruction fetch counts, a warp executes most of the
  // code once or twice)
  const int cb = b <= 16 ? 2 : (b <= 24 ? 3 : 4), cm = m <= 16 ? 2 : 4;
  const bool small = sizeof(TIn) == 4 && b <= 32 && m <= 32, whole = d % 4 == 0;
  auto pick = [&](auto tr) {
    constexpr int TR = decltype(tr)::value;
    if constexpr (sizeof(TIn) == 4) {
      if (small && !whole) return monarch_fused_f32<TIn, TR, 4, 4, false>;
      if (small && cm == 2)
        return cb == 2 ? monarch_fused_f32<TIn, TR, 2, 2, true> : (cb == 3 ? monarch_fused_f32<TIn, TR, 3, 2, true> : monarch_fused_f32<TIn, TR, 4, 2, true>);
      if (small)
        return cb == 2 ? monarch_fused_f32<TIn, TR, 2, 4, true> : (cb == 3 ? monarch_fused_f32<TIn, TR, 3, 4, true> : monarch_fused_f32<TIn, TR, 4, 4, true>);
    }
    return monarch_fused_f32<TIn, TR, 0, 0, false>;
  };
  auto kern = JT == 1 ? pick(std::integral_constant<int, 1>())
                      : (JT == 2 ? pick(std::integral_constant<int, 2>()) : pick(std::integral_constant<int, 4>()));
  const size_t smem = smem_bytes(d, b, m, JT);
  static bool prepared[64][3][8] = {};
  bool& ready = prepared[dev][JT < 4 ? JT - 1 : 2][!small ? 6 : (whole ? cb - 2 + 3 * (cm == 4) : 7)];
  if (!ready) {      // once per device: the kernel may use all of shared memory
    if (cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) !=
        cudaSuccess)
      return 7;
    ready = true;
  }
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((b + JT - 1) / JT, BH);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, (const TIn*)Q, (const TIn*)K, (const TIn*)V, (TIn*)Y, N, d, b, m, T,
                            scale, n_valid, H, JT, lse, clear) == cudaSuccess
             ? 0
             : 7;
}

int launch(const void* Q, const void* K, const void* V, void* Y, int BH, int N, int d, int b, int m,
           int T, int dtype, float scale, int n_valid, int H, float* lse, int* clear, cudaStream_t st) {
  if (dtype == 0) return launch_t<float>(Q, K, V, Y, BH, N, d, b, m, T, scale, n_valid, H, lse, clear, st);
  if (dtype == 1) return launch_t<__half>(Q, K, V, Y, BH, N, d, b, m, T, scale, n_valid, H, lse, clear, st);
  return launch_t<__nv_bfloat16>(Q, K, V, Y, BH, N, d, b, m, T, scale, n_valid, H, lse, clear, st);
}
#endif  // MA_TU_FUSED_F32

}  // namespace ffused
}  // namespace ma
