// Fused kernel for N = 1024 as 32 blocks of 32 (d = 64, f16/bf16): all T rounds of Eq. 7-10 and the
// Monarch multiply of Eq. 4 in ONE launch, the states alpha_L, alpha_R, y, c_L (Sec. 3 'Implementation')
// never leaving shared memory.
//
// A head of this size does not fit one SM (Q, K, V and a state are 128 KB each), so it is split by
// in-block position: within a head the whole recursion is independent across the position j (row
// (l, j) of the Monarch matrix is L[j,:,l] (x) R[:,j,:]; R[k,j,:], c_L[j,k], alpha_L[j,k,:],
// L[j,:,:], alpha_R[k,j,:], c_R[k,j], y[j,k,:] only ever read quantities with the same j, plus all
// of K and V and the 32 rows (l, j) of Q).  A CTA owns PJ = 16 (or 8) positions of one head: its rows of Q
// and ONE state tile stay in shared memory (alpha_R and alpha_L replace each other in place: an R tile
// reads the rows (k, .) it then overwrites, an L tile the rows (., j)).  No CTA exchanges anything with
// another; the CTAs of a head read the same K and V, once from HBM and then from L2.
//
// What bounds it: instruction issue and latency at four warps per scheduler (half of the issue slots are
// busy), then the last wave of CTAs.  K and V stream
// through ONE 4 KB slot per warp.  A warp owns 32 / (warps) key blocks of an R half-step; it reads a block
// into registers as the operand of the scores, at which point the slot is free and TMA brings the next
// block (K of the next, or V of this one in the last round) under the whole work on this one; the
// second product's operand, the block transposed, comes out of the same registers through movmatrix.  So
// K is read from shared memory (and converted from bf16) once per half-step, and the first block of the
// next round arrives under the L half-step.  With 16 positions a K fragment feeds two MMAs.
//
// The R half-step runs transposed, S^T[i,j] = <K(k,i), alpha_R(k,j)> with the positions as the MMA's N: the
// softmax over i is a reduction over accumulator rows (registers, then three shuffles), the weights reach
// the second product as its B operand through movmatrix, and alpha_L^T[v,j] leaves through transposing
// matrix stores.  In the L half-step a warp owns a position.  Contractions are mma.sync m16n8k16 in f16
// (bf16 inputs are converted in registers: exact for magnitudes in [6.1e-5, 65504], clamped beyond).
// Blocks of the Q and state tiles are an odd number of 128-byte lines apart, so that under the 128-byte
// swizzle eight rows are conflict-free both along a block and across blocks.  Reductions over the lanes of
// a column halve the number of values a lane carries at each step, which also leaves one division and one
// logarithm a lane instead of four.
//
// Batch 16, 12 heads, T = 2, bf16: 58 us (f16 54), against 79 (74) with K resident in shared memory, read
// again as the second product's operand, and 8 positions a CTA; 64 (60) before the halving reductions and
// Q converted once.  One head: 8 and 13 us (T = 1, 2).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "status_word.cuh"
#include "tensor_path.cuh"
#include "warp_mma.cuh"

namespace ma {
namespace jsplit {

using tensor::mbar_expect_tx;
using tensor::mbar_init;
using tensor::mbar_wait;
using tensor::tma_load_2d;
using warpmma::Mma;
using warpmma::ex2;
using warpmma::kLog2e;
using warpmma::ldsm_x4;
using warpmma::ldsm_x4_trans;
using warpmma::mma;
using warpmma::put_pair;
using warpmma::row_pair;
using warpmma::lg2;
using warpmma::movm_trans;
using warpmma::quad_max;
using warpmma::scatter_reduce;

constexpr int kN = 1024, kB = 32, kM = 32, kD = 64;
constexpr int kSlot = kB * 128;                          // a block of K or V

// Shared memory for PJ positions per CTA and W warps per position.
template <int PJ, int W>
struct Lay {
  static constexpr int kWarps = PJ * W, kThreads = 32 * kWarps;
  static constexpr int kBlk = (PJ + 1) * 128;            // the PJ rows (k, .) of the Q / state tile and a line of padding
  static constexpr int Q = kWarps * kSlot;               // after the slots, one per warp
  static constexpr int S = Q + kM * kBlk;                // state, [k][jj]
  static constexpr int P = S + kM * kBlk;                // W = 2: weights exchange, per position [32 l][32 k] f16
  static constexpr int X = P + (W - 1) * PJ * 2048;      // W = 2: column maxima, per position [2][32]
  static constexpr int C = X + (W - 1) * PJ * 256;       // -c_L log2 e, [jj][kCp]: conflict-free along k and along jj
  static constexpr int kCp = kM + 2;
  static constexpr int Bar = C + kCp * PJ * 4;
  static constexpr int kSmem = Bar + kWarps * 8 + 1024;  // + alignment slack
  static_assert(Q % 1024 == 0 && S % 1024 == 0 && kSmem <= 227 * 1024, "shared memory layout");
};

__device__ __forceinline__ float col_max(float v) {   // over the 8 row groups (lanes with equal t)
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 4));
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 8));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 16));
}
__device__ __forceinline__ void stsm_x4(uint32_t saddr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(saddr), "r"(r0),
               "r"(r1), "r"(r2), "r"(r3)
               : "memory");
}
__device__ __forceinline__ void stsm_x4_trans(uint32_t saddr, uint32_t r0, uint32_t r1, uint32_t r2,
                                              uint32_t r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(saddr),
               "r"(r0), "r"(r1), "r"(r2), "r"(r3)
               : "memory");
}
// The 128-byte swizzle TMA applies: the 16-byte chunk index is XORed with bits 7..9 of the row's address.
__device__ __forceinline__ uint32_t swz(uint32_t row, int c) { return row + ((c ^ ((row >> 7) & 7)) << 4); }

// NEG: a negative softmax scale, passed as its magnitude, with -K in place of K: the same weights in both half-steps
// (alpha_L changes its sign with K).
template <typename TIn, int PJ, int W, bool NEG>
__global__ void __launch_bounds__(Lay<PJ, W>::kThreads, 1)
monarch_jsplit32(const __grid_constant__ CUtensorMap tmQ,    // Q as rows of d, box of PJ rows
                 const __grid_constant__ CUtensorMap tmK,    // K, box of 32 rows
                 const __grid_constant__ CUtensorMap tmV,    // V, box of 32 rows
                 TIn* __restrict__ Y, int T_steps, float scale, int* status, int* clear, int H) {
  typedef Mma<__half> M;
  using L = Lay<PJ, W>;
  constexpr int NW = L::kWarps, NB = kM / NW;   // key blocks of a warp: warp, warp + NW, ..
  constexpr int NT = PJ / 8;                    // 8-position tiles
  extern __shared__ uint8_t smem_raw[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  uint8_t* smem = align_smem<1024>(smem_raw);
  const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(smem);
  float* sCL = reinterpret_cast<float*>(smem + L::C);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::Bar);      // by warp: what it asked for has landed in its slot
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, t = lane & 3;
  const int jc = blockIdx.x * PJ;               // first position
  // H = 0: tensors [batch][heads][N][d], a head is 1024 rows of the maps; H = heads: tensors
  // [batch][N][heads][d], the maps see rows of heads * 64 columns (d = 64) and a head is a column offset
  const int hb = H ? (int)blockIdx.y / H : (int)blockIdx.y;
  const int x0 = H ? ((int)blockIdx.y - hb * H) * kD : 0;
  const int row0 = hb * kN;
  const float fl = scale * kLog2e;
  if (lane == 0) mbar_init(&bars[warp], 1);
  tensor::fence_barrier_init();
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  clear_status(clear);

  // rows of the tiles: Q (l, jj), state (k, jj)
  auto rq = [&](int l, int jj) { return s0 + L::Q + l * L::kBlk + jj * 128; };
  auto rs = [&](int k, int jj) { return s0 + L::S + k * L::kBlk + jj * 128; };
  // y(k, jj) lies in the slot of the warp that owns block k; rows are turned by k so that eight blocks
  // are conflict-free
  auto ry = [&](int k, int jj) { return s0 + (k % NW) * kSlot + ((k / NW) * PJ + ((jj + k) & (PJ - 1))) * 128; };
  const uint32_t slot = s0 + warp * kSlot;
  uint32_t par = 0;
  constexpr uint32_t kDead = 1u << 31;          // in `par`: a wait ran out; no further ones and no further requests
  auto request = [&](const CUtensorMap* tm, int k) {      // block k of K or V into the slot
    tensor::fence_proxy_async();
    __syncwarp();
    if (lane == 0 && !(par & kDead)) {
      mbar_expect_tx(&bars[warp], kSlot);
      tma_load_2d(smem + warp * kSlot, tm, &bars[warp], x0, row0 + k * kB);
    }
  };
  auto landed = [&]() {
    if (!(par & kDead) && !mbar_wait(&bars[warp], par)) {
      par |= kDead;
      tensor::report_timeout(status, 1);
    }
    par ^= 1;
    __syncwarp();
  };
  if (lane == 0) {
    mbar_expect_tx(&bars[warp], kSlot + NB * PJ * 128);
    tma_load_2d(smem + warp * kSlot, &tmK, &bars[warp], x0, row0 + warp * kB);
#pragma unroll
    for (int u = 0; u < NB; ++u)
      tma_load_2d(smem + L::Q + (warp + u * NW) * L::kBlk, &tmQ, &bars[warp], x0, row0 + (warp + u * NW) * kB + jc);
  }
  // bf16 -> f16 of a fragment in registers (a no-op for f16 inputs)
  auto convert_frag = [&](uint32_t* a) {
    if (!Mma<TIn>::is_f16) {
      uint4 v = warpmma::to_f16x8(make_uint4(a[0], a[1], a[2], a[3]), (const TIn*)nullptr);
      a[0] = v.x; a[1] = v.y; a[2] = v.z; a[3] = v.w;
    }
  };

  for (int step = 1; step <= T_steps; ++step) {
    const bool first = step == 1, last = step == T_steps;
    // ================================================================ R half-step (Eq. 7, 9, 10)
    // block k: S^T[i,j] = <K(k,i), alpha_R(k,j)> (alpha_R arrives divided by c_R), softmax over i,
    // alpha_L(k,j) = sum_i R[j,i] K(k,i), c_L(k,j) = sum_i R log R, (last) y(k,j) = sum_i R[j,i] V(k,i)
    uint32_t yk[NB][NT][4][2];                  // y of the warp's blocks, 16-bit
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int k = warp + u * NW;
      landed();
      if (first && u == 0 && !Mma<TIn>::is_f16) {        // the warp's rows of Q, in place
#pragma unroll
        for (int q = 0; q < NB * PJ / 4; ++q) {
          uint4* c = reinterpret_cast<uint4*>(smem + L::Q + (warp + q / (PJ / 4) * NW) * L::kBlk + q % (PJ / 4) * 512 + lane * 16);
          *c = warpmma::to_f16x8(*c, (const TIn*)nullptr);
        }
        __syncwarp();
      }
      uint32_t kf[2][4][4];                     // K(k, .) as A operand: [16 rows i][16 columns v]
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          ldsm_x4(kf[mt][ks], swz(slot + (16 * mt + (lane & 15)) * 128, 2 * ks + (lane >> 4)));
          convert_frag(kf[mt][ks]);
          if (NEG) {
#pragma unroll
            for (int i = 0; i < 4; ++i) kf[mt][ks][i] ^= 0x80008000u;
          }
        }
      // the slot is free: the next block comes under the work on this one
      if (last) request(&tmV, k);
      else request(&tmK, u + 1 < NB ? k + NW : warp);
      uint32_t pb[NT][2][2];                    // the weights P^T[i, j] as the second product's B operand
      float inv[NT][2], red[4 * NT], mxs[2 * NT];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        float s[2][4];
        const uint32_t row = first ? rq(k, 8 * nt + (lane & 7)) : rs(k, 8 * nt + (lane & 7));
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          uint32_t bq[4];                       // alpha_R rows (k, j) (L^(0) = identity: Q rows in the first round)
          ldsm_x4(bq, swz(row, (lane >> 3) + 4 * half));
#pragma unroll
          for (int k2 = 0; k2 < 2; ++k2)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) mma<__half>(half + k2 == 0, s[mt], kf[mt][2 * half + k2], bq + 2 * k2);
        }
        // column j = 8 nt + 2 t + e holds rows i = 16 mt + g (+ 8): softmax over i
        float2 mx, sum = both(0.f), sz = both(0.f);        // of the lane's two columns
        mx.x = col_max(fmaxf(fmaxf(s[0][0], s[0][2]), fmaxf(s[1][0], s[1][2])) * fl);
        mx.y = col_max(fmaxf(fmaxf(s[0][1], s[0][3]), fmaxf(s[1][1], s[1][3])) * fl);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {
            const float2 x = row_pair(s[mt], hh), z = ffma2(x, both(fl), make_float2(-mx.x, -mx.y));
            const float2 p = make_float2(ex2(z.x), ex2(z.y));
            sum = mt + hh ? fadd2(sum, p) : p;
            sz = mt + hh ? ffma2(p, x, sz) : fmul2(p, x);
            put_pair(s[mt], hh, p);
          }
        mxs[2 * nt] = mx.x;
        mxs[2 * nt + 1] = mx.y;
        red[4 * nt] = sum.x;
        red[4 * nt + 1] = sz.x;
        red[4 * nt + 2] = sum.y;
        red[4 * nt + 3] = sz.y;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
          pb[nt][mt][0] = movm_trans(M::pack(s[mt][0], s[mt][1]));
          pb[nt][mt][1] = movm_trans(M::pack(s[mt][2], s[mt][3]));
        }
      }
      {
        // a lane ends up with sum or sum p s (lane bit kSz) of one column: one division and one logarithm
        // a lane, the reciprocals then go to all lanes
        constexpr int kSz = 8 / NT, kCol = NT == 2 ? 3 : 4;
        const float r = scatter_reduce<4 * NT, 16, 4>(red, lane, warpmma::Add());
        const float ri = 1.f / r;
#pragma unroll
        for (int q = 0; q < 2 * NT; ++q) inv[q >> 1][q & 1] = __shfl_sync(0xffffffffu, ri, (q << kCol) + t);
        const float so = __shfl_xor_sync(0xffffffffu, r, kSz), io = __shfl_xor_sync(0xffffffffu, ri, kSz);
        const int q = lane >> kCol;
        float mx = mxs[0];
#pragma unroll
        for (int i = 1; i < 2 * NT; ++i) mx = q == i ? mxs[i] : mx;
        // -c_L log2 e = max + log2 sum - sum R z (z = s fl), the addend of the L logits
        if ((lane & kSz) && (NT == 2 || !(lane & 4)))
          sCL[(8 * (q >> 1) + 2 * t + (q & 1)) * L::kCp + k] = mx + lg2(so) - r * fl * io;
      }
      __syncwarp();
      // alpha_L^T[v, j] = sum_i K(k,i)[v] P^T[i, j]: A = the block's fragments transposed; the rows (k, j)
      // go over the alpha_R rows they were formed from (transposing stores: memory row j receives
      // column j of the accumulator tile)
#pragma unroll
      for (int vp = 0; vp < 2; ++vp) {
        float o[NT][2][4];
#pragma unroll
        for (int v2 = 0; v2 < 2; ++v2)
#pragma unroll
          for (int is = 0; is < 2; ++is) {
            const uint32_t* f = kf[is][2 * vp + v2];
            const uint32_t a[4] = {movm_trans(f[0]), movm_trans(f[2]), movm_trans(f[1]), movm_trans(f[3])};
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) mma<__half>(is == 0, o[nt][v2], a, pb[nt][is]);
          }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          const float2 i2 = make_float2(inv[nt][0], inv[nt][1]);
          stsm_x4_trans(swz(rs(k, 8 * nt + (lane & 7)), 4 * vp + (lane >> 3)), M::pack(fmul2(row_pair(o[nt][0], 0), i2)),
                        M::pack(fmul2(row_pair(o[nt][0], 1), i2)), M::pack(fmul2(row_pair(o[nt][1], 0), i2)),
                        M::pack(fmul2(row_pair(o[nt][1], 1), i2)));
        }
      }
      if (last) {
        // y^T[v, j] = sum_i V(k,i)[v] P^T[i, j]
        landed();
#pragma unroll
        for (int vt = 0; vt < 4; ++vt) {
          float o[NT][4];
#pragma unroll
          for (int is = 0; is < 2; ++is) {
            uint32_t a[4];
            ldsm_x4_trans(a, swz(slot + (16 * is + (lane & 7) + 8 * (lane >> 4)) * 128, 2 * vt + ((lane >> 3) & 1)));
            convert_frag(a);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) mma<__half>(is == 0, o[nt], a, pb[nt][is]);
          }
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
            for (int hh = 0; hh < 2; ++hh)
              yk[u][nt][vt][hh] = M::pack(fmul2(row_pair(o[nt], hh), make_float2(inv[nt][0], inv[nt][1])));
          }
        }
        if (u + 1 < NB) request(&tmK, k + NW);
      }
    }
    if (last) {                                 // the slot has had its last block: y(k, .) of all of them
      __syncwarp();
#pragma unroll
      for (int u = 0; u < NB; ++u)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int vp = 0; vp < 2; ++vp)
            stsm_x4_trans(swz(ry(warp + u * NW, 8 * nt + (lane & 7)), 4 * vp + (lane >> 3)), yk[u][nt][2 * vp][0],
                          yk[u][nt][2 * vp][1], yk[u][nt][2 * vp + 1][0], yk[u][nt][2 * vp + 1][1]);
    }
    __syncthreads();

    // ================================================================ L half-step (Eq. 8, 9 / Eq. 4)
    // position jj: Z_L[l,k] = fl * <Q(l,j), alpha_L(k,j)> - c_L(k,j), softmax over k.  A warp has
    // LT tiles of 16 rows l
    {
      constexpr int LT = 2 / W;
      const int jj = warp / W, l0 = W == 2 ? 16 * (warp & 1) : 0;
      float c[4][2];
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) {
        const float2 v = *reinterpret_cast<const float2*>(sCL + jj * L::kCp + 8 * nt + 2 * t);
        c[nt][0] = v.x;
        c[nt][1] = v.y;
      }
      float s[LT][4][4], inv[LT][2], rsum[2 * LT];
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        uint32_t bf[2][4];
#pragma unroll
        for (int np = 0; np < 2; ++np)
          ldsm_x4(bf[np], swz(rs(16 * np + (lane & 7) + 8 * (lane >> 4), jj), 2 * ks + ((lane >> 3) & 1)));
#pragma unroll
        for (int lt = 0; lt < LT; ++lt) {
          uint32_t a[4];
          ldsm_x4(a, swz(rq(l0 + 16 * lt + (lane & 15), jj), 2 * ks + (lane >> 4)));
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) mma<__half>(ks == 0, s[lt][nt], a, bf[nt >> 1] + 2 * (nt & 1));
        }
      }
#pragma unroll
      for (int lt = 0; lt < LT; ++lt)
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          float mx = -INFINITY;
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) {
            const float2 z = ffma2(row_pair(s[lt][nt], hh), both(fl), make_float2(c[nt][0], c[nt][1]));
            put_pair(s[lt][nt], hh, z);
            mx = fmaxf(mx, fmaxf(z.x, z.y));
          }
          mx = quad_max(mx);
          float2 sum = both(0.f);
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) {
            const float2 z = fadd2(row_pair(s[lt][nt], hh), both(-mx));
            const float2 p = make_float2(ex2(z.x), ex2(z.y));
            put_pair(s[lt][nt], hh, p);
            sum = nt ? fadd2(sum, p) : p;
          }
          rsum[2 * lt + hh] = sum.x + sum.y;
        }
      const float ri = 1.f / scatter_reduce<2 * LT, 2, 1>(rsum, lane, warpmma::Add());
#pragma unroll
      for (int i = 0; i < 2 * LT; ++i) inv[i >> 1][i & 1] = __shfl_sync(0xffffffffu, ri, (lane & ~3) + i * (2 / LT));
      __syncwarp();
      if (last) {
        // Y(l,j) = sum_k L[j,k,l] y(k,j): A = the weights, rows l; staged over the rows (l, j) of Q the
        // scores were formed from (only this warp reads them)
        uint32_t pa[LT][2][4];
#pragma unroll
        for (int lt = 0; lt < LT; ++lt)
#pragma unroll
          for (int k2 = 0; k2 < 2; ++k2) {
            pa[lt][k2][0] = M::pack(s[lt][2 * k2][0], s[lt][2 * k2][1]);
            pa[lt][k2][1] = M::pack(s[lt][2 * k2][2], s[lt][2 * k2][3]);
            pa[lt][k2][2] = M::pack(s[lt][2 * k2 + 1][0], s[lt][2 * k2 + 1][1]);
            pa[lt][k2][3] = M::pack(s[lt][2 * k2 + 1][2], s[lt][2 * k2 + 1][3]);
          }
#pragma unroll
        for (int vp = 0; vp < 4; ++vp) {          // two 8-column tiles of v per load
          uint32_t bf[2][4];      // B[k][v] = y(k,j)[v], read transposed
#pragma unroll
          for (int k2 = 0; k2 < 2; ++k2) ldsm_x4_trans(bf[k2], swz(ry(16 * k2 + (lane & 15), jj), 2 * vp + (lane >> 4)));
#pragma unroll
          for (int lt = 0; lt < LT; ++lt) {
            float o[2][4];
#pragma unroll
            for (int k2 = 0; k2 < 2; ++k2) {
              mma<__half>(k2 == 0, o[0], pa[lt][k2], bf[k2]);
              mma<__half>(k2 == 0, o[1], pa[lt][k2], bf[k2] + 2);
            }
            const float2 i0 = both(inv[lt][0]), i1 = both(inv[lt][1]);
            stsm_x4(swz(rq(l0 + 16 * lt + (lane & 15), jj), 2 * vp + (lane >> 4)), M::pack(fmul2(row_pair(o[0], 0), i0)),
                    M::pack(fmul2(row_pair(o[0], 1), i1)), M::pack(fmul2(row_pair(o[1], 0), i0)),
                    M::pack(fmul2(row_pair(o[1], 1), i1)));
          }
        }
        __syncwarp();
        // the rows (l, j) of Y are complete: 16 bytes per lane and store
        const int ch = lane & 7;
#pragma unroll
        for (int r = 0; r < 4 * LT; ++r) {
          const int l = l0 + (lane >> 3) + 4 * r;
          const uint4 v = *reinterpret_cast<const uint4*>(smem + (swz(rq(l, jj), ch) - s0));
          TIn* gp = Y + ((size_t)row0 + l * kB + jc + jj) * (size_t)(H ? H * kD : kD) + x0 + ch * 8;
          *reinterpret_cast<uint4*>(gp) = warpmma::from_f16x8(v, gp);
        }
      } else {
        // alpha_R(k,j) = sum_l L[j,k,l] Q(l,j) / c_R, c_R(k,j) = sum_l L[j,k,l]: the contraction runs over
        // the ROW index of the weights, so the A fragments are their transpose.  The result does not
        // change when column k is multiplied by any g_k > 0: g_k = 2^-(exponent of the column's largest
        // weight) keeps every column's significant weights in the normal f16 range however small c_R
        // is; c_R comes out of the same MMAs (a B operand of ones), i.e. summed over the weights AS
        // ROUNDED like the numerator.
        // Two warps that share a position exchange their column maxima, then their scaled weights, and
        // each forms 16 of the rows k.
        float cms[8];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
          cms[2 * nt] = cms[2 * nt + 1] = 0.f;
#pragma unroll
          for (int lt = 0; lt < LT; ++lt)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
              const float2 v = fmul2(row_pair(s[lt][nt], hh), both(inv[lt][hh]));
              put_pair(s[lt][nt], hh, v);
              cms[2 * nt] = fmaxf(cms[2 * nt], v.x);
              cms[2 * nt + 1] = fmaxf(cms[2 * nt + 1], v.y);
            }
        }
        float cm = scatter_reduce<8, 16, 4>(cms, lane, warpmma::Max());     // of column 8 (g / 2) + 2 t + g % 2
        if constexpr (W == 2) {
          float* xm = reinterpret_cast<float*>(smem + L::X + jj * 256);
          xm[2 * l0 + lane] = cm;
          asm volatile("bar.sync %0, 64;" ::"r"(1 + jj) : "memory");
          cm = fmaxf(cm, xm[32 - 2 * l0 + lane]);
        }
        const float gl = cm > 0.f ? __uint_as_float((253u << 23) - (__float_as_uint(cm) & 0x7f800000u)) : 0.f;
        uint32_t w[LT][2][4];      // [row tile][half][8-column tile]
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
          float gk[2];
#pragma unroll
          for (int e = 0; e < 2; ++e) gk[e] = __shfl_sync(0xffffffffu, gl, (2 * nt + e) * 4 + t);
#pragma unroll
          for (int lt = 0; lt < LT; ++lt)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) w[lt][hh][nt] = M::pack(fmul2(row_pair(s[lt][nt], hh), make_float2(gk[0], gk[1])));
        }
        uint32_t pk[LT][2][4];     // A[k][l], the weights transposed: row tile kt, contraction step ls
        if constexpr (W == 2) {
          // row l (64 bytes), 16-byte chunk c of the exchanged weights
          auto pt = [&](int l, int c) { return s0 + L::P + jj * 2048 + l * 64 + ((c ^ ((l >> 1) & 3)) << 4); };
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) stsm_x4(pt(l0 + 8 * hh + (lane & 7), lane >> 3), w[0][hh][0], w[0][hh][1], w[0][hh][2], w[0][hh][3]);
          asm volatile("bar.sync %0, 64;" ::"r"(1 + jj) : "memory");
#pragma unroll
          for (int ls = 0; ls < 2; ++ls)
            ldsm_x4_trans(pk[0][ls], pt(16 * ls + (lane & 7) + 8 * (lane >> 4), l0 / 8 + ((lane >> 3) & 1)));
        } else {
#pragma unroll
          for (int kt = 0; kt < LT; ++kt)
#pragma unroll
            for (int ls = 0; ls < 2; ++ls)
#pragma unroll
              for (int i = 0; i < 4; ++i) pk[kt][ls][i] = movm_trans(w[ls * (LT - 1)][i >> 1][2 * kt + (i & 1)]);
        }
        const uint32_t ones[2] = {0x3C003C00u, 0x3C003C00u};
        float ic[LT][2], c1 = 0.f;
#pragma unroll
        for (int kt = 0; kt < LT; ++kt) {
          float cr[4];
#pragma unroll
          for (int ls = 0; ls < 2; ++ls) mma<__half>(ls == 0, cr, pk[kt][ls], ones);
          if (t == 2 * kt) c1 = cr[0];            // a division a lane
          if (t == 2 * kt + 1) c1 = cr[2];
        }
        c1 = c1 > 1e-30f ? 1.f / c1 : 0.f;
#pragma unroll
        for (int i = 0; i < 2 * LT; ++i) ic[i >> 1][i & 1] = __shfl_sync(0xffffffffu, c1, (lane & ~3) + i);
#pragma unroll
        for (int vp = 0; vp < 4; ++vp) {
          uint32_t bf[2][4];       // B[l][v] = Q(l,j)[v], read transposed; two 8-column tiles
#pragma unroll
          for (int ls = 0; ls < 2; ++ls) ldsm_x4_trans(bf[ls], swz(rq(16 * ls + (lane & 15), jj), 2 * vp + (lane >> 4)));
#pragma unroll
          for (int kt = 0; kt < LT; ++kt) {
            float o[2][4];
#pragma unroll
            for (int ls = 0; ls < 2; ++ls) {
              mma<__half>(ls == 0, o[0], pk[kt][ls], bf[ls]);
              mma<__half>(ls == 0, o[1], pk[kt][ls], bf[ls] + 2);
            }
            // alpha_R rows (k, j) over the alpha_L rows (whose readers have formed their scores)
            stsm_x4(swz(rs(l0 + 16 * kt + (lane & 15), jj), 2 * vp + (lane >> 4)), M::pack(fmul2(row_pair(o[0], 0), both(ic[kt][0]))),
                    M::pack(fmul2(row_pair(o[0], 1), both(ic[kt][1]))), M::pack(fmul2(row_pair(o[1], 0), both(ic[kt][0]))),
                    M::pack(fmul2(row_pair(o[1], 1), both(ic[kt][1]))));
          }
        }
      }
    }
    if (!last) __syncthreads();
  }
  if (par & kDead) tensor::let_copies_land();
}

inline bool supported(int N, int d, int b, int m, int dtype, int BH) {
  return (dtype == 1 || dtype == 2) && N == kN && d == kD && b == kB && m == kM && BH <= 65535;
}

// `status`: device word that a bounded wait which ran out sets; `clear`: word to clear first, or nullptr.
int launch(const void* Q, const void* K, const void* V, void* Y, int BH, int T, int dtype, float scale,
           int* status, int* clear, const tensor::Waits& waits, cudaStream_t st, int H = 0);

#ifdef MA_TU_FUSED_JSPLIT
struct Maps {
  const void *q = nullptr, *k = nullptr, *v = nullptr;
  int BH = 0, dtype = 0, dev = -1, H = 0, q_rows = 0;
  CUtensorMap tmQ, tmK, tmV;
};
inline bool make_map(CUtensorMap* tm, int dtype, const void* base, uint64_t rows, uint32_t box_rows, int H) {
  tensor::EncodeTiledFn fn = tensor::encode_fn();
  if (!fn) return false;
  const uint64_t cols = H ? (uint64_t)H * kD : kD;
  if (H) rows /= H;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {kD, box_rows};
  cuuint32_t es[2] = {1, 1};
  return fn(tm, dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
            const_cast<void*>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <typename TIn, int PJ, int W, bool NEG>
inline int launch_k(const Maps& mp, void* Y, int BH, int T, float scale, int* status, int* clear, cudaStream_t st, int H) {
  auto kern = monarch_jsplit32<TIn, PJ, W, NEG>;
  using L = Lay<PJ, W>;
  static warpmma::SmemOptIn opt_in;
  if (!opt_in.done((const void*)kern, L::kSmem)) return 7;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kB / PJ, BH);      // the CTAs of a head are neighbours: they share K and V in L2
  cfg.blockDim = dim3(L::kThreads);
  cfg.dynamicSmemBytes = L::kSmem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, mp.tmQ, mp.tmK, mp.tmV, (TIn*)Y, T, fabsf(scale), status, clear, H) == cudaSuccess ? 0 : 7;
}

template <typename TIn, int PJ, int W>
inline int launch_t(const Maps& mp, void* Y, int BH, int T, float scale, int* status, int* clear, cudaStream_t st, int H) {
  return scale < 0.f ? launch_k<TIn, PJ, W, true>(mp, Y, BH, T, scale, status, clear, st, H)
                     : launch_k<TIn, PJ, W, false>(mp, Y, BH, T, scale, status, clear, st, H);
}

int launch(const void* Q, const void* K, const void* V, void* Y, int BH, int T, int dtype, float scale,
           int* status, int* clear, const tensor::Waits& waits, cudaStream_t st, int H) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 7;
  // As long as one wave holds four CTAs a head, two warps share a position: 13.5 us against 19.0 (T = 2).
  // Beyond that a K fragment used for two tiles of positions wins: 48 heads 20.6 against 26.9 us, 80 heads
  // (three waves against two) 38.2 against 38.6, 192 heads 58.1 against 76.1.
  const int pj = BH * (kB / 8) <= 148 ? 8 : 16, q_rows = waits.starve ? 1 : pj;
  // the tensor maps of the last few (Q, K, V) triples are kept: encoding three maps costs more host
  // time than the launch itself
  static thread_local Maps cache[8];
  static thread_local int next = 0;
  const Maps* mp = nullptr;
  for (int i = 0; i < 8; ++i)
    if (cache[i].q == Q && cache[i].k == K && cache[i].v == V && cache[i].BH == BH && cache[i].dtype == dtype &&
        cache[i].dev == dev && cache[i].H == H && cache[i].q_rows == q_rows)
      mp = &cache[i];
  if (!mp) {
    Maps& m = cache[next];
    next = (next + 1) % 8;
    m.dev = -1;
    const uint64_t rows = (uint64_t)BH * kN;
    if (!make_map(&m.tmQ, dtype, Q, rows, q_rows, H) || !make_map(&m.tmK, dtype, K, rows, kB, H) ||
        !make_map(&m.tmV, dtype, V, rows, kB, H))
      return 7;
    m.q = Q; m.k = K; m.v = V; m.BH = BH; m.dtype = dtype; m.dev = dev; m.H = H; m.q_rows = q_rows;
    mp = &m;
  }
  if (dtype == 1)
    return pj == 8 ? launch_t<__half, 8, 2>(*mp, Y, BH, T, scale, status, clear, st, H) : launch_t<__half, 16, 1>(*mp, Y, BH, T, scale, status, clear, st, H);
  return pj == 8 ? launch_t<__nv_bfloat16, 8, 2>(*mp, Y, BH, T, scale, status, clear, st, H)
                 : launch_t<__nv_bfloat16, 16, 1>(*mp, Y, BH, T, scale, status, clear, st, H);
}
#endif  // MA_TU_FUSED_JSPLIT

}  // namespace jsplit
}  // namespace ma
