// Fused kernel for short sequences, a head at a time: N = m b with 9 <= m, b <= 32 (m need not equal
// b), d <= 64 (a multiple of 8), f16 / bf16, plain f16 states, key padding mask or per-sequence lengths
// (App. C.3), either layout, row log-sum-exp.  All T rounds of Eq. 7-10 and Eq. 4 in one launch; Q, K, V
// are read from HBM once, the states stay in shared memory, Y is written once.
//
// What bounds it.  A head is 3 N d 16-bit values in and N d out for a few dozen small MMAs per block: the
// time is HBM traffic if the loads of the next head run under the arithmetic of this one and the
// instruction stream is short enough.  Hence
//   * an SM works on as many heads at a time as its shared memory holds: three or two small CTAs, or one CTA that
//     starts on a head by requesting the next (every warp asks TMA for the Q, K and V rows of the blocks it will own
//     there, zero-filled past d); `plan` (head_plan.h) chooses.  A head of 16 x 24 takes 157 KB: one, with its loads exposed;
//   * rows of a tile lie k bp + i with an odd block pitch bp = b | 1: under the 128-byte swizzle of the TMA
//     eight rows are then free of bank conflicts along a block (R half-step) and across blocks
//     (L half-step), so the permutation between the half-steps is only a choice of rows;
//   * a warp owns a block (R) or a position (L) and holds its scores and weights in registers, in as many
//     8-column tiles as b or m need;
//   * few heads of more than 16 rows a block go to two CTAs each, by in-block position (`plan`).
// One round: alpha_L goes over K, y over V, Y over Q.  More rounds: alpha_R and alpha_L replace each
// other in place in a state tile.  Arithmetic is f16 whatever the input type (see fused_small.cuh).
//
// Measured (B200, us per call, against the general per-head kernel): 768 heads of 256 = 16 x 16, one
// round 23.7 / 27.7 (65 % of the copy bandwidth); 768 of 210 = 15 x 14, two rounds 36.4 / 47.7; 384 of
// lengths up to 384 = 16 x 24 23.6 / 28.9.  24 of 210 4.4, two rounds 7.0; 720 of 396 = 22 x 18 53, 94.  Row and column
// reductions that halve the values a lane carries, with one division a lane, took 3 % (16 x 16) to 11 %
// (10 x 24, two rounds) off.  The tiles wait on latencies: 32 warps with two heads at work, where two 8-column tiles either way
// fit 64 registers, took 41 to 36.3 us (15 x 14, two rounds) and 24.8 to 23.8 (16 x 16, one).  What is left is latency at four to eight
// warps per scheduler, and the last turn of heads, which few SMs take.
#pragma once
#include <cuda.h>

#include "head_plan.h"
#include "status_word.cuh"
#include "tensor_path.cuh"
#include "warp_mma.cuh"

namespace ma {
namespace fhead {

using tensor::mbar_expect_tx;
using tensor::mbar_init;
using tensor::smem_u32;
using warpmma::Mma;
using warpmma::ex2;
using warpmma::kLn2;
using warpmma::kLog2e;
using warpmma::ldsm_x4;
using warpmma::ldsm_x4_trans;
using warpmma::lg2;
using warpmma::movm_trans;
using warpmma::quad_max;
using warpmma::scatter_reduce;

constexpr float kMasked = -3.0e38f;      // finite, and far below any score

struct Params {
  CUtensorMap q, k, v;      // (d, b, m, heads, batch), box (64, bp, 1, 1, 1)
  void* Y;
  float* lse;
  const int* seq_len;
  int *status, *clear;      // set by a wait that ran out; to clear first, or nullptr
  int BH, N, d, b, m, T, H, heads, n_valid;
  int bp;                   // block pitch in rows
  int tile;                 // bytes of a tile
  int bufs;                 // heads in shared memory
  int part;                 // positions of a CTA (a head to two CTAs)
  float scale;
};

__device__ __forceinline__ void stsm_x4(uint32_t saddr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(saddr), "r"(r0),
               "r"(r1), "r"(r2), "r"(r3)
               : "memory");
}
__device__ __forceinline__ void load_5d(uint32_t dst, const CUtensorMap* tm, uint64_t* bar, int blk, int h0, int h1) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %3, %4, %5, %6}], [%2];" ::"r"(
          dst),
      "l"((uint64_t)tm), "r"(smem_u32(bar)), "r"(0), "r"(blk), "r"(h0), "r"(h1)
      : "memory");
}
__device__ __forceinline__ void prefetch_5d(const CUtensorMap* tm, int blk, int h0, int h1) {
  asm volatile("cp.async.bulk.prefetch.tensor.5d.L2.global [%0, {%1, %1, %2, %3, %4}];" ::"l"((uint64_t)tm), "r"(0), "r"(blk), "r"(h0),
               "r"(h1)
               : "memory");
}
// Four 8 x 8 pieces of an accumulator pair (two 8-column tiles of 16 rows) as 16-bit rows.
__device__ __forceinline__ void put(uint32_t addr, const float (&o)[2][4], float m0, float m1) {
  typedef Mma<__half> M;
  const float2 a = both(m0), b = both(m1);
  stsm_x4(addr, M::pack(fmul2(make_float2(o[0][0], o[0][1]), a)), M::pack(fmul2(make_float2(o[0][2], o[0][3]), b)),
          M::pack(fmul2(make_float2(o[1][0], o[1][1]), a)), M::pack(fmul2(make_float2(o[1][2], o[1][3]), b)));
}
// Byte offset of a 16-byte chunk of a row under the 128-byte swizzle.
__device__ __forceinline__ uint32_t at(uint32_t base, int row, int chunk) {
  return base + (uint32_t)(row * 128 + ((chunk ^ (row & 7)) << 4));
}
// Rows row_of(0 .. 8 NT - 1) of a tile as B operands of NT 8-column tiles, four 16-column steps.
template <int NT, typename RowOf>
__device__ __forceinline__ void load_b(uint32_t (&kb)[NT][4][2], uint32_t base, int lane, RowOf row_of) {
#pragma unroll
  for (int np = 0; np < NT / 2; ++np) {
    const uint32_t ad = at(base, row_of(16 * np + (lane & 7) + (lane >> 4) * 8), (lane >> 3) & 1);
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      uint32_t r[4];
      ldsm_x4(r, ad ^ (ks << 5));
      kb[2 * np][ks][0] = r[0]; kb[2 * np][ks][1] = r[1];
      kb[2 * np + 1][ks][0] = r[2]; kb[2 * np + 1][ks][1] = r[3];
    }
  }
  if (NT & 1) {
    const uint32_t ad = at(base, row_of(8 * (NT - 1) + (lane & 7)), lane >> 3);
#pragma unroll
    for (int k2 = 0; k2 < 2; ++k2) {
      uint32_t r[4];
      ldsm_x4(r, ad ^ (k2 << 6));
      kb[NT - 1][2 * k2][0] = r[0]; kb[NT - 1][2 * k2][1] = r[1];
      kb[NT - 1][2 * k2 + 1][0] = r[2]; kb[NT - 1][2 * k2 + 1][1] = r[3];
    }
  }
}
// The 16 x 8 NT weights of a row tile as A fragments of (NT + 1) / 2 16-column steps.
template <int NT>
__device__ __forceinline__ void pack_a(uint32_t (&pa)[(NT + 1) / 2][4], const float (&s)[NT][4]) {
  typedef Mma<__half> M;
#pragma unroll
  for (int kk = 0; kk < (NT + 1) / 2; ++kk) {
    pa[kk][0] = M::pack(s[2 * kk][0], s[2 * kk][1]);
    pa[kk][1] = M::pack(s[2 * kk][2], s[2 * kk][3]);
    pa[kk][2] = 2 * kk + 1 < NT ? M::pack(s[(2 * kk + 1) % NT][0], s[(2 * kk + 1) % NT][1]) : 0u;
    pa[kk][3] = 2 * kk + 1 < NT ? M::pack(s[(2 * kk + 1) % NT][2], s[(2 * kk + 1) % NT][3]) : 0u;
  }
}

// Two 8-column tiles of a product over KT 16-row steps.
template <int KT>
__device__ __forceinline__ void products(float (&o)[2][4], const uint32_t (&a)[KT][4], const uint32_t (&b)[KT][4]) {
  typedef Mma<__half> M;
#pragma unroll
  for (int kk = 0; kk < KT; ++kk)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      if (kk == 0) M::first(o[v], a[kk], b[kk] + 2 * v);
      else M::run(o[v], a[kk], b[kk] + 2 * v);
    }
}

// NB, NM: 8-column tiles that hold b keys / m blocks.  WARPS: on an SM.  RT: 16-row tiles of a block's positions that a CTA has: all of
// them, or one where a head goes to two CTAs (nothing couples two positions but K and V, which both read).
template <typename TIn, int NB, int NM, int ROUNDS, int WARPS, int RT = (NB + 1) / 2>
__global__ void __launch_bounds__(32 * WARPS, 1) monarch_fused_head(const __grid_constant__ Params P) {
  typedef Mma<__half> M;
  constexpr bool MULTI = ROUNDS != kOne, V_LAST = ROUNDS == kMoreVLast;
  constexpr int RB = (NB + 1) / 2, RM = (NM + 1) / 2;      // 16-row tiles
  constexpr bool SPLIT = RT < RB;
  extern __shared__ uint8_t smem_raw[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  uint8_t* smem = align_smem<1024>(smem_raw);
  const int tile = P.tile, b = P.b, bp = P.bp;
  const uint32_t s0 = smem_u32(smem);
  const int tiles = V_LAST ? 3 : 3 * P.bufs + (MULTI ? 1 : 0);
  const uint32_t sS = s0 + (tiles - 1) * tile;             // state tile (MULTI)
  uint8_t* tail = smem + tiles * tile;
  float* sCL = reinterpret_cast<float*>(tail + 128);
  const int tid = threadIdx.x, warp = warp_of_cta(), lane = tid & 31, g = lane >> 2, t = lane & 3;
  const uint32_t dump = smem_u32(tail) + (lane & 7) * 16;
  Bars* bars = reinterpret_cast<Bars*>(sCL + b * NM * 8);
  if (tid == 0) {
    for (int i = 0; i < (V_LAST ? 2 : P.bufs); ++i)
      for (int k = 0; k < P.m; ++k) mbar_init(&bars->full[i][k], 1);
    tensor::fence_barrier_init();
  }
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  clear_status(P.clear);

  auto valid_of = [&](int h) { return P.seq_len != nullptr ? min(max(P.seq_len[h / P.heads], 1), P.N) : P.n_valid; };
  const int nw = blockDim.x >> 5;
  const float fl = P.scale * kLog2e;
  // per-lane row within 16 and 16-byte chunk: A operands, transposed B operands, matrix stores
  const int a_row = lane & 15, a_ch = lane >> 4;

  // Requests the blocks of head h that this warp owns in the R half-step (absent ones excepted).
  auto request = [&](int h, int buf) {
    if (lane != 0 || h >= P.BH) return;
    const int h0 = P.H ? h % P.H : h, h1 = P.H ? h / P.H : 0;
    const int m = P.seq_len != nullptr ? (valid_of(h) + b - 1) / b : P.m;
    for (int k = warp; k < m; k += nw) {
      uint64_t* bar = &bars->full[buf][k];
      const uint32_t dst = s0 + 3 * buf * tile + k * bp * 128;
      mbar_expect_tx(bar, (V_LAST ? 2 : 3) * bp * 128);
      load_5d(dst, &P.q, bar, k, h0, h1);
      load_5d(dst + tile, &P.k, bar, k, h0, h1);
      if (!V_LAST) load_5d(dst + 2 * tile, &P.v, bar, k, h0, h1);
      else prefetch_5d(&P.v, k, h0, h1);
    }
  };
  // bf16: to f16 in place, `n` operands of a block, a tile apart.
  auto convert = [&](uint32_t block, int n) {
    if (Mma<TIn>::is_f16) return;
    for (int e = lane; e < b * 8; e += 32) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if (a >= n) break;
        uint4* p = reinterpret_cast<uint4*>(smem + (block - s0) + a * tile + e * 16);
        *p = warpmma::to_f16x8(*p, (const TIn*)nullptr);
      }
    }
  };
  const int first_head = SPLIT ? (int)blockIdx.x >> 1 : (int)blockIdx.x, step_heads = SPLIT ? P.BH : (int)gridDim.x;
  const int j0 = SPLIT && (blockIdx.x & 1) ? P.part : 0, j1 = SPLIT ? min(j0 + P.part, b) : b;      // the CTA's positions
  request(first_head, 0);
  int buf = 0;
  uint32_t par = 0;                 // bit 16 buf + r: parity of the warp's r-th block in that buffer
  constexpr uint32_t kDead = 1u << 31;      // in `par`: a wait ran out; the warp waits no more and leaves after this head
  auto landed = [&](uint64_t* bar, int bit) {
    if (!(par & kDead) && !tensor::mbar_wait(bar, (par >> bit) & 1)) {
      tensor::report_timeout(P.status, 2);
      par |= kDead;
    }
    par ^= 1u << bit;
  };
  for (int h = first_head; h < P.BH; h += step_heads) {
    if (!V_LAST && P.bufs == 2) request(h + step_heads, buf ^ 1);
    const uint32_t sQ = s0 + 3 * buf * tile, sK = sQ + tile, sV = V_LAST ? sS : sK + tile;
    const int n_valid = valid_of(h);
    const int m = P.seq_len != nullptr ? (n_valid + b - 1) / b : P.m;
    const size_t head_base = P.H == 0 ? (size_t)h * P.N * P.d : ((size_t)(h / P.H) * P.N * P.H + (h % P.H)) * P.d;
    const size_t row_stride = P.H == 0 ? (size_t)P.d : (size_t)P.H * P.d;
    for (int step = 1; step <= P.T; ++step) {
      const bool first = !MULTI || step == 1, last = !MULTI || step == P.T;
      // ================================================================ R half-step (Eq. 7, 9, 10)
      for (int k = warp, r = 0; k < m; k += nw, ++r) {
        const int r0 = k * bp;
        if (first) {
          landed(&bars->full[buf][k], 16 * buf + r);
          convert(sQ + r0 * 128, V_LAST ? 2 : 3);
          __syncwarp();
        }
        const uint32_t sA = first ? sQ : sS;                 // alpha_R (= Q rows while L is the identity)
        const uint32_t dst = !MULTI || (V_LAST && last) ? sK : sS;      // alpha_L
        const int lim = min(b, n_valid - k * b);             // keys of this block that count
        uint32_t pa[RT][RB][4];                              // unnormalised weights: the largest is exactly 1
        float inv[RT][2], off[2 * RT], red[4 * RT];          // red: sum of the weights, sum of weight times score
        {
          uint32_t kb[NB][4][2];
          load_b<NB>(kb, sK, lane, [&](int i) { return r0 + min(i, b - 1); });
#pragma unroll
          for (int rt = 0; rt < RT; ++rt) {
            float s[NB][4];
            const uint32_t ad = at(sA, r0 + min(j0 + 16 * rt + a_row, b - 1), a_ch);
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
              uint32_t a[4];
              ldsm_x4(a, ad ^ (ks << 5));
#pragma unroll
              for (int nt = 0; nt < NB; ++nt) {
                if (ks == 0) M::first(s[nt], a, kb[nt][ks]);
                else M::run(s[nt], a, kb[nt][ks]);
              }
            }
            // rows j = j0 + 16 rt + g (c0, c1) and + 8 (c2, c3); columns i = 8 nt + 2 t, + 1.  Columns past the
            // block, in the last column tile, and padded keys of the last block: a score of weight 0.
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (8 * (NB - 1) + 2 * t + (e & 1) >= lim) s[NB - 1][e] = kMasked;
            if (lim < b) {
#pragma unroll
              for (int nt = 0; nt < NB - 1; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                  if (8 * nt + 2 * t + (e & 1) >= lim) s[nt][e] = kMasked;
            }
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
              float mx = kMasked;
#pragma unroll
              for (int nt = 0; nt < NB; ++nt) mx = fmaxf(mx, fmaxf(s[nt][2 * hh], s[nt][2 * hh + 1]));
              mx = quad_max(mx);
              off[2 * rt + hh] = -mx * fl;
              float2 sum = both(0.f), sz = both(0.f);
#pragma unroll
              for (int nt = 0; nt < NB; ++nt) {
                const float2 x = make_float2(s[nt][2 * hh], s[nt][2 * hh + 1]);
                const float2 z = ffma2(x, both(fl), both(off[2 * rt + hh]));
                const float2 p = make_float2(ex2(z.x), ex2(z.y));
                s[nt][2 * hh] = p.x;
                s[nt][2 * hh + 1] = p.y;
                sum = nt ? fadd2(sum, p) : p;
                sz = nt ? ffma2(p, x, sz) : fmul2(p, x);      // 0 times a finite number where masked (0 log 0 = 0)
              }
              red[2 * (2 * rt + hh)] = sum.x + sum.y;
              red[2 * (2 * rt + hh) + 1] = sz.x + sz.y;
            }
            pack_a<NB>(pa[rt], s);
          }
          // a lane ends up with both sums of row q = t (two row tiles), or with one of them: one division a
          // lane, the reciprocals then go to the row's four lanes
          const float r = scatter_reduce<4 * RT, 2, 1>(red, lane, warpmma::Add());
          const float ri = 1.f / r;
          const int q = RT == 2 ? t : t >> 1, j = j0 + 16 * (q >> 1) + g + 8 * (q & 1);
#pragma unroll
          for (int i = 0; i < 2 * RT; ++i) inv[i >> 1][i & 1] = __shfl_sync(0xffffffffu, ri, (lane & ~3) + i * (2 / RT));
          float so = r, sz = red[1], io = ri, mo = off[0];
          if (RT == 1) {
            sz = r;
            so = __shfl_xor_sync(0xffffffffu, r, 1);
            io = __shfl_xor_sync(0xffffffffu, ri, 1);
          }
#pragma unroll
          for (int i = 1; i < 2 * RT; ++i) mo = q == i ? off[i] : mo;
          // -c_L log2 e = log2 sum + max - sum R z (Eq. 10), the addend of the L logits
          if ((RT == 2 || (t & 1)) && j < j1) sCL[j * NM * 8 + k] = lg2(so) - mo - fl * (sz * io);
        }
        if (V_LAST && last) {      // the block's rows of alpha_R have been read, V takes their place
          tensor::fence_proxy_async();
          __syncwarp();
          if (lane == 0 && !(par & kDead)) {
            mbar_expect_tx(&bars->full[1][k], bp * 128);
            load_5d(sV + r0 * 128, &P.v, &bars->full[1][k], k, P.H ? h % P.H : h, P.H ? h / P.H : 0);
          }
        }
        __syncwarp();
        // second products, 16 columns at a time; a warp alone reads and writes the rows of its block
        uint32_t kt[RB], st[RT];
#pragma unroll
        for (int kk = 0; kk < RB; ++kk) kt[kk] = at(sK, r0 + min(16 * kk + a_row, b - 1), a_ch);
#pragma unroll
        for (int rt = 0; rt < RT; ++rt) st[rt] = j0 + 16 * rt + a_row < j1 ? at(dst, r0 + j0 + 16 * rt + a_row, a_ch) : dump;
        // (from the K tile's addresses to the V tile's, from those of alpha_L to y's)
        const uint32_t to_v = sV - sK;
        uint32_t sy[RT];
#pragma unroll
        for (int rt = 0; rt < RT; ++rt) sy[rt] = j0 + 16 * rt + a_row < j1 ? st[rt] - dst + sV : dump;
#pragma unroll
        for (int np = 0; np < 4; ++np) {
          uint32_t bk[RB][4], bv[RB][4];
#pragma unroll
          for (int kk = 0; kk < RB; ++kk) {
            const uint32_t ad = kt[kk] ^ (np << 5);
            ldsm_x4_trans(bk[kk], ad);
            if (!V_LAST && last) ldsm_x4_trans(bv[kk], ad + to_v);
          }
          __syncwarp();
#pragma unroll
          for (int rt = 0; rt < RT; ++rt) {
            float o[2][4];
            products<RB>(o, pa[rt], bk);
            put(st[rt] ^ (np << 5), o, inv[rt][0], inv[rt][1]);
            if (!V_LAST && last) {
              products<RB>(o, pa[rt], bv);
              put(sy[rt] ^ (np << 5), o, inv[rt][0], inv[rt][1]);
            }
          }
        }
        if (V_LAST && last) {
          landed(&bars->full[1][k], 16 + r);
          convert(sV + r0 * 128, 1);
          __syncwarp();
#pragma unroll
          for (int np = 0; np < 4; ++np) {
            uint32_t bv[RB][4];
#pragma unroll
            for (int kk = 0; kk < RB; ++kk) ldsm_x4_trans(bv[kk], (kt[kk] ^ (np << 5)) + to_v);
            __syncwarp();
#pragma unroll
            for (int rt = 0; rt < RT; ++rt) {
              float o[2][4];
              products<RB>(o, pa[rt], bv);
              put(sy[rt] ^ (np << 5), o, inv[rt][0], inv[rt][1]);
            }
          }
        }
      }
      __syncthreads();

      // ================================================================ L half-step (Eq. 8, 9 / Eq. 4)
      for (int j = j0 + warp; j < j1; j += nw) {
        const uint32_t sA = !MULTI || (V_LAST && last) ? sK : sS;       // alpha_L
        float c[NM][2];
#pragma unroll
        for (int nt = 0; nt < NM; ++nt) {
          const float2 v = *reinterpret_cast<const float2*>(sCL + j * NM * 8 + 8 * nt + 2 * t);
          c[nt][0] = 8 * nt + 2 * t < m ? v.x : kMasked;
          c[nt][1] = 8 * nt + 2 * t + 1 < m ? v.y : kMasked;
        }
        uint32_t pa[RM][RM][4];                              // weights, rows l (final, unnormalised)
        float inv[RM][2], red[2 * RM], mxs[2 * RM];
        float w[MULTI ? RM : 1][MULTI ? NM : 1][4];          // normalised weights (non-final)
        {
          uint32_t kb[NM][4][2];
          load_b<NM>(kb, sA, lane, [&](int k) { return min(k, m - 1) * bp + j; });
#pragma unroll
          for (int rt = 0; rt < RM; ++rt) {
            float s[NM][4];
            const uint32_t ad = at(sQ, min(16 * rt + a_row, m - 1) * bp + j, a_ch);
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
              uint32_t a[4];
              ldsm_x4(a, ad ^ (ks << 5));
#pragma unroll
              for (int nt = 0; nt < NM; ++nt) {
                if (ks == 0) M::first(s[nt], a, kb[nt][ks]);
                else M::run(s[nt], a, kb[nt][ks]);
              }
            }
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
              float mx = kMasked;
#pragma unroll
              for (int nt = 0; nt < NM; ++nt) {
                const float2 z = ffma2(make_float2(s[nt][2 * hh], s[nt][2 * hh + 1]), both(fl), make_float2(c[nt][0], c[nt][1]));
                s[nt][2 * hh] = z.x;
                s[nt][2 * hh + 1] = z.y;
                mx = fmaxf(mx, fmaxf(z.x, z.y));
              }
              mx = quad_max(mx);
              float2 sum = both(0.f);
#pragma unroll
              for (int nt = 0; nt < NM; ++nt) {
                const float2 z = fadd2(make_float2(s[nt][2 * hh], s[nt][2 * hh + 1]), both(-mx));
                const float2 p = make_float2(ex2(z.x), ex2(z.y));
                s[nt][2 * hh] = p.x;
                s[nt][2 * hh + 1] = p.y;
                sum = nt ? fadd2(sum, p) : p;
              }
              red[2 * rt + hh] = sum.x + sum.y;
              mxs[2 * rt + hh] = mx;
            }
            if (last) {
              pack_a<NM>(pa[rt], s);
            } else if (MULTI) {
#pragma unroll
              for (int nt = 0; nt < NM; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) w[MULTI ? rt : 0][MULTI ? nt : 0][e] = s[nt][e];
            }
          }
          const float r = scatter_reduce<2 * RM, 2, 1>(red, lane, warpmma::Add());     // of row q
          const float ri = 1.f / r;
#pragma unroll
          for (int i = 0; i < 2 * RM; ++i) inv[i >> 1][i & 1] = __shfl_sync(0xffffffffu, ri, (lane & ~3) + i * (2 / RM));
          // log-sum-exp of row b l + j of the final L half-step: summed over a head's rows it is the
          // objective (Eq. 6) at the returned matrix
          if (last && P.lse != nullptr) {
            const int q = RM == 2 ? t : t >> 1, l = 16 * (q >> 1) + g + 8 * (q & 1);
            float mx = mxs[0];
#pragma unroll
            for (int i = 1; i < 2 * RM; ++i) mx = q == i ? mxs[i] : mx;
            if ((RM == 2 || !(t & 1)) && l < m) P.lse[(size_t)h * P.N + (size_t)l * b + j] = (mx + lg2(r)) * kLn2;
          }
        }
        __syncwarp();
        uint32_t kt[RM], st[RM];
#pragma unroll
        for (int kk = 0; kk < RM; ++kk) {
          kt[kk] = at(last ? sV : sQ, min(16 * kk + a_row, m - 1) * bp + j, a_ch);
          st[kk] = 16 * kk + a_row < m ? at(last ? sQ : sS, (16 * kk + a_row) * bp + j, a_ch) : dump;
        }
        if (last) {
          // Y(l,j) = sum_k L[j,k,l] y(k,j), over the rows of Q the scores were formed from
#pragma unroll
          for (int np = 0; np < 4; ++np) {
            uint32_t by[RM][4];
#pragma unroll
            for (int kk = 0; kk < RM; ++kk) ldsm_x4_trans(by[kk], kt[kk] ^ (np << 5));
#pragma unroll
            for (int rt = 0; rt < RM; ++rt) {
              float o[2][4];
              products<RM>(o, pa[rt], by);
              put(st[rt] ^ (np << 5), o, inv[rt][0], inv[rt][1]);
            }
          }
          __syncwarp();
          const int ch = lane & 7;
          if (ch * 8 < P.d)
            for (int l = lane >> 3; l < P.m; l += 4) {
              // (rows of blocks that are absent from a shorter sequence: zeros)
              const uint4 v = l < m ? *reinterpret_cast<const uint4*>(smem + (at(sQ, l * bp + j, ch) - s0)) : make_uint4(0u, 0u, 0u, 0u);
              TIn* gp = (TIn*)P.Y + head_base + (size_t)(l * b + j) * row_stride + ch * 8;
              *reinterpret_cast<uint4*>(gp) = warpmma::from_f16x8(v, gp);
            }
        } else if constexpr (MULTI) {
          // alpha_R(k,j) = sum_l L[j,k,l] Q(l,j) / c_R, c_R(k,j) = sum_l L[j,k,l]: the contraction runs over
          // the rows of the weights, so the A fragments are their transpose.  Column k is multiplied by
          // g_k = 2^-(exponent of its largest weight) first (the quotient is invariant), which keeps its
          // significant weights in the normal f16 range however small c_R is; c_R comes out of the same
          // MMAs against a B fragment of ones, i.e. over the weights as rounded.
          constexpr int kCols = NM == 2 ? 4 : 8, kColStep = 32 / kCols;     // columns 8 (i / 2) + 2 t + i % 2 by i
          float cms[kCols];
#pragma unroll
          for (int i = 0; i < kCols; ++i) cms[i] = 0.f;
#pragma unroll
          for (int rt = 0; rt < RM; ++rt)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
              // (rows past the last block: not in sums over rows)
              const float on = 16 * rt + g + 8 * hh < m ? inv[rt][hh] : 0.f;
#pragma unroll
              for (int nt = 0; nt < NM; ++nt) {
                const float2 v = fmul2(make_float2(w[rt][nt][2 * hh], w[rt][nt][2 * hh + 1]), both(on));
                w[rt][nt][2 * hh] = v.x;
                w[rt][nt][2 * hh + 1] = v.y;
                cms[2 * nt] = fmaxf(cms[2 * nt], v.x);
                cms[2 * nt + 1] = fmaxf(cms[2 * nt + 1], v.y);
              }
            }
          const float cm = scatter_reduce<kCols, 16, 4>(cms, lane, warpmma::Max());
          const float gl = __uint_as_float((253u << 23) - (__float_as_uint(cm) & 0x7f800000u));
          uint32_t tp[RM][2][NM];
#pragma unroll
          for (int nt = 0; nt < NM; ++nt) {
            float gk[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) gk[e] = __shfl_sync(0xffffffffu, gl, (2 * nt + e) * kColStep + t);
#pragma unroll
            for (int rt = 0; rt < RM; ++rt)
#pragma unroll
              for (int hh = 0; hh < 2; ++hh)
                tp[rt][hh][nt] = movm_trans(M::pack(fmul2(make_float2(w[rt][nt][2 * hh], w[rt][nt][2 * hh + 1]), make_float2(gk[0], gk[1]))));
          }
          const uint32_t ones[2] = {0x3C003C00u, 0x3C003C00u};
          uint32_t pk[RM][RM][4];    // A[k][l]: rows k = 16 kq .., contraction over l = 16 ls ..
          float c1 = 0.f;
#pragma unroll
          for (int kq = 0; kq < RM; ++kq) {
            float cr[4];
#pragma unroll
            for (int ls = 0; ls < RM; ++ls) {
              pk[kq][ls][0] = tp[ls][0][2 * kq];
              pk[kq][ls][1] = 2 * kq + 1 < NM ? tp[ls][0][(2 * kq + 1) % NM] : 0u;
              pk[kq][ls][2] = tp[ls][1][2 * kq];
              pk[kq][ls][3] = 2 * kq + 1 < NM ? tp[ls][1][(2 * kq + 1) % NM] : 0u;
              if (ls == 0) M::first(cr, pk[kq][ls], ones);
              else M::run(cr, pk[kq][ls], ones);
            }
            if (t == 2 * kq) c1 = cr[0];      // a division a lane
            if (t == 2 * kq + 1) c1 = cr[2];
          }
          c1 = c1 > 1e-30f ? 1.f / c1 : 0.f;
#pragma unroll
          for (int kq = 0; kq < RM; ++kq) {
            const float i0 = __shfl_sync(0xffffffffu, c1, (lane & ~3) + 2 * kq), i1 = __shfl_sync(0xffffffffu, c1, (lane & ~3) + 2 * kq + 1);
#pragma unroll
            for (int np = 0; np < 4; ++np) {
              float o[2][4];
              uint32_t bq[RM][4];      // B[l][v] = Q(l,j)[v], read transposed
#pragma unroll
              for (int ls = 0; ls < RM; ++ls) ldsm_x4_trans(bq[ls], kt[ls] ^ (np << 5));
              products<RM>(o, pk[kq], bq);
              put(st[kq] ^ (np << 5), o, i0, i1);
            }
          }
        }
      }
      if (!last) __syncthreads();
    }
    // The head's buffer is free (and c_L, and the state tile) when every warp is done with it.
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (__any_sync(0xffffffffu, par & kDead)) {      // (barriers wait for the threads that have not left)
      tensor::let_copies_land();
      return;
    }
    if (!V_LAST && P.bufs == 2) buf ^= 1;
    else request(h + step_heads, 0);
  }
}

inline bool shape_ok(int d, int b, int m, int dtype) {
  return (dtype == 1 || dtype == 2) && d % 8 == 0 && d <= 64 && b > 8 && b <= 32 && m > 8 && m <= 32;
}
inline bool supported(int N, int d, int b, int m, int dtype, int T) {
  (void)N;
  Plan p;
  return shape_ok(d, b, m, dtype) && plan(b, m, T, 1, 1, &p);
}
struct Args {
  const void *Q, *K, *V;
  void* Y;
  int BH, N, d, b, m, T, dtype, H, heads, n_valid;
  float scale;
  float* lse;
  const int* seq_len;
  int *status, *clear;
  tensor::Waits waits;
};
int launch(const Args& a, cudaStream_t st);

#ifdef MA_TU_FUSED_HEAD
inline bool make_map(CUtensorMap* tm, const Args& a, const void* base, int box_rows) {
  tensor::EncodeTiledFn fn = tensor::encode_fn();
  if (!fn) return false;
  const cuuint64_t d2 = (cuuint64_t)a.d * 2, H = a.H ? a.H : 1, row = d2 * H, N = a.N, BH = a.BH;
  cuuint64_t dims[5] = {(cuuint64_t)a.d, (cuuint64_t)a.b, (cuuint64_t)a.m, a.H ? (cuuint64_t)a.H : BH, a.H ? BH / a.H : 1};
  cuuint64_t strides[4] = {row, a.b * row, a.H ? d2 : N * d2, N * d2 * (a.H ? H : BH)};
  cuuint32_t box[5] = {64, (cuuint32_t)box_rows, 1, 1, 1}, es[5] = {1, 1, 1, 1, 1};
  return fn(tm, a.dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims,
            strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
struct MapKey {
  const void *Q, *K, *V;
  int BH, N, d, b, dtype, H, box_rows, dev;
  bool operator==(const MapKey& o) const {
    return Q == o.Q && K == o.K && V == o.V && BH == o.BH && N == o.N && d == o.d && b == o.b && dtype == o.dtype && H == o.H &&
           box_rows == o.box_rows && dev == o.dev;
  }
};
// The maps of the last few problems are kept (encoding three costs more host time than the launch).
struct MapCache {
  static constexpr int kEntries = 16;
  MapKey key[kEntries];
  CUtensorMap maps[kEntries][3];
  bool used[kEntries] = {};
  int next = 0;
};
inline bool get_maps(Params* P, const Args& a, const Plan& p, int dev) {
  static thread_local MapCache c;
  const int rows = a.waits.starve ? 1 : p.bp;      // (a pitch is 9 or more)
  const MapKey key{a.Q, a.K, a.V, a.BH, a.N, a.d, a.b, a.dtype, a.H, rows, dev};
  int e = 0;
  while (e < MapCache::kEntries && !(c.used[e] && c.key[e] == key)) ++e;
  if (e == MapCache::kEntries) {
    e = c.next;
    c.next = (c.next + 1) % MapCache::kEntries;
    c.used[e] = false;
    if (!make_map(&c.maps[e][0], a, a.Q, rows) || !make_map(&c.maps[e][1], a, a.K, rows) || !make_map(&c.maps[e][2], a, a.V, rows))
      return false;
    c.key[e] = key;
    c.used[e] = true;
  }
  P->q = c.maps[e][0];
  P->k = c.maps[e][1];
  P->v = c.maps[e][2];
  return true;
}
template <typename TIn, int NB, int NM, int ROUNDS, int WARPS = max_warps(NB, NM, ROUNDS), int RT = (NB + 1) / 2>
inline int launch_k(const Params& P, const Plan& p, int num_sms, cudaStream_t st) {
  if constexpr (!any_fits(NB, NM)) return 4;
  else {
    auto kern = monarch_fused_head<TIn, NB, NM, ROUNDS, WARPS, RT>;
    static warpmma::SmemOptIn opt_in;
    if (!opt_in.done((const void*)kern, (int)kMaxSmem)) return 7;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    const int slots = p.ctas * num_sms, parts = p.parts * P.BH;
    cfg.gridDim = dim3(parts < slots ? parts : slots);
    cfg.blockDim = dim3(32 * p.warps);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, P) == cudaSuccess ? 0 : 7;
  }
}
template <typename TIn, int ROUNDS>
inline int launch_n(const Params& P, const Plan& p, int num_sms, cudaStream_t st) {
  const int nb = (P.b + 7) / 8, nm = (P.m + 7) / 8;
  if (p.bound == 16 && nb == 2 && nm == 2) return launch_k<TIn, 2, 2, ROUNDS, 16>(P, p, num_sms, st);
  if (p.bound == 24 && nb == 3 && nm == 2) return launch_k<TIn, 3, 2, ROUNDS, 24>(P, p, num_sms, st);
  if (p.parts == 2) {
#define MA_FH(B)                                                   \
  (nm == 2 ? launch_k<TIn, B, 2, ROUNDS, 16, 1>(P, p, num_sms, st) \
           : (nm == 3 ? launch_k<TIn, B, 3, ROUNDS, 16, 1>(P, p, num_sms, st) : launch_k<TIn, B, 4, ROUNDS, 16, 1>(P, p, num_sms, st)))
    return nb == 3 ? MA_FH(3) : MA_FH(4);
#undef MA_FH
  }
#define MA_FH(B)                                            \
  (nm == 2 ? launch_k<TIn, B, 2, ROUNDS>(P, p, num_sms, st) \
           : (nm == 3 ? launch_k<TIn, B, 3, ROUNDS>(P, p, num_sms, st) : launch_k<TIn, B, 4, ROUNDS>(P, p, num_sms, st)))
  return nb == 2 ? MA_FH(2) : (nb == 3 ? MA_FH(3) : MA_FH(4));
#undef MA_FH
}
template <typename TIn>
inline int launch_t(const Params& P, const Plan& p, int num_sms, cudaStream_t st) {
  if (p.rounds == kMoreVLast) return launch_k<TIn, 2, 2, kMoreVLast>(P, p, num_sms, st);
  return p.rounds == kMore ? launch_n<TIn, kMore>(P, p, num_sms, st) : launch_n<TIn, kOne>(P, p, num_sms, st);
}
int launch(const Args& a, cudaStream_t st) {
  static int sms[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 7;
  if (sms[dev] == 0 && cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 7;
  Plan p;
  Params P;
  if (!plan(a.b, a.m, a.T, a.BH, sms[dev], &p)) return 4;
  if (!get_maps(&P, a, p, dev)) return 7;
  P.Y = a.Y; P.lse = a.lse; P.seq_len = a.seq_len; P.status = a.status; P.clear = a.clear;
  P.BH = a.BH; P.N = a.N; P.d = a.d; P.b = a.b; P.m = a.m; P.T = a.T; P.H = a.H; P.heads = a.heads; P.n_valid = a.n_valid;
  P.bp = p.bp; P.tile = p.tile; P.bufs = p.bufs; P.part = (a.b + 1) / 2;
  P.scale = a.scale;
  return a.dtype == 1 ? launch_t<__half>(P, p, sms[dev], st) : launch_t<__nv_bfloat16>(P, p, sms[dev], st);
}
#endif  // MA_TU_FUSED_HEAD

}  // namespace fhead
}  // namespace ma
