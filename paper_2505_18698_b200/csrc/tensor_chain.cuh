// Persistent tensor-core kernel for m = b = 64 or 128 with tiles enough to fill the GPU (MA_PATH_TENSOR): tiles, order,
// tensor maps and dependency counters as described in tensor_persistent.cuh.
//
// What bounds a tile is its chain load -> score MMA -> softmax -> apply MMA -> rows -> store, nearly all of it latency; what bounds the
// kernel is how many chains an SM has in flight and what the states cost on their way through L2.  So, against the one chain with
// a stage per warpgroup of tensor_decoupled.cuh:
//   * two CTAs per SM with two compute groups of four warps each; a group (thread = score row) takes a tile from its scores
//     to its staged rows, and its first warp issues the tile's MMAs itself (hand-overs: tile_group.cuh; trying at mbarriers in a tighter loop, a
//     quarter more branches in all, cost 4 %).  Issuing a tile's eight score MMAs took
//     a thread about 1000 cycles and a release 500 (clock stamps) while the warp's number came from threadIdx and the release's word
//     went through shared memory: 74.0 us, 70.7 with uniform descriptors and a vote in the barrier;
//   * three 16 KB slots a group.  Which of them a tile's operands take follows from the order in which the tile before gives
//     its slots up (Slots), so that loads of the next tile run under the softmax of this one;
//   * the weights go back to tensor memory over the scores and are the A operand of the apply MMA; in the non-final L
//     half-step, which contracts over their rows, they go over the alpha_L operand, and c_R comes out of the same MMA as sixteen
//     more columns, of a tile of ones;
//   * alpha_R is stored divided by c_R: no c_R vector.  f16: the weights of that half-step carry 2^14 (the quotient does not change), so
//     that columns of small weights keep their bits.
// Service warps: a producer thread and a store warp per group.
//
// Measured (B200, us per call in loops of tenths of a second, against tensor_decoupled.cuh): 64 heads of 4096, T = 2 71 / 87, 16 of 16384 (the weights
// of a non-final L half-step then take two of the three slots) 88 / 98, 12 of 16300 masked 76 / 93.  GPUs differ by 5 %.  Measured and not kept:
// tiles dealt out in advance (81 against 78 us in bursts at the time: SMs differ in speed), a row of 64 scores in registers instead of read
// twice (no difference, masked 5 % slower), heads in groups that stay in L2 (more tiles are in work and
// requested, twice 592, than a half-step of 1024 leaves room for: 91 against 82), waits that do not suspend (2 % slower).
#pragma once
#include <type_traits>

#include "tensor_persistent.cuh"
#include "tile_group.cuh"
#include "tile_tc.cuh"

namespace ma {
namespace tp3 {

using namespace ma::group;
using ma::tp::Params;
using ma::tp::Tile;
using ma::tp::bulk_load_1d;
using ma::tp::ld_acquire;
using ma::tp::mbar_arrive;
using ma::tp::tma_store_commit;
using ma::tp::tma_store_wait_all;
using ma::tp::tma_store_wait_read;
using ma::ttc::ld_col;
using ma::ttc::st_cols;
using ma::ttc::umma_ts;

constexpr int kThreads = 384, kCtasPerSm = 2;
constexpr int kSlot = kTileBytes, kSlots = 6;
constexpr int kOffOnes = kSlots * kSlot;              // 2 KB of ones, above the slots
constexpr int kOffVec = kOffOnes + 2048;              // c_L, two tiles of 128 floats a group
constexpr int kOffBar = kOffVec + 4 * 512;
constexpr int kSmem = kOffBar + 512 + 1024;           // + alignment slack
static_assert(kCtasPerSm * (kSmem + 1024) <= 228 * 1024, "two CTAs per SM");

struct __align__(16) Shared {
  uint64_t full[2][2], third[2][2];                   // by group, tiles in turn: first two operands, third slot
  uint64_t empty[kSlots];
  uint64_t mma1[2], first[2], mma2[2], out_free[2];
  int through[2];                                     // tiles of a group that have left tensor memory
  int4 tile[2][2];                                    // {half-step, head, first block or position} of a tile, or {-1, ..}
  int4 out[2];                                        // {head or -1, first block or position, slot | Rows << 4 | last << 8, half-step}
  uint32_t tmem;
  volatile int abort_flag;
};
static_assert(sizeof(Shared) <= 512, "barrier block");
enum Rows { kAlphaL = 0, kY = 1, kAlphaR = 2, kOut = 3 };

__device__ __forceinline__ bool uses_third(const Tile& t) { return t.isR ? t.withV : t.final_; }      // a half-step of the last round
// Tile p, h, idx0 as its roles see it.
__device__ __forceinline__ Tile tile_of(const Params& P, int p, int h, int idx0) {
  Tile t;
  t.p = p;
  t.h = h;
  t.idx0 = idx0;
  t.isR = (p & 1) == 0;
  t.first = p == 0;
  t.withV = p == 2 * P.T - 2;
  t.final_ = p == 2 * P.T - 1;
  return t;
}

// EXTRA 1: inputs laid out [batch][N][heads][d], row log-sum-exp output; 2: the padding mask too, whose selects every tile pays for (40 heads
// of 4096 in the other layout 58.8 us with them, 56.0 without).
template <typename T, int B, int EXTRA>
struct Chain {
  static constexpr bool MASK = EXTRA == 2;
  static constexpr int FT = Fmt<T>::code, kBlocks = kRows / B;
  static constexpr float kWeightScale = std::is_same<T, __half>::value ? 16384.f : 1.f;      // of the non-final L weights

  // ================================================================ producer of group w (one thread)
  // Takes the next tile of the list (the order of tensor_persistent.cuh) from a counter: SMs differ in speed, and with tiles dealt
  // out in advance the slowest set the time (a sixth of it).
  static __device__ __forceinline__ void produce(const Params& P, uint8_t* smem, Shared* sh, int w) {
    const int tpg = P.tiles_per_phase / P.head_groups, per_group = 2 * P.T * tpg, hpg = P.BH / P.head_groups;
    Slots<B> x(w);
    uint32_t busy = 0, par = 0;              // by slot: a use is to be waited for; parity of that wait
    auto take = [&](int s) {
      const uint32_t bit = 1u << s;
      if ((busy & bit) && !wait_bar(&sh->empty[s], (par & bit) != 0, sh, P, 11)) return false;
      if (busy & bit) par ^= bit;
      busy |= bit;
      return true;
    };
    const uint64_t pol_first = policy_evict_first();
    const int m = P.m;
    int claim = atomicAdd(P.status + 2, 1);
    for (uint32_t q = 0;; ++q) {
      const int g = P.g_begin + claim;
      uint64_t *bar = &sh->full[w][q & 1], *bar3 = &sh->third[w][q & 1];
      // The end: once all threads are through all tiles, the word and the barrier are free.
      if (g >= P.g_end) {
        if (!wait_through(sh, w, q, P)) return;
        sh->tile[w][q & 1] = make_int4(-1, 0, 0, 0);
        mbar_arrive(bar);
        return;
      }
      claim = atomicAdd(P.status + 2, 1);    // the next one's comes back under this one's loads
      const int grp = g / per_group, p = (g - grp * per_group) / tpg, local = g - grp * per_group - p * tpg;
      const int h_in = local / P.tiles_per_head;
      const Tile t = tile_of(P, p, grp * hpg + h_in, (local - h_in * P.tiles_per_head) * kBlocks);
      const int* counter = P.counters + (t.p - 1) * P.BH + t.h;
      bool ready = t.p == 0 || !P.check_deps || ld_acquire(counter) >= P.tiles_per_head;
      auto depend = [&]() {                  // the head's half-step before has been stored
        if (!ready) {
          const long long t0 = clock64();
          while (ld_acquire(counter) < P.tiles_per_head) {
            if (sh->abort_flag) return false;
            if (clock64() - t0 > P.wait_cycles) {
              report_timeout(P.report, 10);
              sh->abort_flag = 1;
              return false;
            }
            __nanosleep(100);
          }
          ready = true;
        }
        asm volatile("fence.proxy.async.global;" ::: "memory");
        return true;
      };
      auto describe = [&]() { sh->tile[w][q & 1] = make_int4(t.p, t.h, t.idx0, 0); };
      uint8_t *s0 = smem + x.x0 * kSlot, *s1 = smem + x.x1 * kSlot, *s2 = smem + x.x2 * kSlot;
      const int xin = (EXTRA && P.H) ? (t.h % P.H) * kD : 0, hin = (EXTRA && P.H) ? t.h / P.H : t.h;
      if (t.isR) {
        const int row0 = (t.h * m + t.idx0) * B, row_in = (hin * m + t.idx0) * B;
        if (!take(x.x0) || !take(x.x1)) return;
        describe();
        mbar_expect_tx(bar, 2 * kSlot);
        tma_load_2d_hint(s1, &P.tmK, bar, xin, row_in, pol_first);
        if (t.first) {
          tma_load_2d(s0, &P.tmQ, bar, xin, row_in);
        } else {
          if (!depend()) return;
          tma_load_2d(s0, &P.tmAR, bar, 0, row0);
        }
        if (t.withV) {
          if (!take(x.x2)) return;
          mbar_expect_tx(bar3, kSlot);
          tma_load_2d_hint(s2, &P.tmV, bar3, xin, row_in, pol_first);
        }
      } else {
        const int row0 = (t.h * B + t.idx0) * m;
        if (!take(x.x0)) return;
        describe();
        mbar_expect_tx(bar, 2 * kSlot + 512);
        tma_load_3d(s0, &P.tmQs, bar, xin, hin * m, t.idx0);
        if (!take(x.x1) || !depend()) return;
        tma_load_2d(s1, &P.tmAL, bar, 0, row0);
        bulk_load_1d(reinterpret_cast<float*>(smem + kOffVec) + (2 * w + (q & 1)) * 128, P.cL + row0, 512, bar);
        if (t.final_) {
          if (!take(x.x2)) return;
          mbar_expect_tx(bar3, kSlot);
          tma_load_2d(s2, &P.tmY, bar3, 0, row0);
        } else if (B == 128) {                 // weights alone
          if (!take(x.x2)) return;
          mbar_arrive(bar3);
        }
      }
      x.next(t.isR, uses_third(t));
    }
  }

  // ================================================================ store warp of group w (its first lane)
  static __device__ __forceinline__ void store(const Params& P, uint8_t* smem, Shared* sh, int w) {
    const uint64_t pol_first = policy_evict_first();
    const bool lane0 = (threadIdx.x & 31) == 0;
    for (;;) {
      bar_sync(kStaged + w, 160);
      const int4 o = sh->out[w];
      __syncwarp();
      if (lane0) mbar_arrive(&sh->out_free[w]);
      if (o.x < 0) break;
      if (lane0) {
        const int slot = o.z & 15, rows = (o.z >> 4) & 15;
        const uint8_t* s = smem + slot * kSlot;
        if (rows == kAlphaL) tma_store_3d(&P.tmALs, s, 0, o.x * B, o.y);
        else if (rows == kY) tma_store_3d(&P.tmYs, s, 0, o.x * B, o.y);
        else if (rows == kAlphaR) tma_store_3d(&P.tmARs, s, 0, o.x * P.m, o.y);
        else tma_store_3d_hint(&P.tmOut, s, (EXTRA && P.H) ? (o.x % P.H) * kD : 0, ((EXTRA && P.H) ? o.x / P.H : o.x) * P.m, o.y, pol_first);
        tma_store_commit();
        tma_store_wait_read();
        mbar_arrive(&sh->empty[slot]);
        if (o.z >> 8) {                        // the tile's last rows: counted once they (and c_L) are in global memory
          tma_store_wait_all();
          asm volatile("fence.proxy.async.global;" ::: "memory");
          asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(P.counters + o.w * P.BH + o.x) : "memory");
        }
      }
      __syncwarp();
    }
    if (lane0) tma_store_wait_all();
  }

  // ================================================================ MMAs (one thread of the group's first warp)
  static __device__ __forceinline__ void apply(uint32_t d, uint32_t sX) {     // weights (TMEM) times the rows of a slot
    constexpr uint32_t id = instr_desc(B, 64, FT, 0, 1);
    const uint64_t dX = smem_desc(sX, 16, 1024);
#pragma unroll
    for (int t = 0; t < Geo<B>::kTiles; ++t) {
      const uint32_t lane = (uint32_t)(t * 16) << 16;
#pragma unroll
      for (int ks = 0; ks < B / 16; ++ks) {
        const uint64_t db = dX + (uint64_t)((t * (B * 128) + ks * 2048) >> 4);
        if (ks == 0) umma_ts<false>(d + lane + 64, d + lane, db, id);
        else umma_ts<true>(d + lane + 64, d + lane + 8 * ks, db, id);
      }
    }
  }
  // Rows k of sum_l P[l, k] [Q(l, .) | 1]: the ones are a second 64-column chunk of the B operand, whose distance shrinks as
  // the address walks down the rows of Q.
  static __device__ __forceinline__ void apply_transposed(uint32_t d, uint32_t sP, uint32_t chunk, uint32_t sQ, uint32_t sOnes) {
    constexpr uint32_t id = instr_desc(B, 80, FT, 1, 1);
    const uint64_t dP = smem_desc(sP, chunk, 1024);
#pragma unroll
    for (int t = 0; t < Geo<B>::kTiles; ++t)
#pragma unroll
      for (int ks = 0; ks < B / 16; ++ks) {
        const uint32_t off = t * (B * 128) + ks * 2048;
        const uint64_t db = smem_desc(sQ + off, sOnes - sQ - off, 1024);
        if (ks == 0) umma_c<false>(d + ((uint32_t)(t * 16) << 16) + 48, dP + (off >> 4), db, id);
        else umma_c<true>(d + ((uint32_t)(t * 16) << 16) + 48, dP + (off >> 4), db, id);
      }
  }

  // ================================================================ compute group w (thread = score row)
  static __device__ __forceinline__ void compute(const Params& P, uint8_t* smem, Shared* sh, uint32_t tmem, int warp_of_cta) {
    const int t_row = threadIdx.x & 127, warp = warp_of_cta & 3, w = warp_of_cta >> 2;
    const int blk = Geo<B>::tile(t_row), r = Geo<B>::row(t_row), srow = blk * B + r;
    const uint32_t d = tmem + 128 * w, tS = d + ((uint32_t)(warp * 32) << 16);
    const uint32_t sm = smem_u32(smem);
    const int m = P.m;
    constexpr int NC = B / 16;
    Slots<B> x(w);
    uint32_t par_1 = 0;
    uint32_t par_3 = 0;                        // bit i: parity of third[w][i]
    Group<Shared, Params> group(sh, P, w, warp, t_row);
    for (uint32_t q = 0;; ++q) {
      const uint32_t par = q & 1;
      const uint32_t a0 = sm + x.x0 * kSlot, a1 = sm + x.x1 * kSlot, a2 = sm + x.x2 * kSlot;
      bool more = true;
      if (warp == 0) {
        group.begin(q);
        group.await(&sh->full[w][q & 1], (q >> 1) & 1, 30);
        const int4 it = sh->tile[w][q & 1];
        more = group.ok && it.x >= 0;
        if (more) {
          const Tile t = tile_of(P, it.x, it.y, it.z);
          if (elect_one()) {
            issue_scores<B, FT>(d, a0, a1, P.negate);
            umma_commit(&sh->mma1[w]);
            if (t.isR || t.final_) umma_commit(&sh->empty[x.x0]);
            if (t.final_) umma_commit(&sh->empty[x.x1]);
          }
          __syncwarp();
          group.await(&sh->mma1[w], par, 31);
          more = group.ok;
        }
      }
      if (!group.release(more)) break;
      const int4 it = sh->tile[w][q & 1];
      const Tile t = tile_of(P, it.x, it.y, it.z);
      // the state rows the score MMA consumed are read exactly once: drop them from L2
      if (!t.isR) discard_line(P.aL + ((size_t)(t.h * B + t.idx0) * m + t_row) * 128);
      else if (!t.first) discard_line(P.aR + ((size_t)(t.h * m + t.idx0) * B + t_row) * 128);
      const float f = P.scale * kLog2e;
      float2 s2[2] = {both(0.f), both(0.f)};
      float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
      float c[2][16];
      float mul;                               // of the rows in the epilogue
      if (t.isR) {
        // Z_R = scale S (Eq. 7; alpha_R arrives divided by c_R), -c_L log2 e = log2 sum + max - sum R z (Eq. 10)
        int lim = B;                           // keys of the block that count (App. C.3)
        if (MASK && P.n_valid != 0 && t.idx0 + blk == m - 1) lim = P.n_valid - (m - 1) * B;
        float2 z2[2] = {both(0.f), both(0.f)};
        tmem_ld16(tS, c[0]);
#pragma unroll
        for (int cc = 0; cc < NC; ++cc) {
          float* cur = c[cc & 1];
          tmem_ld_wait();
          tmem_ld16(tS + 16 * ((cc + 1) % NC), c[(cc + 1) & 1]);      // wraps to the first chunk of pass 2
          if (MASK && lim < B) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (16 * cc + i >= lim) cur[i] = -INFINITY;
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) m4[i & 3] = max3(m4[i & 3], cur[2 * i], cur[2 * i + 1]);
        }
        const float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
        const float2 f2 = both(f), off2 = both(-mx * f);
#pragma unroll
        for (int cc = 0; cc < NC; ++cc) {
          float* cur = c[cc & 1];
          tmem_ld_wait();
          if (cc + 1 < NC) tmem_ld16(tS + 16 * (cc + 1), c[(cc + 1) & 1]);
          uint32_t u[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            float2 v = make_float2(cur[2 * i], cur[2 * i + 1]);
            if (MASK && lim < B) {            // masked keys: score 0 (any finite value), weight 0 below
              if (16 * cc + 2 * i >= lim) v.x = 0.f;
              if (16 * cc + 2 * i + 1 >= lim) v.y = 0.f;
            }
            const float2 e = ffma2(v, f2, off2);
            float2 p = make_float2(fast_exp2(e.x), fast_exp2(e.y));
            if (MASK && lim < B) {
              if (16 * cc + 2 * i >= lim) p.x = 0.f;
              if (16 * cc + 2 * i + 1 >= lim) p.y = 0.f;
            }
            z2[i & 1] = ffma2(p, v, z2[i & 1]);
            s2[i & 1] = fadd2(s2[i & 1], p);
            u[i] = pack2<T>(p.x, p.y);
          }
          st_cols<8>(tS + 8 * cc, u);          // over columns of the scores already read
        }
        const float sum = (s2[0].x + s2[0].y) + (s2[1].x + s2[1].y);
        const float sz = (z2[0].x + z2[0].y) + (z2[1].x + z2[1].y);
        mul = 1.f / sum;
        P.cL[((size_t)t.h * B + r) * m + t.idx0 + blk] = fast_log2(sum) - f * (sz * mul - mx);
        tmem_st_wait();
      } else {
        // Z_L = scale S' - c_L (Eq. 8), softmax over the blocks: logits back over the scores, then weights
        const float* cv = reinterpret_cast<const float*>(smem + kOffVec) + (2 * w + (q & 1)) * 128 + blk * B;
        const float2 f2 = both(f);
        tmem_ld16(tS, c[0]);
#pragma unroll
        for (int cc = 0; cc < NC; ++cc) {
          float* cur = c[cc & 1];
          tmem_ld_wait();
          if (cc + 1 < NC) tmem_ld16(tS + 16 * (cc + 1), c[(cc + 1) & 1]);
          const float4* cv4 = reinterpret_cast<const float4*>(cv + 16 * cc);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 k4 = cv4[i];
            const float2 za = ffma2(make_float2(cur[4 * i], cur[4 * i + 1]), f2, make_float2(k4.x, k4.y));
            const float2 zb = ffma2(make_float2(cur[4 * i + 2], cur[4 * i + 3]), f2, make_float2(k4.z, k4.w));
            m4[0] = max3(m4[0], za.x, za.y);
            m4[1] = max3(m4[1], zb.x, zb.y);
            cur[4 * i] = za.x; cur[4 * i + 1] = za.y; cur[4 * i + 2] = zb.x; cur[4 * i + 3] = zb.y;
          }
          tmem_st16(tS + 16 * cc, cur);
        }
        const float mx = fmaxf(m4[0], m4[1]);
        const float2 nmx2 = both(-mx);
        tmem_st_wait();
        tmem_ld16(tS, c[0]);
#pragma unroll
        for (int cc = 0; cc < NC; ++cc) {
          float* cur = c[cc & 1];
          tmem_ld_wait();
          if (cc + 1 < NC) tmem_ld16(tS + 16 * (cc + 1), c[(cc + 1) & 1]);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float2 e = fadd2(make_float2(cur[2 * i], cur[2 * i + 1]), nmx2);
            const float2 p = make_float2(fast_exp2(e.x), fast_exp2(e.y));
            s2[i & 1] = fadd2(s2[i & 1], p);
            cur[2 * i] = p.x;
            cur[2 * i + 1] = p.y;
          }
          if (t.final_) {
            uint32_t u[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) u[i] = pack2<T>(cur[2 * i], cur[2 * i + 1]);
            st_cols<8>(tS + 8 * cc, u);
          } else {
            tmem_st16(tS + 16 * cc, cur);
          }
        }
        tmem_st_wait();
        const float sum = (s2[0].x + s2[0].y) + (s2[1].x + s2[1].y);
        mul = 1.f / sum;
        // Row b l + j (l = r, j = idx0 + blk) of the final L half-step: its log-sum-exp; summed over
        // the rows of a head it is the value of the objective (Eq. 6) at the returned matrix.
        if (EXTRA && t.final_ && P.lse != nullptr)
          P.lse[(size_t)t.h * (B * m) + (size_t)r * B + t.idx0 + blk] = (mx + fast_log2(sum)) * kLn2;
        if (!t.final_) {
          // the contraction runs over the rows of the weights: normalised in fp32, rounded once, to shared memory
          const float2 n2 = both(mul * kWeightScale);
          // (128 columns: the slot of the second half is free; every warp looks for itself)
          if (B == 128) group.await(&sh->third[w][q & 1], (par_3 >> (q & 1)) & 1, 36);
          uint8_t* lower = smem + (B == 128 ? min(x.x1, x.x2) : x.x1) * kSlot + srow * 128;
          uint8_t* upper = smem + max(x.x1, x.x2) * kSlot + srow * 128;
          tmem_ld16(tS, c[0]);
#pragma unroll
          for (int cc = 0; cc < NC; ++cc) {
            float* cur = c[cc & 1];
            tmem_ld_wait();
            if (cc + 1 < NC) tmem_ld16(tS + 16 * (cc + 1), c[(cc + 1) & 1]);
            uint32_t u[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float2 v = fmul2(make_float2(cur[2 * i], cur[2 * i + 1]), n2);
              u[i] = pack2<T>(v.x, v.y);
            }
            const int c0 = 2 * cc & 7;
            uint8_t* base = cc < 4 ? lower : upper;
            *reinterpret_cast<uint4*>(base + ((c0 ^ (srow & 7)) << 4)) = make_uint4(u[0], u[1], u[2], u[3]);
            *reinterpret_cast<uint4*>(base + (((c0 + 1) ^ (srow & 7)) << 4)) = make_uint4(u[4], u[5], u[6], u[7]);
          }
          fence_proxy_async();
        }
      }
      group.collect();
      const bool third = uses_third(t) || (B == 128 && !t.isR);
      if (warp == 0) {
        if (t.final_) group.await(&sh->third[w][q & 1], (par_3 >> (q & 1)) & 1, 36);
        if (group.ok && elect_one()) {
          if (t.isR) {
            apply(d, a1);
            umma_commit(t.withV ? &sh->first[w] : &sh->mma2[w]);
          } else if (t.final_) {
            apply(d, a2);
            umma_commit(&sh->mma2[w]);
          } else {
            // (128 columns of weights: the first 64 in the lower of the two slots)
            if (B == 128) apply_transposed(d, min(a1, a2), max(a1, a2) - min(a1, a2), a0, sm + kOffOnes);
            else apply_transposed(d, a1, kSlot, a0, sm + kOffOnes);
            umma_commit(&sh->mma2[w]);
            umma_commit(&sh->empty[x.x1]);
            if (B == 128) umma_commit(&sh->empty[x.x2]);
          }
        }
        __syncwarp();
      }
      // ============================================================== rows
      float o[64];
      if (t.isR && t.withV) {                  // alpha_L, over K; then y = R V through the same columns, over V
        if (!group.await_rows(&sh->first[w], par_1, 32)) break;
        par_1 ^= 1;
        tmem_ld32(tS + 64, o);
        tmem_ld32(tS + 96, o + 32);
        tmem_ld_wait();
        group.collect();
        if (warp == 0) {
          group.await(&sh->third[w][q & 1], (par_3 >> (q & 1)) & 1, 36);
          if (group.ok && elect_one()) {
            apply(d, a2);
            umma_commit(&sh->mma2[w]);
          }
          __syncwarp();
        }
        store_row32<T>(smem + x.x1 * kSlot, srow, 0, o, mul);
        store_row32<T>(smem + x.x1 * kSlot, srow, 32, o + 32, mul);
        fence_proxy_async();
        group.hand_over(t.h, t.idx0, x.x1 | kAlphaL << 4, t.p);
      }
      if (!group.await_rows(&sh->mma2[w], par, 33)) break;
      if (t.final_) discard_line(P.y + ((size_t)(t.h * B + t.idx0) * m + t_row) * 128);
      const bool turned = !t.isR && !t.final_;
      float cr = 1.f;
      if (turned) cr = ld_col(tS + 112);
      const uint32_t tO = tS + (turned ? 48 : 64);
      tmem_ld32(tO, o);
      tmem_ld32(tO + 32, o + 32);
      tmem_ld_wait();
      group.leave();
      if (turned) mul = cr > 1e-30f ? 1.f / cr : 0.f;
      const int slot = t.isR ? (t.withV ? x.x2 : x.x1) : (t.final_ ? x.x2 : x.x0);
      store_row32<T>(smem + slot * kSlot, srow, 0, o, mul);
      store_row32<T>(smem + slot * kSlot, srow, 32, o + 32, mul);
      fence_proxy_async();
      group.hand_over(t.h, t.idx0, slot | (t.isR ? (t.withV ? kY : kAlphaL) : (t.final_ ? kOut : kAlphaR)) << 4 | 1 << 8, t.p);
      if (third) par_3 ^= 1u << (q & 1);
      x.next(t.isR, uses_third(t));
    }
    group.finish();
  }
};

template <typename T, int B, int EXTRA>
__global__ void __launch_bounds__(kThreads, kCtasPerSm) monarch_chain(const __grid_constant__ Params P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align_smem<1024>(smem_raw);
  Shared* sh = reinterpret_cast<Shared*>(smem + kOffBar);
  const int tid = threadIdx.x, warp = warp_of_cta();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (tid == 0) {
    for (int i = 0; i < kSlots; ++i) mbar_init(&sh->empty[i], 1);
    for (int w = 0; w < 2; ++w) {
      for (int i = 0; i < 2; ++i) {
        mbar_init(&sh->full[w][i], 1);
        mbar_init(&sh->third[w][i], 1);
      }
      mbar_init(&sh->mma1[w], 1);
      mbar_init(&sh->first[w], 1);
      mbar_init(&sh->mma2[w], 1);
      mbar_init(&sh->out_free[w], 1);
      sh->through[w] = 0;
    }
    sh->abort_flag = 0;
    fence_barrier_init();
  }
  if (tid < 128) {
    const uint32_t one2 = pack2<T>(1.f, 1.f);
    *reinterpret_cast<uint4*>(smem + kOffOnes + tid * 16) = make_uint4(one2, one2, one2, one2);
  }
  if (warp == 8) tmem_alloc(&sh->tmem, 256);
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, sh->tmem, 0);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  using C = Chain<T, B, EXTRA>;
  // registers: 384 threads at the launch's 80; 128 x 64 + 256 x 88 make use of all of them (nothing is spilled; with 48 the producers spill)
  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    if (warp >= 10) C::store(P, smem, sh, warp - 10);
    else if (elect_one()) C::produce(P, smem, sh, warp - 8);
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 88;");
    C::compute(P, smem, sh, tmem, warp);
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (sh->abort_flag) {                 // what is in flight lands before the CTA leaves
    let_copies_land();
    __syncthreads();
  }
  if (warp == 8) tmem_dealloc(tmem, 256);
  if (tid == 0) {                       // the last CTA re-arms the dependency counters and the tile counter
    __threadfence();
    if (atomicAdd(P.status + 1, 1) == (int)gridDim.x - 1) {
      for (int i = 0; i < P.n_counters; ++i) P.counters[i] = 0;
      P.status[1] = P.status[2] = 0;
    }
  }
}

template <typename T, int B, int EXTRA>
inline cudaError_t launch_kernel(const Params& P, int grid, cudaStream_t st) {
  auto kern = monarch_chain<T, B, EXTRA>;
  static bool prepared[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!prepared[dev]) {
    e = cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e != cudaSuccess) return e;
    prepared[dev] = true;
  }
  // (the next call's CTAs set up while the last tiles of this one are on their way)
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, P);
}

}  // namespace tp3

namespace tp {
template <typename T, int B>
cudaError_t launch_chain(const Params& P, int grid, cudaStream_t st) {
  if (P.n_valid != 0) return tp3::launch_kernel<T, B, 2>(P, grid, st);
  if (P.H != 0 || P.lse != nullptr) return tp3::launch_kernel<T, B, 1>(P, grid, st);
  return tp3::launch_kernel<T, B, 0>(P, grid, st);
}
#ifdef MA_TU_TENSOR_CHAIN
template cudaError_t launch_chain<__half, 64>(const Params&, int, cudaStream_t);
template cudaError_t launch_chain<__half, 128>(const Params&, int, cudaStream_t);
template cudaError_t launch_chain<__nv_bfloat16, 64>(const Params&, int, cudaStream_t);
template cudaError_t launch_chain<__nv_bfloat16, 128>(const Params&, int, cudaStream_t);
#endif
}  // namespace tp
}  // namespace ma
