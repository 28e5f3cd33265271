// Tensor-core tiles of both half-steps for sm_100a (tcgen05 + TMA), one launch per half-step: 16-bit
// inputs, d <= 64 (a multiple of 8), any b, m <= 128, key padding mask and per-sequence lengths (App.
// C.3), either layout, row log-sum-exp output.  MA_PATH_TILE_MMA takes these kernels for up to two
// rounds where there are tiles enough, and full enough, to pay for their longer chain (the rule is in api.cu).
//
// What bounds a tile.  Its chain load -> score MMA -> softmax -> apply MMA -> epilogue -> store is mostly
// latency (a launch with less than a tile a compute group takes 9 us), while its pipe time is
// half a microsecond (128 x 128 exponentials at 16 per clock and SM).  So as many chains as possible have to be in flight with as few hand-overs as
// possible: two CTAs share an SM, each with two compute groups of four warps (thread = score row, one tile per group: softmax and
// epilogue).  A group has three 16 KB slots, a producer thread and a store warp of its own; its first warp issues its MMAs, and
// hand-overs inside a group are hardware barriers.  The producers ask for inputs (Q, K, V) before the half-step before has ended.
// (With a ring of slots and a polling MMA thread shared by the groups, and loads that all waited: 8 heads of 7600, T = 2 39.5 us, now
// 35.3; 48 of 47 x 64 83.4 / 75.6; 16 of 94 x 128, T = 1 54.2 / 56.4, the only one that lost: a whole tile was requested ahead there.)
//
// One tile shape for everything: 128 score rows = 128 / B blocks of B rows (B = b or m rounded up
// to 32, 64 or 128; rows past the block are zero-filled by TMA), one M = N = 128 score MMA, of which a
// row owns the B columns of its own block (at B = 64 the wasted half costs no time: M = 64 MMAs run
// at half rate).  The weights go back to tensor memory over the scores, zeros outside the window,
// and are the A operand of the apply MMA; only the non-final L half-step, whose contraction runs
// over the rows of the weights, passes them through shared memory.
//   TMEM columns of a group: scores 0-127; weights (16-bit pairs) 0-63; apply accumulator 64-127; in
//   the non-final L half-step sixteen copies of c_R in 0-15.
//
// Arithmetic and states are f16 (bf16 inputs are converted in shared memory: the rounding of alpha_L
// is the dominant error of a 16-bit pipeline and f16 has three more bits).  alpha_R is stored divided
// by c_R, and the columns of the non-final L weights are rescaled by powers of two before they are
// rounded (the quotient is invariant), so that a column of small weights keeps its bits however small
// c_R is; c_R sums the weights as rounded.
//
// Measured when they came (B200, us per call, against the warp-MMA tiles that served these shapes): 8 heads of N =
// 7600 in blocks of 128, d = 48, two rounds 43.9 / 61.9; 32 heads of N = 8192 as 128 blocks of 64, one
// round (bf16) 64 / 95, two rounds (f16) 119 / 214; 64 heads of 60 blocks of 64, two rounds 102 / 150.
#pragma once
#include <type_traits>

#include "status_word.cuh"
#include "tile_group.cuh"

namespace ma {
namespace ttc {

using namespace ma::group;

constexpr int kThreads = 384;                // two compute groups of four warps, four service warps
constexpr int kCtasPerSm = 2;
constexpr int kSlot = kTileBytes;            // 16 KB
constexpr int kSlots = 6;
constexpr int kOffOnes = kSlots * kSlot;     // 2 KB of ones
constexpr int kOffVec = kOffOnes + 2048;     // c_L of a tile's rows: two tiles of 128 floats a group
constexpr int kOffCol = kOffVec + 4 * 512;   // per group, two sets in turn: column maxima of the non-final L weights
constexpr int kOffBar = kOffCol + 4 * 512;
constexpr int kSmem = kOffBar + 384 + 1024;  // + alignment slack
static_assert(kCtasPerSm * (kSmem + 1024) <= 228 * 1024, "two CTAs per SM");

struct Params {
  // Loads and stores of one tile, all with 64-column rows and 128 rows in 128-byte swizzle.
  // R: dims (d, b, m, heads, batch), box (64, B, 128 / B, 1, 1): blocks of rows (k, .)
  // L: dims (d, m, b, heads, batch), box (64, B, 128 / B, 1, 1): blocks of rows (., j)
  CUtensorMap rQ, rK, rV, rAR, rAL, rY;      // R half-step: loads Q, K, V, alpha_R; stores alpha_L, y
  CUtensorMap lQ, lAL, lY, lAR, lOut;        // L half-step: loads Q, alpha_L, y; stores alpha_R, Y
  float* cL;               // [BH][b][mp]: -c_L log2 e, the addend of the next L half-step's logits
  uint8_t *aL, *aR, *y;    // state arrays, for L2 discards once a tile has been consumed (d = 64)
  float* lse;              // optional [BH][N]
  const int* seq_len;      // optional [BH / heads]
  int* report;             // status word, set by a wait that ran out
  int* clear;              // status word to clear first, or nullptr
  int N, b, m, mp, BH, H, heads, n_valid;
  int first, last;         // this launch's half-step: of the first round, of the last round
  int tiles, per_head;     // tiles of this launch, tiles of a head
  int discard;
  long long wait_cycles;
  float scale;
};

struct __align__(16) Shared {
  uint64_t full[2][2], third[2][2];                    // by group, tiles in turn: first two operands, third slot
  uint64_t empty[kSlots];
  uint64_t mma1[2], first[2], mma2[2], out_free[2];      // by group from here on
  int4 tile[2][2];           // {head or -1, first block or position, keys that count}
  int4 out[2];               // {head or -1, first block or position, slot, is y}
  int through[2];            // tiles of a group that have left tensor memory
  int taken;                 // tiles of the CTA that its groups have taken
  uint32_t tmem;
  volatile int abort_flag;
};
static_assert(sizeof(Shared) <= 384, "barrier block");

__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ------------------------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ void load_5d(void* dst, const CUtensorMap* tm, uint64_t* bar, int r, int blk, int h0, int h1) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(
          smem_u32(dst)),
      "l"((uint64_t)tm), "r"(smem_u32(bar)), "r"(0), "r"(r), "r"(blk), "r"(h0), "r"(h1)
      : "memory");
}
__device__ __forceinline__ void store_5d(const CUtensorMap* tm, const void* src, int blk, int h0, int h1) {
  asm volatile("cp.async.bulk.tensor.5d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5, %6}], [%1];" ::"l"((uint64_t)tm),
               "r"(smem_u32(src)), "r"(0), "r"(0), "r"(blk), "r"(h0), "r"(h1)
               : "memory");
}
__device__ __forceinline__ void bulk_1d(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
template <int N>
__device__ __forceinline__ void st_cols(uint32_t taddr, const uint32_t* r);
template <>
__device__ __forceinline__ void st_cols<8>(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
template <>
__device__ __forceinline__ void st_cols<16>(uint32_t taddr, const uint32_t* r) {
  tmem_st16(taddr, reinterpret_cast<const float*>(r));
}
template <>
__device__ __forceinline__ void st_cols<32>(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, "
      "%30, %31, %32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
      "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
      "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
// 32 rows x 32 columns of the warp's part of tensor memory as matrix fragments: v[16 h + 4 o + 2 q + e] is row
// 16 h + 8 q + lane / 4, column 8 o + 2 (lane % 4) + e.
__device__ __forceinline__ void ld_frag16(uint32_t taddr, float* v) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void ld_frag32(uint32_t taddr, float* v) {
  ld_frag16(taddr, v);
  ld_frag16(taddr + (16u << 16), v + 16);
}
__device__ __forceinline__ void stmatrix_x4(uint32_t saddr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(saddr), "r"(a), "r"(b), "r"(c), "r"(d)
               : "memory");
}
__device__ __forceinline__ float ld_col(uint32_t taddr) {
  uint32_t r;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr) : "memory");
  return __uint_as_float(r);
}
template <bool ACC>
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "n"(ACC ? 1 : 0)
      : "memory");
}

__device__ __forceinline__ void arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// ------------------------------------------------------------------------------------ kernel
// MODE 0: R tiles, 1: L tiles of blocks (rows of blocks) padded to B.  FULL: nothing is padded or masked.
template <typename TIn, int B, bool FULL, int MODE>
struct Kernel {
  typedef __half TA;                    // arithmetic and states
  static constexpr bool kConvert = !std::is_same<TIn, TA>::value;
  static constexpr bool R = MODE == 0;
  static constexpr int kBlocks = 128 / B;
  static constexpr int FT = Fmt<TA>::code;
  static constexpr uint32_t kIdScore = instr_desc(128, 128, FT, 0, 0), kIdApply = instr_desc(128, 64, FT, 0, 1);

  static __device__ __forceinline__ bool prepares(const Params& P) { return kConvert || (!FULL && P.seq_len != nullptr); }

  // ================================================================ producer of group w (one thread)
  // The groups of a CTA take its tiles in turn, each when it has slots for one.  Q, K, V and the lengths are asked for before the end of the
  // half-step before (the first launch of a call lets the next ones start only once it has waited for whatever wrote them).
  static __device__ __forceinline__ void produce(const Params& P, uint8_t* smem, Shared* sh, int w) {
    const bool last = P.last != 0;
    bool waited = R && P.first;
    if (waited) {
      grid_wait();
      grid_launch_dependents();
    }
    Slots<B> x(w);
    uint32_t busy = 0, par = 0;               // by slot: a use is to be waited for; parity of that wait
    auto take = [&](int s) {
      const uint32_t bit = 1u << s;
      if ((busy & bit) && !wait_bar(&sh->empty[s], (par & bit) != 0, sh, P, 11)) return false;
      if (busy & bit) par ^= bit;
      busy |= bit;
      return true;
    };
    for (uint32_t q = 0;; ++q) {
      uint64_t *bar = &sh->full[w][q & 1], *bar3 = &sh->third[w][q & 1];
      int h, idx0, n_valid = P.n_valid;
      bool end;
      do {
        const int g = blockIdx.x + atomicAdd(&sh->taken, 1) * gridDim.x;
        end = g >= P.tiles;
        h = end ? -1 : g / P.per_head;
        idx0 = end ? 0 : (g - h * P.per_head) * kBlocks;
        if (!FULL && !end && P.seq_len != nullptr) n_valid = min(max(P.seq_len[h / P.heads], 1), P.N);
      } while (!FULL && R && !end && P.seq_len != nullptr && idx0 * P.b >= n_valid);      // key blocks that a shorter sequence does not have
      // The end: once all threads are through all tiles, the word and the barrier are free.
      if (end) {
        if (!wait_through(sh, w, q, P)) return;
        sh->tile[w][q & 1] = make_int4(-1, 0, 0, 0);
        arrive(bar);
        return;
      }
      if (!take(x.x0) || !take(x.x1)) return;
      sh->tile[w][q & 1] = make_int4(h, idx0, n_valid, 0);
      const int h0 = P.H ? h % P.H : h, h1 = P.H ? h / P.H : 0;
      uint8_t *s0 = smem + x.x0 * kSlot, *s1 = smem + x.x1 * kSlot, *s2 = smem + x.x2 * kSlot;
      if (R) {
        const bool v_first = last && !waited;      // (its slot is free then)
        auto load_v = [&]() {
          if (!take(x.x2)) return false;
          mbar_expect_tx(bar3, kSlot);
          load_5d(s2, &P.rV, bar3, 0, idx0, h0, h1);
          return true;
        };
        mbar_expect_tx(bar, 2 * kSlot);
        load_5d(s1, &P.rK, bar, 0, idx0, h0, h1);
        if (v_first && !load_v()) return;
        if (!waited) grid_wait();
        if (P.first) load_5d(s0, &P.rQ, bar, 0, idx0, h0, h1);
        else load_5d(s0, &P.rAR, bar, 0, idx0, h, 0);
        if (last && !v_first && !load_v()) return;
      } else {
        float* sC = reinterpret_cast<float*>(smem + kOffVec) + (2 * w + (q & 1)) * 128;
        const int nj = min(kBlocks, P.b - idx0);
        mbar_expect_tx(bar, 2 * kSlot + nj * P.mp * 4);
        load_5d(s0, &P.lQ, bar, 0, idx0, h0, h1);
        if (!waited) grid_wait();
        load_5d(s1, &P.lAL, bar, 0, idx0, h, 0);
        const float* c = P.cL + ((size_t)h * P.b + idx0) * P.mp;
        for (int jj = 0; jj < nj; ++jj) bulk_1d(sC + jj * B, c + (size_t)jj * P.mp, P.mp * 4, bar);
        if (last || B == 128) {
          if (!take(x.x2)) return;
          if (last) {
            mbar_expect_tx(bar3, kSlot);
            load_5d(s2, &P.lY, bar3, 0, idx0, h, 0);
          } else {
            arrive(bar3);                     // for weights
          }
        }
      }
      waited = true;
      x.next(R, last);
    }
  }

  // ================================================================ store warp of group w (its first lane)
  // Stores what the group has staged; sh->out[w] says what and where.
  static __device__ __forceinline__ void store(const Params& P, uint8_t* smem, Shared* sh, int w) {
    const bool lane0 = (threadIdx.x & 31) == 0;
    for (;;) {
      bar_sync(kStaged + w, 160);
      const int4 o = sh->out[w];          // head, first block or position, slot, y?
      __syncwarp();
      if (lane0) arrive(&sh->out_free[w]);
      if (o.x < 0) break;
      if (lane0) {
        const uint8_t* s = smem + o.z * kSlot;
        if (R) store_5d(o.w ? &P.rY : &P.rAL, s, o.y, o.x, 0);
        else if (!P.last) store_5d(&P.lAR, s, o.y, o.x, 0);
        else store_5d(&P.lOut, s, o.y, P.H ? o.x % P.H : o.x, P.H ? o.x / P.H : 0);
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        arrive(&sh->empty[o.z]);
      }
      __syncwarp();
    }
    if (lane0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }

  // ================================================================ MMAs (one thread of the group's first warp)
  static __device__ __forceinline__ void scores(uint32_t d, const uint8_t* s0, const uint8_t* s1) {
    const uint64_t da = smem_desc(smem_u32(s0), 16, 1024), db = smem_desc(smem_u32(s1), 16, 1024);
    umma_c<false>(d, da, db, kIdScore);
    umma_c<true>(d, da + 2, db + 2, kIdScore);
    umma_c<true>(d, da + 4, db + 4, kIdScore);
    umma_c<true>(d, da + 6, db + 6, kIdScore);
  }
  static __device__ __forceinline__ void apply(uint32_t d, const uint8_t* x) {     // weights (TMEM) times the rows of a slot
    const uint64_t dX = smem_desc(smem_u32(x), 16, 1024);
    umma_ts<false>(d + 64, d, dX, kIdApply);
#pragma unroll
    for (int ks = 1; ks < 8; ++ks) umma_ts<true>(d + 64, d + 8 * ks, dX + 128 * ks, kIdApply);
  }
  // Rows k of sum_l P[l, k] Q(l, .), and the sums of the weights against ones.  chunk: from the first 64 columns of P to the others.
  static __device__ __forceinline__ void apply_transposed(uint32_t d, const uint8_t* p, uint32_t chunk, const uint8_t* q, const uint8_t* ones) {
    const uint64_t dP = smem_desc(smem_u32(p), chunk, 1024), dQ = smem_desc(smem_u32(q), 16, 1024), dO = smem_desc(smem_u32(ones), 16, 1024);
    if constexpr (B == 128) {
      constexpr uint32_t id = instr_desc(128, 64, FT, 1, 1), id1 = instr_desc(128, 16, FT, 1, 0);
      umma_c<false>(d + 64, dP, dQ, id);
      umma_c<false>(d, dP, dO, id1);
#pragma unroll
      for (int ks = 1; ks < 8; ++ks) {
        umma_c<true>(d + 64, dP + 128 * ks, dQ + 128 * ks, id);
        umma_c<true>(d, dP + 128 * ks, dO, id1);
      }
    } else {
      // two groups of 64 rows; their accumulators take the lower and upper 16 lanes of
      // every warp's part of tensor memory
      constexpr uint32_t id = instr_desc(64, 64, FT, 1, 1), id1 = instr_desc(64, 16, FT, 1, 0);
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        const uint32_t dg = d + ((uint32_t)(16 * g) << 16);
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          const uint64_t off = 512 * g + 128 * ks;
          if (ks == 0) {
            umma_c<false>(dg + 64, dP + off, dQ + off, id);
            umma_c<false>(dg, dP + off, dO, id1);
          } else {
            umma_c<true>(dg + 64, dP + off, dQ + off, id);
            umma_c<true>(dg, dP + off, dO, id1);
          }
        }
      }
    }
  }

  // ================================================================ compute warps (thread = score row)
  // bf16 -> f16 in a slot, rows of absent blocks zeroed.
  static __device__ __forceinline__ void prepare(const Params& P, uint8_t* tile, bool convert, int idx0, int mv, int row) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int ch = q * 128 + row, r = ch >> 3;
      uint4* p = reinterpret_cast<uint4*>(tile + ch * 16);
      const bool absent = !FULL && P.seq_len != nullptr && (R ? idx0 + r / B >= mv : r % B >= mv);
      if (absent) {
        *p = make_uint4(0u, 0u, 0u, 0u);
      } else if (kConvert && convert) {
        uint4 v = *p;
        uint32_t* w = reinterpret_cast<uint32_t*>(&v);
#pragma unroll
        for (int e = 0; e < 4; ++e)     // a bf16 is the upper half of an fp32; saturates at +-65504
          asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;"
              : "=r"(w[e])
              : "f"(__uint_as_float(w[e] & 0xffff0000u)), "f"(__uint_as_float(w[e] << 16)));
        *p = v;
      }
    }
    fence_proxy_async();
  }
  // Zero weights beside the B columns of a row's own block, in tensor memory.
  static __device__ __forceinline__ void zeros_beside(uint32_t t_row, int r_blk) {
    if constexpr (B < 128) {
      uint32_t z[B / 2];
#pragma unroll
      for (int i = 0; i < B / 2; ++i) z[i] = 0u;
#pragma unroll
      for (int q = 1; q < 128 / B; ++q) st_cols<B / 2>(t_row + (B / 2) * ((r_blk + q) % (128 / B)), z);
    }
  }
  // CH scores of an R row: p = exp2(f s - f mx), sums of p and p s, packed weights.
  template <int CH>
  static __device__ __forceinline__ void r_weights(const float* s, int col0, int lim, float f, float off, float2* a2,
                                                   float2* z2, uint32_t* u) {
    if (FULL || lim >= col0 + CH) {
      const float2 f2 = make_float2(f, f), off2 = make_float2(off, off);
#pragma unroll
      for (int i = 0; i < CH / 2; ++i) {
        const float2 x = make_float2(s[2 * i], s[2 * i + 1]);
        const float2 z = ffma2(x, f2, off2);
        const float2 p = make_float2(fast_exp2(z.x), fast_exp2(z.y));
        z2[i & 1] = ffma2(p, x, z2[i & 1]);
        a2[i & 1] = fadd2(a2[i & 1], p);
        u[i] = pack2<TA>(p.x, p.y);
      }
    } else {       // keys past the block or past n_valid: weight 0
#pragma unroll
      for (int i = 0; i < CH / 2; ++i) {
        const bool v0 = col0 + 2 * i < lim, v1 = col0 + 2 * i + 1 < lim;
        const float p0 = v0 ? fast_exp2(fmaf(s[2 * i], f, off)) : 0.f, p1 = v1 ? fast_exp2(fmaf(s[2 * i + 1], f, off)) : 0.f;
        z2[i & 1].x = fmaf(p0, v0 ? s[2 * i] : 0.f, z2[i & 1].x);
        z2[i & 1].y = fmaf(p1, v1 ? s[2 * i + 1] : 0.f, z2[i & 1].y);
        a2[i & 1] = fadd2(a2[i & 1], make_float2(p0, p1));
        u[i] = pack2<TA>(p0, p1);
      }
    }
  }
  template <int CH>
  static __device__ __forceinline__ void mask(float* s, int col0, int lim) {
    if (!FULL && lim < col0 + CH) {
#pragma unroll
      for (int i = 0; i < CH; ++i)
        if (col0 + i >= lim) s[i] = -INFINITY;
    }
  }
  template <int CH>
  static __device__ __forceinline__ void fold_max(const float* s, float* m4) {
#pragma unroll
    for (int i = 0; i < CH / 2; ++i) m4[i & 3] = max3(m4[i & 3], s[2 * i], s[2 * i + 1]);
  }

  // R: softmax over the keys of the row's block (Eq. 7; alpha_R arrives divided by c_R), weights to
  // tensor memory, -c_L log2 e (Eq. 10) to global.  Returns 1 / sum.
  static __device__ __forceinline__ float r_softmax(const Params& P, int h, int k, int n_valid, uint32_t t_row, int r_blk, int r_pos) {
    const float f = P.scale * kLog2e;
    const uint32_t tS = t_row + B * r_blk;
    const int lim = FULL ? B : max(1, min(P.b, n_valid - k * P.b));      // keys of this block that count
    float2 a2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}, z2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
    float mx;
    if constexpr (B >= 64) {
      // two passes over the scores (a row does not fit the registers that four CTAs leave a thread), the
      // next chunk's load in flight
      {
        float x[32];
#pragma unroll
        for (int cc = 0; cc < B / 32; ++cc) {
          tmem_ld32(tS + 32 * cc, x);
          tmem_ld_wait();
          mask<32>(x, 32 * cc, lim);
          fold_max<32>(x, m4);
        }
      }
      float c16[2][16];
      tmem_ld16(tS, c16[0]);
      mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
#pragma unroll
      for (int cc = 0; cc < B / 16; ++cc) {
        tmem_ld_wait();
        if (cc < B / 16 - 1) tmem_ld16(tS + 16 * (cc + 1), c16[(cc + 1) & 1]);
        uint32_t u[8];
        r_weights<16>(c16[cc & 1], 16 * cc, lim, f, -mx * f, a2, z2, u);
        st_cols<8>(t_row + (B / 2) * r_blk + 8 * cc, u);       // over columns of the scores already read
      }
    } else {
      float x[B];
#pragma unroll
      for (int cc = 0; cc < B / 32; ++cc) tmem_ld32(tS + 32 * cc, x + 32 * cc);
      tmem_ld_wait();
      mask<B>(x, 0, lim);
      fold_max<B>(x, m4);
      mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
#pragma unroll
      for (int cc = 0; cc < B / 32; ++cc) {
        uint32_t u[16];
        r_weights<32>(x + 32 * cc, 32 * cc, lim, f, -mx * f, a2, z2, u);
        st_cols<16>(t_row + (B / 2) * r_blk + 16 * cc, u);
      }
    }
    zeros_beside(t_row, r_blk);
    const float sum = (a2[0].x + a2[0].y) + (a2[1].x + a2[1].y);
    const float sz = (z2[0].x + z2[0].y) + (z2[1].x + z2[1].y);
    const float inv_s = 1.f / sum;
    if (FULL || (r_pos < P.b && k < P.m))
      P.cL[((size_t)h * P.b + r_pos) * P.mp + k] = fast_log2(sum) - f * (sz * inv_s - mx);
    tmem_st_wait();
    return inv_s;
  }

  // CH scores of an L row to logits z = f s - c_L (Eq. 8), in place.
  template <int CH>
  static __device__ __forceinline__ void l_logits(float* s, const float* c, float f) {
    const float4* c4 = reinterpret_cast<const float4*>(c);
    const float2 f2 = make_float2(f, f);
#pragma unroll
    for (int i = 0; i < CH / 4; ++i) {
      const float4 k4 = c4[i];
      const float2 za = ffma2(make_float2(s[4 * i], s[4 * i + 1]), f2, make_float2(k4.x, k4.y));
      const float2 zb = ffma2(make_float2(s[4 * i + 2], s[4 * i + 3]), f2, make_float2(k4.z, k4.w));
      s[4 * i] = za.x; s[4 * i + 1] = za.y; s[4 * i + 2] = zb.x; s[4 * i + 3] = zb.y;
    }
  }
  // CH logits to weights exp2(z - mx), in place.
  template <int CH>
  static __device__ __forceinline__ void l_weights(float* z, float mx, float2* a2) {
    const float2 nmx2 = make_float2(-mx, -mx);
#pragma unroll
    for (int i = 0; i < CH / 2; ++i) {
      const float2 d = fadd2(make_float2(z[2 * i], z[2 * i + 1]), nmx2);
      const float2 p = make_float2(fast_exp2(d.x), fast_exp2(d.y));
      a2[i & 1] = fadd2(a2[i & 1], p);
      z[2 * i] = p.x;
      z[2 * i + 1] = p.y;
    }
  }
  template <int CH>
  static __device__ __forceinline__ void pack_cols(const float* v, uint32_t* u) {
#pragma unroll
    for (int i = 0; i < CH / 2; ++i) u[i] = pack2<TA>(v[2 * i], v[2 * i + 1]);
  }
  // Scale of a column of the non-final L weights: 2^-(exponent of its largest weight).
  static __device__ __forceinline__ float column_scale(unsigned mx) { return __uint_as_float((253u << 23) - (mx & 0x7f800000u)); }
  // A pair of a lane's weights in fragments (`x` of ld_frag32): column octet o, its i-th row.
  static __device__ __forceinline__ float2 frag_pair(const float* x, int o, int i) {
    const float* p = x + 16 * (i >> 1) + 4 * o + 2 * (i & 1);
    return make_float2(p[0], p[1]);
  }
  // Maxima of 32 columns over the warp's rows, to the shared maxima (weights are not negative: their bits are in
  // their order).  In fragments a lane has four rows of eight columns, and three exchanges finish it: one exchange for every
  // 4.6 columns instead of a warp-wide reduction for each.
  static __device__ __forceinline__ void fold_columns(const float* x, const float* on, unsigned* sMax, int lane) {
    unsigned a[8];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      a[2 * o] = a[2 * o + 1] = 0u;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 v = fmul2(frag_pair(x, o, i), make_float2(on[i], on[i]));
        a[2 * o] = max(a[2 * o], __float_as_uint(v.x));
        a[2 * o + 1] = max(a[2 * o + 1], __float_as_uint(v.y));
      }
    }
#pragma unroll
    for (int n = 4, m = 16; n >= 1; n >>= 1, m >>= 1)
#pragma unroll
      for (int i = 0; i < n; ++i) {
        const unsigned keep = lane & m ? a[i + n] : a[i], send = lane & m ? a[i] : a[i + n];
        a[i] = max(keep, __shfl_xor_sync(0xffffffffu, send, m));
      }
    atomicMax(sMax + 8 * (lane >> 3) + 2 * (lane & 3) + ((lane >> 2) & 1), a[0]);
  }
  // The same 32 columns to the shared-memory operand, normalised and scaled.  row_at: the lane's row of the 64-column chunk
  // (128-byte swizzle); c0: the first of the four 16-byte pieces.
  static __device__ __forceinline__ void emit_columns(const float* x, const float* on, const unsigned* sMax, uint32_t row_at, int c0,
                                                      int row, int lane) {
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const uint2 mx = *reinterpret_cast<const uint2*>(sMax + 8 * o + 2 * (lane & 3));
      const float2 g = make_float2(column_scale(mx.x), column_scale(mx.y));
      uint32_t u[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 v = fmul2(fmul2(frag_pair(x, o, i), make_float2(on[i], on[i])), g);
        u[i] = pack2<TA>(v.x, v.y);
      }
      stmatrix_x4(row_at + (((c0 + o) ^ (row & 7)) << 4), u[0], u[1], u[2], u[3]);
    }
  }

  static __device__ __forceinline__ void compute(const Params& P, uint8_t* smem, Shared* sh, uint32_t tmem, int warp_of_cta) {
    const int row = threadIdx.x & 127, warp = warp_of_cta & 3, w = warp_of_cta >> 2, lane = threadIdx.x & 31;
    const uint32_t d = tmem + 128 * w, t_row = d + ((uint32_t)(warp * 32) << 16);     // the group's columns, this warp's lanes
    const bool prep = prepares(P), last = P.last != 0;
    Slots<B> x(w);
    Group<Shared, Params> group(sh, P, w, warp, row);
    for (uint32_t q = 0;; ++q) {
      const uint32_t par = q & 1, par2 = (q >> 1) & 1;
      uint8_t *s0 = smem + x.x0 * kSlot, *s1 = smem + x.x1 * kSlot, *s2 = smem + x.x2 * kSlot;
      const int r_blk = row / B, r_pos = row % B;   // block of the tile, row in it
      auto score = [&]() {                     // first warp
        if (elect_one()) {
          scores(d, s0, s1);
          umma_commit(&sh->mma1[w]);
          if (R || last) umma_commit(&sh->empty[x.x0]);
          if (!R && last) umma_commit(&sh->empty[x.x1]);
        }
        __syncwarp();
        group.await(&sh->mma1[w], par, 31);
        if (prep && last) group.await(&sh->third[w][par], par2, 36);
      };
      bool more = true;
      if (warp == 0) {
        group.begin(q);
        group.await(&sh->full[w][par], par2, 30);
        more = group.ok && sh->tile[w][par].x >= 0;
        if (more && !prep) {
          score();
          more = group.ok;
        }
      }
      if (!group.release(more)) break;
      const int4 t = sh->tile[w][par];         // head, first block or position, keys that count
      const int h = t.x, idx0 = t.y;
      const int mv = FULL ? P.m : (t.z + P.b - 1) / P.b;                            // blocks that are present
      if (prep) {
        prepare(P, s0, !R || P.first, idx0, mv, row);      // Q, but not alpha_R
        prepare(P, s1, R, idx0, mv, row);                   // K, but not alpha_L
        group.collect();
        if (warp == 0) score();
        if (!group.release(group.ok)) break;
      }
      const float* sC = reinterpret_cast<const float*>(smem + kOffVec) + (2 * w + par) * 128;
      if (FULL && P.discard) {     // the state rows the score MMA consumed are read exactly once: drop them from L2
        if (!R) discard_line(P.aL + ((size_t)(h * P.b + idx0) * P.m + row) * 128);
        else if (!P.first) discard_line(P.aR + ((size_t)(h * P.m + idx0) * P.b + row) * 128);
      }
      float mul;                                 // of the accumulator rows in the epilogue
      if constexpr (R) {
        mul = r_softmax(P, h, idx0 + r_blk, t.z, t_row, r_blk, r_pos);
      } else {
        // ============================================================ L: softmax over the blocks
        const float f = P.scale * kLog2e;
        const uint32_t tS = t_row + B * r_blk;
        const float* cv = sC + B * r_blk;
        const int lim = FULL ? B : mv;
        float2 a2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        float mx;
        {
          // logits back over the scores, then weights (final: 16-bit, as the MMA's operand)
          float v[2][16];
          tmem_ld16(tS, v[0]);
#pragma unroll
          for (int cc = 0; cc < B / 16; ++cc) {
            float* cur = v[cc & 1];
            tmem_ld_wait();
            if (cc < B / 16 - 1) tmem_ld16(tS + 16 * (cc + 1), v[(cc + 1) & 1]);
            l_logits<16>(cur, cv + 16 * cc, f);
            mask<16>(cur, 16 * cc, lim);
            fold_max<16>(cur, m4);
            tmem_st16(tS + 16 * cc, cur);
          }
          mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
          tmem_st_wait();
          tmem_ld16(tS, v[0]);
#pragma unroll
          for (int cc = 0; cc < B / 16; ++cc) {
            float* cur = v[cc & 1];
            tmem_ld_wait();
            if (cc < B / 16 - 1) tmem_ld16(tS + 16 * (cc + 1), v[(cc + 1) & 1]);
            l_weights<16>(cur, mx, a2);
            if (last) {
              uint32_t u[8];
              pack_cols<16>(cur, u);
              st_cols<8>(t_row + (B / 2) * r_blk + 8 * cc, u);
            } else {
              tmem_st16(tS + 16 * cc, cur);
            }
          }
        }
        if (last) zeros_beside(t_row, r_blk);
        const float sum = (a2[0].x + a2[0].y) + (a2[1].x + a2[1].y);
        mul = 1.f / sum;
        tmem_st_wait();
        if (last) {
          // Row b l + j (l = r_pos, j = idx0 + r_blk) of the final L half-step: its log-sum-exp; summed
          // over the rows of a head it is the value of the objective (Eq. 6) at the returned matrix.
          if (P.lse != nullptr && r_pos < P.m && idx0 + r_blk < P.b)
            P.lse[(size_t)h * P.N + (size_t)r_pos * P.b + idx0 + r_blk] = (mx + fast_log2(sum)) * kLn2;
          if (!FULL && r_pos >= mv) mul = 0.f;        // rows of absent blocks
        } else {
          // (zeros beside the window keep blocks apart only if what they multiply is finite: a row of Q
          // that made its own weights NaN leaves the operand, its block has NaN from the weights)
          if (B < 128 && !(sum == sum)) zero_row(s0, row);
          // alpha_R(k,j) = sum_l L[l,k] Q(l,j) / c_R: the contraction runs over the rows of the weights,
          // so they are normalised before they are rounded, and go through shared memory (over
          // alpha_L, which the score MMA has read; at B = 128 with a slot of their own for one half).
          const float on = FULL || r_pos < mv ? mul : 0.f;     // rows past the last block: weight 0
          float onr[4];                          // of the lane's rows in fragments
#pragma unroll
          for (int i = 0; i < 4; ++i) onr[i] = __shfl_sync(0xffffffffu, on, 8 * i + (lane >> 2));
          // column k times 2^-(exponent of its largest weight)
          unsigned* sMax = reinterpret_cast<unsigned*>(smem + kOffCol) + 128 * (2 * w + par);
          float v[32];
#pragma unroll
          for (int cc = 0; cc < B / 32; ++cc) {
            ld_frag32(tS + 32 * cc, v);
            tmem_ld_wait();
            fold_columns(v, onr, sMax + B * r_blk + 32 * cc, lane);
          }
          ld_frag32(tS, v);
          // (128 columns: the slot of the second half is free; every warp looks for itself)
          if (B == 128) group.await(&sh->third[w][par], par2, 36);
          bar_sync(kRelease + w, 128);
          // (the set of the tile before: all warps are done with it, and none begins the next tile before all have come by)
          reinterpret_cast<unsigned*>(smem + kOffCol)[128 * (2 * w + (par ^ 1)) + row] = 0u;
          uint8_t* p_lo = smem + (B == 128 ? min(x.x1, x.x2) : x.x1) * kSlot + row * 128;
          uint8_t* p_hi = smem + (B == 128 ? max(x.x1, x.x2) : x.x1) * kSlot + row * 128;
          const int win = B == 32 ? 32 * (r_blk & 1) : 0;
#pragma unroll
          for (int cc = 0; cc < B / 32; ++cc) {
            if (cc > 0) ld_frag32(tS + 32 * cc, v);
            tmem_ld_wait();
            emit_columns(v, onr, sMax + B * r_blk + 32 * cc, smem_u32(cc < 2 ? p_lo : p_hi), (win >> 3) + (4 * cc & 7), row, lane);
          }
          if constexpr (B == 32) {               // zeros beside the window
            const int c0 = (32 - win) >> 3;
#pragma unroll
            for (int c = 0; c < 4; ++c) *reinterpret_cast<uint4*>(p_lo + (((c0 + c) ^ (row & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
          }
          fence_proxy_async();
        }
      }
      if (last && prep) prepare(P, s2, R, idx0, mv, row);   // V, but not y
      group.collect();
      if (warp == 0) {
        if (!R && last && !prep) group.await(&sh->third[w][par], par2, 36);
        if (group.ok && elect_one()) {
          if (R) {
            apply(d, s1);
            umma_commit(last ? &sh->first[w] : &sh->mma2[w]);
          } else if (last) {
            apply(d, s2);
            umma_commit(&sh->mma2[w]);
          } else {
            // (128 columns of weights: the first 64 in the lower of the two slots)
            const uint8_t* lower = B == 128 ? smem + min(x.x1, x.x2) * kSlot : s1;
            apply_transposed(d, lower, B == 128 ? (max(x.x1, x.x2) - min(x.x1, x.x2)) * kSlot : 16, s0, smem + kOffOnes);
            umma_commit(&sh->mma2[w]);
            umma_commit(&sh->empty[x.x1]);
            if (B == 128) umma_commit(&sh->empty[x.x2]);
          }
        }
        __syncwarp();
      }
      // ============================================================== epilogue
      float o[32];
      if (R && last) {                           // alpha_L, over K; then y, over V
        if (!group.await_rows(&sh->first[w], par, 32)) break;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          tmem_ld32(t_row + 64 + 32 * hf, o);
          tmem_ld_wait();
          if (hf == 1) {
            group.collect();
            if (warp == 0) {
              if (!prep) group.await(&sh->third[w][par], par2, 36);
              if (group.ok && elect_one()) {
                apply(d, s2);
                umma_commit(&sh->mma2[w]);
              }
              __syncwarp();
            }
          }
          store_row32<TA>(s1, row, 32 * hf, o, mul);
        }
        fence_proxy_async();
        group.hand_over(h, idx0, x.x1, 0);
      }
      if (!group.await_rows(&sh->mma2[w], par, 33)) break;
      int out_row = row;
      if (!R && !last) {
        if constexpr (!R && B < 128) out_row = ((lane >> 4) << 6) + 16 * warp + (lane & 15);
        const float cr = ld_col(t_row);
        tmem_ld_wait();
        mul = cr > 1e-30f ? 1.f / cr : 0.f;
      }
      if (FULL && P.discard && !R && last) discard_line(P.y + ((size_t)(h * P.b + idx0) * P.m + row) * 128);
      // rows go: alpha_L over K, y over V, alpha_R over Q, Y over y
      const int slot = last ? x.x2 : (R ? x.x1 : x.x0);
      uint8_t* dst = smem + slot * kSlot;
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        tmem_ld32(t_row + 64 + 32 * hf, o);
        tmem_ld_wait();
        if (hf == 1) group.leave();              // the next tile's scores may come
        if (R && last && !(mul == mul)) {      // NaN weights, and c_L is: the final L tiles hold several positions
          zero_row(dst, row);
        } else if (!R && last) {
          if (!FULL && mul == 0.f) {
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] = 0.f;
          }
          store_row32<TIn>(dst, out_row, 32 * hf, o, mul);
        } else {
          store_row32<TA>(dst, out_row, 32 * hf, o, mul);
        }
      }
      fence_proxy_async();
      group.hand_over(h, idx0, slot, R && last);
      x.next(R, last);
    }
    group.finish();
  }
};

template <typename TIn, int B, bool FULL, int MODE>
__global__ void __launch_bounds__(kThreads, kCtasPerSm) monarch_tiles(const __grid_constant__ Params P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align_smem<1024>(smem_raw);
  Shared* sh = reinterpret_cast<Shared*>(smem + kOffBar);
  const int tid = threadIdx.x, warp = warp_of_cta();
  const bool starts = MODE == 0 && P.first;      // the first launch of a call
  if (!starts) grid_launch_dependents();
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
      sh->through[w] = 0;
      mbar_init(&sh->out_free[w], 1);
    }
    sh->taken = 0;
    sh->abort_flag = 0;
    fence_barrier_init();
  }
  if (tid < 128) {
    const uint32_t one2 = pack2<__half>(1.f, 1.f);
    *reinterpret_cast<uint4*>(smem + kOffOnes + tid * 16) = make_uint4(one2, one2, one2, one2);
  }
  for (int i = tid; i < 4 * 128; i += kThreads) reinterpret_cast<float*>(smem + kOffVec)[i] = 0.f;
  for (int i = tid; i < 4 * 128; i += kThreads) reinterpret_cast<unsigned*>(smem + kOffCol)[i] = 0u;
  if (warp == 8) tmem_alloc(&sh->tmem, 256);
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, sh->tmem, 0);
  using K = Kernel<TIn, B, FULL, MODE>;
  // registers: 384 threads at the launch's 80; 128 x 64 + 256 x 88 make use of all of them
  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    if (warp < 10) {
      if (elect_one()) K::produce(P, smem, sh, warp - 8);
    } else {
      grid_wait();
      K::store(P, smem, sh, warp - 10);
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 88;");
    grid_wait();
    if (starts) {
      grid_launch_dependents();
      clear_status(P.clear);
    }
    K::compute(P, smem, sh, tmem, warp);
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (sh->abort_flag) {                 // what is in flight lands before the CTA leaves
    let_copies_land();
    __syncthreads();
  }
  if (warp == 8) tmem_dealloc(tmem, 256);
}

// ------------------------------------------------------------------------------------ host side
struct Args {
  const void *Q, *K, *V;
  void* Y;
  int BH, N, d, b, m, T, dtype, H, heads, n_valid;
  float scale;
  float* lse;
  const int* seq_len;
  Waits waits;
};
struct States {
  void *aL, *aR, *y;       // f16, BH * N rows of d
  float* cL;               // BH * b rows of pad4(m)
  int *status, *clear;
};
inline int pad4(int m) { return (m + 3) & ~3; }
inline bool supported(int N, int d, int b, int m, int dtype, int BH) {
  return (dtype == 1 || dtype == 2) && d % 8 == 0 && d <= 64 && b <= 128 && m <= 128 && (long long)BH * N < (1LL << 31);
}
// 2T launches, one per half-step.
int launch(const Args& a, const States& s, cudaStream_t st);

#ifdef MA_TU_TILE_TC
inline int pad_block(int x) { return x <= 32 ? 32 : (x <= 64 ? 64 : 128); }

// View (d, i, k, h0, h1) with byte strides s1 .. s4; box of 128 rows: B of the second dimension,
// 128 / B of the third.
inline bool make_map5(CUtensorMap* tm, int dtype, const void* base, const uint64_t (&n)[5], const uint64_t (&s)[4], int B,
                      int rows = 0) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[5], strides[4];
  for (int i = 0; i < 5; ++i) dims[i] = n[i];
  for (int i = 0; i < 4; ++i) strides[i] = s[i];
  cuuint32_t box[5] = {kD, (cuuint32_t)(rows ? rows : B), (cuuint32_t)(128 / B), 1, 1}, es[5] = {1, 1, 1, 1, 1};
  return fn(tm, dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base),
            dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
inline bool make_maps(Params* P, const Args& a, const States& s) {
  const uint64_t d2 = (uint64_t)a.d * 2, b = a.b, m = a.m, N = a.N, BH = a.BH, H = a.H ? a.H : 1;
  const int BR = pad_block(a.b), BL = pad_block(a.m), BK = a.waits.starve ? 1 : BR;
  // inputs and output: rows d2 (or heads * d2) apart
  const uint64_t row = d2 * H, h0 = a.H ? a.H : BH, h1 = a.H ? BH / a.H : 1;
  const uint64_t s0 = a.H ? d2 : N * d2, s1 = N * d2 * (a.H ? H : BH);
  const uint64_t rn[5] = {(uint64_t)a.d, b, m, h0, h1}, rs[4] = {row, b * row, s0, s1};
  const uint64_t ln[5] = {(uint64_t)a.d, m, b, h0, h1}, ls[4] = {b * row, row, s0, s1};
  // states: alpha_L, y [BH][b][m][d]; alpha_R [BH][m][b][d] -- every load reads contiguous rows, the
  // permutation between the half-steps is in the strides of the stores
  const uint64_t srn[5] = {(uint64_t)a.d, b, m, BH, 1}, sln[5] = {(uint64_t)a.d, m, b, BH, 1};
  const uint64_t l_st[4] = {m * d2, d2, N * d2, N * d2 * BH}, l_ld[4] = {d2, m * d2, N * d2, N * d2 * BH};
  const uint64_t r_ld[4] = {d2, b * d2, N * d2, N * d2 * BH}, r_st[4] = {b * d2, d2, N * d2, N * d2 * BH};
  return make_map5(&P->rQ, a.dtype, a.Q, rn, rs, BR) && make_map5(&P->rK, a.dtype, a.K, rn, rs, BR, BK) &&
         make_map5(&P->rV, a.dtype, a.V, rn, rs, BR) && make_map5(&P->rAR, 1, s.aR, srn, r_ld, BR) &&
         make_map5(&P->rAL, 1, s.aL, srn, l_st, BR) && make_map5(&P->rY, 1, s.y, srn, l_st, BR) &&
         make_map5(&P->lQ, a.dtype, a.Q, ln, ls, BL) && make_map5(&P->lAL, 1, s.aL, sln, l_ld, BL) &&
         make_map5(&P->lY, 1, s.y, sln, l_ld, BL) && make_map5(&P->lAR, 1, s.aR, sln, r_st, BL) &&
         make_map5(&P->lOut, a.dtype, a.Y, ln, ls, BL);
}
// Tensor maps depend only on the addresses and the shape; encoding eleven of them costs several
// times the launch, so the maps of the last few problems are kept.
struct MapKey {
  const void *Q, *K, *V, *Y, *aL, *aR;
  int BH, N, d, b, dtype, H, dev;
  bool starve;
  bool operator==(const MapKey& o) const {
    return starve == o.starve && Q == o.Q && K == o.K && V == o.V && Y == o.Y && aL == o.aL && aR == o.aR && BH == o.BH && N == o.N && d == o.d &&
           b == o.b && dtype == o.dtype && H == o.H && dev == o.dev;
  }
};
struct MapCache {
  static constexpr int kEntries = 16;
  MapKey key[kEntries];
  Params maps[kEntries];
  bool used[kEntries] = {};
  int next = 0, last = 0;
};
inline bool cached_maps(Params* P, const Args& a, const States& s, int dev) {
  static thread_local MapCache c;
  const MapKey key{a.Q, a.K, a.V, a.Y, s.aL, s.aR, a.BH, a.N, a.d, a.b, a.dtype, a.H, dev, a.waits.starve};
  for (int i = 0; i < MapCache::kEntries; ++i) {
    const int e = (c.last + i) % MapCache::kEntries;
    if (c.used[e] && c.key[e] == key) {
      c.last = e;
      *P = c.maps[e];
      return true;
    }
  }
  if (!make_maps(P, a, s)) return false;
  const int e = c.next;
  c.next = (c.next + 1) % MapCache::kEntries;
  c.key[e] = key;
  c.maps[e] = *P;
  c.used[e] = true;
  c.last = e;
  return true;
}
struct Device {
  int dev = -1, sms = 0;
};
inline bool current_device(Device* d) {
  static int sms[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  if (sms[dev] == 0 && cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return false;
  d->dev = dev;
  d->sms = sms[dev];
  return d->sms > 0;
}
template <typename TIn, int B, bool FULL, int MODE>
inline int launch_kernel(const Params& P, const Device& dev, cudaStream_t st) {
  auto kern = monarch_tiles<TIn, B, FULL, MODE>;
  static bool prepared[64] = {};
  if (!prepared[dev.dev]) {
    if (cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem) != cudaSuccess) return 7;
    prepared[dev.dev] = true;
  }
  // (the next half-step's CTAs take SM slots, set up and ask for inputs as this one's drain; they wait for its end before they touch what it
  // writes, and the call's first launch lets the next ones start only once it has waited for whatever wrote the inputs)
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(P.tiles < kCtasPerSm * dev.sms ? P.tiles : kCtasPerSm * dev.sms);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, P) == cudaSuccess ? 0 : 7;
}
template <typename TIn, int MODE>
inline int launch_half(Params& P, const Device& dev, cudaStream_t st, bool masked) {
  const int x = MODE == 0 ? P.b : P.m, n = MODE == 0 ? P.m : P.b, B = pad_block(x);      // n blocks of x rows
  P.per_head = (n + 128 / B - 1) / (128 / B);
  P.tiles = P.BH * P.per_head;
  const bool full = !masked && x == B && n % (128 / B) == 0;
#define MA_H(B) (full ? launch_kernel<TIn, B, true, MODE>(P, dev, st) : launch_kernel<TIn, B, false, MODE>(P, dev, st))
  return B == 32 ? MA_H(32) : (B == 64 ? MA_H(64) : MA_H(128));
#undef MA_H
}
template <typename TIn>
inline int launch_t(const Args& a, const States& s, cudaStream_t st) {
  Device dev;
  Params P;
  if (!current_device(&dev) || !cached_maps(&P, a, s, dev.dev)) return 7;
  P.cL = s.cL;
  P.aL = (uint8_t*)s.aL; P.aR = (uint8_t*)s.aR; P.y = (uint8_t*)s.y;
  P.lse = a.lse; P.seq_len = a.seq_len; P.report = s.status; P.clear = s.clear;
  P.N = a.N; P.b = a.b; P.m = a.m; P.mp = pad4(a.m); P.BH = a.BH; P.H = a.H; P.heads = a.heads; P.n_valid = a.n_valid;
  P.discard = a.d == 64;       // (a row is then a line)
  P.wait_cycles = a.waits.cycles;
  P.scale = a.scale;
  for (int t = 0; t < a.T; ++t) {
    P.first = t == 0;
    P.last = t == a.T - 1;
    const int rc = launch_half<TIn, 0>(P, dev, st, a.n_valid < a.N || a.seq_len != nullptr);
    if (rc != 0) return rc;
    const int rl = launch_half<TIn, 1>(P, dev, st, a.seq_len != nullptr);
    if (rl != 0) return rl;
  }
  return 0;
}
int launch(const Args& a, const States& s, cudaStream_t st) {
  return a.dtype == 1 ? launch_t<__half>(a, s, st) : launch_t<__nv_bfloat16>(a, s, st);
}
#endif  // MA_TU_TILE_TC

}  // namespace ttc
}  // namespace ma
