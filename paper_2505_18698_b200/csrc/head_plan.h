// How the per-head kernel (fused_head.cuh) lays out a head and shares an SM between heads: plain C++, so that the
// choices can be checked without a GPU.
#pragma once
#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace ma {
namespace fhead {

// Shared memory: what a CTA may ask for, what an SM has, and what the system takes of that for each CTA.
constexpr size_t kMaxSmem = 227 * 1024, kSmSmem = 228 * 1024, kCtaReserve = 1024;
constexpr int kMaxBlocks = 32;

struct alignas(16) Bars {
  uint64_t full[2][kMaxBlocks];      // by buffer (V over the states: the second set is V's) and block
};

// What a kernel is for: one round; more, with a state tile beside Q, K and V; more, with V over the states once the last round
// has read them (three tiles a head).
enum Rounds { kOne = 0, kMore = 1, kMoreVLast = 2 };
// Warps an SM has room for, that is, the registers that a kernel is compiled for (65536 / 32 / warps).  More warps pay where a half-step then
// takes fewer turns or a second head is at work, and cost where they make the compiler spill.  Two 8-column tiles either way fit 64
// registers (nothing is spilled): 32 warps.  Up to three either way fit 80 in the one-round kernels (up to 12 bytes spilled): 24 warps take 17 to
// 24 rows or blocks in one turn instead of two (us with 24 / with 16: 768 heads of 20 x 20 59.1 / 62.4 in f16, 66.9 / 74.3 in bf16, 12 heads
// 9.0 / 10.3; 24 x 16 48.0 / 47.9, 56.3 / 56.3, 12 heads 6.9 / 7.1; 10 x 18 29.9 / 30.1, 35.4 / 36.2; 14 x 22 41.9 / 40.8, 50.0 / 50.0).
// 25 to 32 take two turns either way and 80 registers spill 20 to 52 bytes (12 x 32 47.5 / 46.0, 32 x 11 48.1 / 45.9, 32 x 17 79.6 / 71.6, bf16 92.5 / 89.2,
// 26 x 22 bf16 100.3 / 98.1, though 28 x 20 bf16 88.5 / 90.5); so do more rounds (24 x 16 81.5 / 77.6, bf16 88.5 / 85.4, 20 x 12 61.0 / 58.9), a head an SM: 16.
constexpr int max_warps(int nb, int nm, int rounds) { return nb == 2 && nm == 2 ? 32 : (rounds == kOne && nb <= 3 && nm <= 3 ? 24 : 16); }

// Shared memory of a CTA: `bufs` x (Q, K, V), the state tile (more than one round), a dump for matrix-store rows past a
// block (a line of its own: addresses step through a row by an exclusive or of bits 5 and 6), c_L ([position]
// [nm * 8 blocks]), barriers.
inline size_t smem_bytes(int tile, int bufs, int rounds, int b, int nm) {
  return (size_t)tile * (rounds == kMoreVLast ? 3 : 3 * bufs + (rounds == kMore ? 1 : 0)) + 128 + (size_t)b * nm * 8 * 4 + sizeof(Bars) + 1024;
}

// Whether any head of nb and nm 8-column tiles has a plan: Q, K and V of the smallest, 8 nb - 7 rows and 8 nm - 7 blocks, fit a CTA.  (25 x 25 does not.)
constexpr bool any_fits(int nb, int nm) { return (size_t)3 * (8 * nb - 7) * (8 * nm - 7) * 128 <= kMaxSmem; }

struct Plan {
  int bp, tile, bufs, warps, ctas, rounds, bound;      // ctas: per SM; bound: warps an SM that the kernel is compiled for
  int parts;      // CTAs a head goes to
  size_t smem;
};
inline bool plan(int b, int m, int T, int BH, int num_sms, Plan* p) {
  const int nb = (b + 7) / 8, nm = (m + 7) / 8, rounds = T > 1 ? kMore : kOne;
  // The odd pitch where it fits; without it the L half-step's rows conflict (8-way for b = 16, 24, 32,
  // which the general kernel then serves faster: N = 576 as 24 x 24, 768 heads, 120 against 125 us).
  for (int odd = 1; odd >= (b % 8 != 0 ? 0 : 1); --odd) {
    p->bp = odd ? (b | 1) : b;
    p->tile = (m * p->bp * 128 + 1023) / 1024 * 1024;
    p->rounds = rounds;
    p->bufs = 1;
    const size_t two = smem_bytes(p->tile, 2, rounds, b, nm);
    p->smem = smem_bytes(p->tile, 1, rounds, b, nm);
    if (p->smem > kMaxSmem) continue;
    auto fit = [](size_t bytes) { return (int)(kSmSmem / (bytes + kCtaReserve)); };      // CTAs per SM by shared memory
    // At most one head per SM: one CTA with as many warps as a half-step has tiles.  More: the warps an SM holds go to
    // as many CTAs as fit, up to three and up to the heads an SM gets, each with a head of its own (768 heads of 130 = 13 x 10, two rounds:
    // 34.6 us with three, 39.8 with two; 216 of 187 = 11 x 17, one round 8.9 with two, 12.0 with three, 280 of 17 x 9 8.6 / 12.1).  Where no third fits
    // and there are heads left for a second turn, one CTA of all warps with the next head's loads under way is faster with 16 warps an
    // SM (it has the same work in flight), with 32 two CTAs are, and V goes over the states where that makes room for the second.
    p->ctas = std::min({fit(p->smem), 3, (BH + num_sms - 1) / num_sms});
    int most = max_warps(nb, nm, rounds);
    if (p->ctas <= 2 && BH > p->ctas * num_sms) {
      const size_t v_last = smem_bytes(p->tile, 1, kMoreVLast, b, nm);
      // But a turn of two heads an SM takes 1.6 to 1.7 times a turn of one, also where it is less than full, because which SMs the last
      // heads meet is chance (up to half a head an SM it takes 1.1).  So one CTA where that makes fewer of it (us, one CTA / two): 16 x 16, one round
      // 360 heads 14.0 / 13.2, 380 14.1 / 15.2, 440 14.4 / 16.1, 460 17.3 / 16.1, 740 21.9 / 22.7, 768 24.8 / 22.7, 1000 29.0 / 29.1; 14 x 15, two
      // rounds 380 21.4 / 21.9, 440 21.5 / 24.6, 592 27.9 / 25.2, 740 34.0 / 35.9, 768 39.5 / 35.8.
      const bool ahead = two <= kMaxSmem;
      const int left = BH % (2 * num_sms), one_each = 10 * ((BH + num_sms - 1) / num_sms);
      const int two_each = 17 * (BH / (2 * num_sms)) + (left == 0 ? 0 : (2 * left <= num_sms ? 11 : 17));
      const bool pairs = most == 32 && (!ahead || two_each < one_each);
      if (pairs && p->ctas == 2) {
      } else if (pairs && rounds == kMore && fit(v_last) >= 2) {
        p->ctas = 2;
        p->rounds = kMoreVLast;
        p->smem = v_last;
      } else if (ahead) {
        p->ctas = 1;
        p->bufs = 2;
        p->smem = two;
      }
    }
    // (24 x 16 and the like, more rounds: 24 warps where they are two heads: 216 heads of 20 x 10 16.0 us, with 16 17.4)
    if (nb == 3 && nm == 2 && rounds == kMore && p->ctas == 2) most = 24;
    // More than 16 positions and SMs enough for two CTAs a head: half of the positions each, so that a block is one 16-row tile instead of two
    // and a position has a warp to itself (us, one CTA / two: 12 heads of 16 x 24, one round 6.9 / 4.8, two 11.7 / 7.6, 36 of 19 x 22 9.0 / 6.3, 48 of 12 x 20, two
    // rounds 10.0 / 6.8, 72 of 23 x 17 9.6 / 7.3, 24 of 14 x 30 7.6 / 5.1).  It takes more of the GPU in all: two such calls at once on two streams gain up to about a quarter
    // of the SMs each and lose above (us for both: 12 heads of 16 x 24 6.9 / 4.8, 36 7.1 / 5.2, 60 of 10 x 18, two rounds 10.1 / 10.0, 72 of 16 x 24 7.8 / 9.6, of 20 x 20 10.0 / 12.5).
    p->parts = nb > 2 && 2 * BH <= num_sms ? 2 : 1;
    if (p->parts == 2) most = 16;
    // A CTA an SM: so much shared memory (no two of half an SM's fit) that the next call's CTAs do not come to an SM at work (us in loops, without / with:
    // 144 heads of 11 x 12 6.8 / 5.0, of 10 x 10 6.0 / 4.7, 108 of 10 x 10, two rounds 8.1 / 6.5, 72 of 10 x 17 5.6 / 4.6).  That keeps calls on other streams off as well:
    // two at once (us for both) 72 heads of 10 x 10 4.8 / 3.6, but 108 4.8 / 5.2, 144 4.9 / 6.6, two rounds 7.7 / 10.8, 144 of 12 x 11 5.4 / 6.9.  Calls one after another
    // are the rule.  Letting the next call's CTAs come once the call before is gone (griddepcontrol.launch_dependents after the wait) instead leaves room for
    // other streams (144 heads 5.0, two rounds 7.8), but loops of short calls lose 15 to 25 % (132 heads of 12 x 11 4.3 / 5.4, 144 of 10 x 10 in bf16 4.8 / 6.0).
    if (p->parts * BH <= num_sms) p->smem = std::max(p->smem, (size_t)114 * 1024);
    // the fewest warps that take the fewest rounds of tiles over both half-steps
    int best = 1 << 30;
    for (int w = 1; w <= most / p->ctas; ++w) {
      const int turns = (m + w - 1) / w + ((b + p->parts - 1) / p->parts + w - 1) / w;
      if (turns < best) {
        best = turns;
        p->warps = w;
      }
    }
    // Where an SM does not get more than 16 warps (a head an SM or fewer), 64 registers only make the chain longer (us with up to 128 / with
    // 64): two rounds, 12 heads of 12 x 15 6.7 / 7.6, 48 6.7 / 8.7, 148 of 16 x 16 7.6 / 8.3; one round, 48 of 16 x 16 4.6 / 5.3, 100 of 12 x 16 in bf16 5.2 / 7.8.
    p->bound = most == 32 && p->ctas * p->warps <= 16 ? 16 : most;
    return true;
  }
  return false;
}

}  // namespace fhead
}  // namespace ma
