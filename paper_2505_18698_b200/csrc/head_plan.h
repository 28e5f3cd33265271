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
// Warps an SM has room for.  Two 8-column tiles either way fit 64 registers (nothing is spilled), 24 warps' 80 the other one-round
// kernels and 24 x 16 (at most 16 bytes), the rest take 128.
constexpr int max_warps(int nb, int nm, int rounds) { return nb == 2 && nm == 2 ? 32 : (rounds == kOne || (nb == 3 && nm == 2) ? 24 : 16); }

// Shared memory of a CTA: `bufs` x (Q, K, V), the state tile (more than one round), a dump for matrix-store rows past a
// block (a line of its own: addresses step through a row by an exclusive or of bits 5 and 6), c_L ([position]
// [nm * 8 blocks]), barriers.
inline size_t smem_bytes(int tile, int bufs, int rounds, int b, int nm) {
  return (size_t)tile * (rounds == kMoreVLast ? 3 : 3 * bufs + (rounds == kMore ? 1 : 0)) + 128 + (size_t)b * nm * 8 * 4 + sizeof(Bars) + 1024;
}

struct Plan {
  int bp, tile, bufs, warps, ctas, rounds;      // ctas: per SM
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
    // as many CTAs as fit, up to three, each with a head of its own (768 heads of 130 = 13 x 10, two rounds: 34.6 us with
    // three, 39.8 with two).  Where no third fits and there are heads left for a second turn, one CTA of all warps
    // with the next head's loads under way is faster with 16 warps an SM (it has the same work in flight), with 32 two
    // CTAs are, and V goes over the states where that makes room for the second.
    p->ctas = BH <= num_sms ? 1 : std::min(fit(p->smem), 3);
    const int most = max_warps(nb, nm, rounds);
    if (p->ctas <= 2 && BH > p->ctas * num_sms) {
      const size_t v_last = smem_bytes(p->tile, 1, kMoreVLast, b, nm);
      if (most == 32 && p->ctas == 2) {
      } else if (most == 32 && rounds == kMore && fit(v_last) >= 2) {
        p->ctas = 2;
        p->rounds = kMoreVLast;
        p->smem = v_last;
      } else if (two <= kMaxSmem) {
        p->ctas = 1;
        p->bufs = 2;
        p->smem = two;
      }
    }
    // the fewest warps that take the fewest rounds of tiles over both half-steps
    int best = 1 << 30;
    for (int w = 1; w <= most / p->ctas; ++w) {
      const int turns = (m + w - 1) / w + (b + w - 1) / w;
      if (turns < best) {
        best = turns;
        p->warps = w;
      }
    }
    return true;
  }
  return false;
}

}  // namespace fhead
}  // namespace ma
