// What the compute groups of tensor_chain.cuh and tile_tc.cuh share: three slots of shared memory that a group's tiles take in turn, waits that
// run out, and the hand-overs in a group of four compute warps, a producer thread and a store warp.
//
// The first warp of a group alone looks at mbarriers, which means trying again and again, and lets the others go on once it has seen one: four
// warps that try take issue slots from those at work (64 heads of 4096, T = 2 77.8 us with all of them, 76.7 with one).  All other hand-overs
// in the group are barriers in hardware.
#pragma once
#include "status_word.cuh"
#include "tensor_path.cuh"

namespace ma {
namespace group {

using namespace ma::tensor;

// A group's slots as the operands of its current tile; next(): in the order in which the tile gives them up.  B: columns of a block.
//   R:            first  alpha_R (Q), free after the score MMA; second K, alpha_L staged over it; third, last round, V and y over it
//   L, not last:  first  Q(.,j), alpha_R staged over it; second alpha_L, then weights, free after the apply MMA (128 columns: and third)
//   L, last:      first  Q(.,j), second alpha_L, both free after the score MMA; third y, Y staged over it
template <int B>
struct Slots {
  int x0, x1, x2;
  __device__ __forceinline__ explicit Slots(int w) : x0(3 * w), x1(3 * w + 1), x2(3 * w + 2) {}
  __device__ __forceinline__ void next(bool is_r, bool last_round) {      // (half-steps of the last round keep their order)
    const int a = x0, b = x1, c = x2;
    if (last_round) return;
    if (B == 128 && !is_r) {
      x0 = b;
      x1 = c;
      x2 = a;
      return;
    }
    x0 = c;
    x1 = is_r ? a : b;
    x2 = is_r ? b : a;
  }
};

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }
// The same with a vote: whether it is true for all of them.
__device__ __forceinline__ bool bar_all(int id, int n, bool on) {
  uint32_t all;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %3, 0;\n\tbarrier.cta.red.and.pred q, %1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(all)
      : "r"(id), "r"(n), "r"((uint32_t)on)
      : "memory");
  return all != 0;
}
// By group: the first warp lets the others go on, it waits for them, the store warp waits for staged rows.
enum BarId { kRelease = 1, kCollect = 3, kStaged = 5 };

// Bounded wait: after a timeout (status word and abort flag set) every wait of the CTA returns at once (HEED: but for those that come to an end
// by themselves), and its groups stop.
template <bool HEED = true, typename Shared, typename Params>
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, Shared* sh, const Params& P, int where) {
  const uint32_t addr = smem_u32(bar);
  uint32_t done = 0;
  long long t0 = 0;
  for (int n = 0;; ++n) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
    if (HEED && sh->abort_flag) return false;
    if (n == 0) {
      t0 = clock64();
    } else if (clock64() - t0 > P.wait_cycles) {
      report_timeout(P.report, where);
      sh->abort_flag = 1;
      return false;
    }
  }
}
// Tiles that a group is through with: its first warp says so once all warps have come by (`Group::begin`), the producer waits for it at the end of its
// list, where the word of a tile and its barrier have to be free.  A count: by the parity of a barrier a producer that comes late cannot tell the last tile
// from the one before the last but one.
template <typename Shared, typename Params>
__device__ __forceinline__ bool wait_through(Shared* sh, int w, uint32_t tiles, const Params& P) {
  const long long t0 = clock64();
  while (*(volatile int*)&sh->through[w] < (int)tiles) {
    if (sh->abort_flag) return false;
    if (clock64() - t0 > P.wait_cycles) {
      report_timeout(P.report, 12);
      sh->abort_flag = 1;
      return false;
    }
    __nanosleep(100);
  }
  __threadfence_block();
  return true;
}

// The hand-overs of compute group w, as one of its warps takes part in them.  Shared has through[2], out[2], out_free[2] and abort_flag, Params
// report and wait_cycles.
template <typename Shared, typename Params>
struct Group {
  Shared* sh;
  const Params& P;
  int w, warp, row;                          // the thread's row of the tile
  uint32_t par_o = 1;
  bool ok = true;                            // (the first warp's decides) no wait has run out
  __device__ __forceinline__ Group(Shared* s, const Params& p, int group, int warp_of_group, int row_of_group)
      : sh(s), P(p), w(group), warp(warp_of_group), row(row_of_group) {}

  __device__ __forceinline__ void await(uint64_t* bar, uint32_t parity, int where) {
    ok = __all_sync(0xffffffffu, wait_bar(bar, parity, sh, P, where)) && ok;
  }
  // First warp, before tile q: every row of the tile before has left tensor memory.
  __device__ __forceinline__ void begin(uint32_t q) {
    if (q > 0) {
      bar_sync(kCollect + w, 128);
      tc_fence_after();
      if (row == 0) {
        __threadfence_block();
        *(volatile int*)&sh->through[w] = (int)q;
      }
    }
  }
  // Of the group, by its first warp; false: no more tiles.  A wait that ran out reaches the other warps here.
  __device__ __forceinline__ bool release(bool on) {
    tc_fence_before();
    const bool go = bar_all(kRelease + w, 128, on);
    tc_fence_after();
    return go;
  }
  // All warps have come by: the first one waits.
  __device__ __forceinline__ void collect() {
    tc_fence_before();
    if (warp == 0) {
      bar_sync(kCollect + w, 128);
      tc_fence_after();
    } else {
      bar_arrive(kCollect + w, 128);
    }
  }
  // The tile's accumulator has been read: the first warp waits for that in `begin`.
  __device__ __forceinline__ void leave() {
    tc_fence_before();
    if (warp != 0) bar_arrive(kCollect + w, 128);
  }
  // An accumulator is done, and the store warp has taken the word of the rows before: nobody comes by at kStaged a second time
  // before the store warp has.
  __device__ __forceinline__ bool await_rows(uint64_t* bar, uint32_t parity, int where) {
    if (warp == 0) {
      await(bar, parity, where);
      if (ok) await(&sh->out_free[w], par_o, 38);
      if (ok) par_o ^= 1;
    }
    return release(ok);
  }
  // Staged rows, for the store warp.
  __device__ __forceinline__ void hand_over(int h, int idx0, int z, int v) {
    if (row == 0) sh->out[w] = make_int4(h, idx0, z, v);
    __syncwarp();
    bar_arrive(kStaged + w, 160);
  }
  // No more tiles.  (Aborted or not: rows handed over before are on their way, and the store warp comes back for this word.)
  __device__ __forceinline__ void finish() {
    if (warp == 0) __all_sync(0xffffffffu, wait_bar<false>(&sh->out_free[w], par_o, sh, P, 38));
    release(false);
    hand_over(-1, 0, 0, 0);
  }
};

}  // namespace group
}  // namespace ma
