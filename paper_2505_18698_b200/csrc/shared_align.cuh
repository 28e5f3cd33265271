// Two things that the compiler cannot see by itself: where dynamic shared memory starts, and that a warp has one number.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ma {

// First multiple of A at or after `p`, as an offset from it: a pointer that went through an integer is a generic one to the compiler,
// and every access through it pays for a 64-bit address and the generic load/store path (B200, us per call, integer / offset: 8
// heads of 7600 40.9 / 39.5, 64 heads of 4096 81.8 / 79.3, 16 of 16384 104.3 / 102.0, 192 of 1024 56.3 / 54.5, 768 of 197, T = 2 35.3 / 34.4).
template <uint32_t A>
__device__ __forceinline__ uint8_t* align_smem(uint8_t* p) {
  return p + ((A - ((uint32_t)__cvta_generic_to_shared(p) & (A - 1))) & (A - 1));
}

// A thread's warp of the CTA, by a shuffle, so that the compiler knows it to be the same for all 32 lanes: what is computed from it (barriers,
// descriptors, tile indexes, loop bounds) then stays in uniform registers and instructions.  us per call, threadIdx.x >> 5 / this: 768 heads of
// 256 22.6 / 22.3, of 20 x 20 59.0 / 57.2, 192 of 210, T = 3 30.8 / 30.2, 16 of 4096 on monarch_decoupled 38.5 / 37.2; what it gives where single
// threads issue MMAs stands in tensor_chain.cuh.  The position-split kernel (fused_jsplit.cuh) lost 5 % to it and does without.
__device__ __forceinline__ int warp_of_cta() { return __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0); }

}  // namespace ma
