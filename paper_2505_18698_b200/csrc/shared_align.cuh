// Alignment of dynamic shared memory.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ma {

// First multiple of A at or after `p`, as an offset from it: a pointer that went through an integer is a generic one to the compiler,
// and every access through it pays for a 64-bit address and the generic load/store path (B200, us per call, integer / offset: 8
// heads of 7600 40.9 / 39.5, 64 heads of 4096 81.8 / 79.3, 16 of 16384 104.3 / 102.0, 192 of 1024 56.3 / 54.5).  The per-head kernels
// address shared memory by 32-bit addresses throughout and lost 1 % to it where heads are few.
template <uint32_t A>
__device__ __forceinline__ uint8_t* align_smem(uint8_t* p) {
  return p + ((A - ((uint32_t)__cvta_generic_to_shared(p) & (A - 1))) & (A - 1));
}

}  // namespace ma
