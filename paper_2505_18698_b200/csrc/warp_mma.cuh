// Warp-level MMA helpers shared by the fused per-head kernel and the warp-MMA tile kernels:
// mma.sync m16n8k16 wrappers for f16 / bf16, matrix loads and transposes, quad and column
// reductions over the accumulator layout, and the bf16 <-> f16 conversions of 16-byte chunks.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "f32x2.cuh"

namespace ma {
namespace warpmma {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

template <typename T> struct Mma;
template <> struct Mma<__half> {
  static __device__ __forceinline__ void run(float* c, const uint32_t* a, const uint32_t* b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
  }
  // The first product of a sum: c = a b (nothing to clear beforehand).
  static __device__ __forceinline__ void first(float* c, const uint32_t* a, const uint32_t* b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(0.f));
  }
  static constexpr bool is_f16 = true;
  static __device__ __forceinline__ uint32_t pack(float x, float y) {
    __half2 h = __floats2half2_rn(x, y);
    return *reinterpret_cast<uint32_t*>(&h);
  }
  static __device__ __forceinline__ uint32_t pack(float2 v) { return pack(v.x, v.y); }
  static __device__ __forceinline__ float2 unpack(uint32_t u) {
    return __half22float2(*reinterpret_cast<__half2*>(&u));
  }
};
template <> struct Mma<__nv_bfloat16> {
  static __device__ __forceinline__ void run(float* c, const uint32_t* a, const uint32_t* b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
  }
  static constexpr bool is_f16 = false;
  static __device__ __forceinline__ uint32_t pack(float x, float y) {
    __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    return *reinterpret_cast<uint32_t*>(&h);
  }
  static __device__ __forceinline__ float2 unpack(uint32_t u) {
    return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
  }
};

// c = a b where `fresh`, else c += a b.
template <typename T>
__device__ __forceinline__ void mma(bool fresh, float* c, const uint32_t* a, const uint32_t* b) {
  if (fresh) Mma<T>::first(c, a, b);
  else Mma<T>::run(c, a, b);
}
// The two rows of an accumulator tile, as pairs.
__device__ __forceinline__ float2 row_pair(const float* c, int hh) { return make_float2(c[2 * hh], c[2 * hh + 1]); }
__device__ __forceinline__ void put_pair(float* c, int hh, float2 v) {
  c[2 * hh] = v.x;
  c[2 * hh + 1] = v.y;
}

// Lets a kernel use up to `bytes` of dynamic shared memory: once per kernel and device (the call
// costs most of a microsecond of host time).
struct SmemOptIn {
  bool prepared[64] = {};
  bool done(const void* kernel, int bytes) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    if (!prepared[dev])
      prepared[dev] = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
    return prepared[dev];
  }
};

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void ldsm_x4(uint32_t* r, uint32_t saddr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(saddr));
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t* r, uint32_t saddr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(saddr));
}
__device__ __forceinline__ uint32_t movm_trans(uint32_t a) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}
__device__ __forceinline__ float quad_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}
__device__ __forceinline__ float col_sum(float v) {   // over the 8 row groups (lanes with equal t)
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 8);
  return v + __shfl_xor_sync(0xffffffffu, v, 16);
}

// Reduction of NV values (a power of two) over the lanes that differ in bits HI .. LO of `lane`.  Each step
// halves the values a lane carries as long as there is more than one: lane bits HI, HI / 2, .. are the
// leading bits of the index of the values it ends up with, NV / (lanes) of them, or one, in v[0], ..
template <int NV, int HI, int LO, typename Op>
__device__ __forceinline__ float scatter_reduce(float* v, int lane, Op op) {
  int n = NV / 2;
#pragma unroll
  for (int m = HI; m >= LO; m >>= 1, n >>= 1) {
    if (n >= 1) {
#pragma unroll
      for (int i = 0; i < NV / 2; ++i)
        if (i < n) {
          const float keep = lane & m ? v[i + n] : v[i], send = lane & m ? v[i] : v[i + n];
          v[i] = op(keep, __shfl_xor_sync(0xffffffffu, send, m));
        }
    } else {
      v[0] = op(v[0], __shfl_xor_sync(0xffffffffu, v[0], m));
    }
  }
  return v[0];
}
struct Add { __device__ __forceinline__ float operator()(float a, float b) const { return a + b; } };
struct Max { __device__ __forceinline__ float operator()(float a, float b) const { return fmaxf(a, b); } };

__device__ __forceinline__ uint4 to_f16x8(uint4 v, const __half*) { return v; }
__device__ __forceinline__ uint4 to_f16x8(uint4 v, const __nv_bfloat16*) {
  uint32_t* w = reinterpret_cast<uint32_t*>(&v);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    // a bf16 is the upper half of an fp32; the conversion saturates at +-65504
    asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;"
        : "=r"(w[i])
        : "f"(__uint_as_float(w[i] & 0xffff0000u)), "f"(__uint_as_float(w[i] << 16)));
  }
  return v;
}
__device__ __forceinline__ uint4 from_f16x8(uint4 v, __half*) { return v; }
__device__ __forceinline__ uint4 from_f16x8(uint4 v, __nv_bfloat16*) {
  uint32_t* w = reinterpret_cast<uint32_t*>(&v);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = Mma<__half>::unpack(w[i]);
    w[i] = Mma<__nv_bfloat16>::pack(f.x, f.y);
  }
  return v;
}
}  // namespace warpmma
}  // namespace ma
