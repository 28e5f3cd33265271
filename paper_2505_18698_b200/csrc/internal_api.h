// Entry of the library that its Python extension uses: one description of a call for every device
// entry point of monarch_attn.h, plus an allocator the library asks for the scratch the path it
// picks needs (so that the caller neither resolves the path itself nor allocates for the largest).
// Not part of the C ABI in include/.
#pragma once
#include <stddef.h>

namespace ma {

enum class Entry : int { kFwd = 0, kEx = 1, kPadded = 2, kVarlen = 3, kObjective = 4, kBshd = 5 };

struct Call {
  Entry entry;
  const void *Q, *K, *V;
  void* Y;
  int batch, heads, N, d, b, T, dtype;
  float scale;          // not read for kFwd (1 / sqrt(d))
  int path;             // kEx, kObjective, kBshd
  int n_valid;          // kPadded
  const int* seq_len;   // kVarlen
  float* lse;           // kObjective
  void* ws;             // nullptr: ask `alloc` (kFwd uses the library's own)
  size_t ws_bytes;
  void* stream;
  void* (*alloc)(void* ctx, size_t bytes);
  void* ctx;
  int whole;            // heads of the call that this one is a part of, whose kernels it then takes; 0: it is no part
};

}  // namespace ma

extern "C" int monarch_attn_internal_run(const ma::Call* call);
