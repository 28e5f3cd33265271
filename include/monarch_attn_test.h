/* libmonarch_attn -- test and profiling hooks.  Not part of the production interface: the first
 * two change process-wide state, and knob 2 makes the library return garbage on purpose.  They exist so
 * that the tests can watch a bounded device-side wait run out without faulting or hanging a GPU,
 * and so that the pipeline of the persistent kernels can be timed stage by stage. */
#ifndef MONARCH_ATTN_TEST_H_
#define MONARCH_ATTN_TEST_H_

#include <stddef.h>

#ifdef __cplusplus
extern "C" {
#endif

/* Profiling aid for the persistent tensor path.  With a DEVICE buffer of at least 4*64*8 int64
 * set, CTAs 0-3 of later MA_PATH_TENSOR / MA_PATH_TENSOR_TMEM launches write SM-clock stamps
 * [cta][tile][event] for their first 64 tiles; events: 0 operands requested, 1 score MMA issued,
 * 2 softmax group sees the scores, 3 P written, 4 apply MMA issued, 5 softmax group sees O,
 * 6 rows staged, 7 rows stored and signalled (MA_PATH_TENSOR_TMEM: output unit given back).  NULL switches it off (the default).  Process-wide;
 * the buffer stays owned by the caller. */
int monarch_attn_set_trace_buffer(void* device_buffer, size_t bytes);

/* Test and tuning knobs (process-wide; not for production use):
 *   knob 1: bound, in SM clocks, of the waits of the persistent tensor path and of the tcgen05 tiles (value <= 0
 *           restores the default 2e9, which the other kernels keep);
 *   knob 2: non-zero withholds something that later launches wait for: the persistent tensor path leaves its first
 *           half-step out, so that the dependency waits of the second can never be satisfied, the kernels whose
 *           operands come by TMA (position split, per-head, tcgen05 tiles) ask for less than they wait for.
 *           Together the two let a test watch a wait run out: the kernel ends by itself, results are
 *           garbage, and monarch_attn_device_status reports MA_ERR_TIMEOUT.  Nothing faults or hangs.
 *   knob 3: number of chunks monarch_attn_fwd_host cuts a call into (1..8; 0, the default: by
 *           the size of the tensors). */
int monarch_attn_debug_knob(int knob, long long value);

/* Which set of kernels served the last successful call on this host thread: "generic", "fused_small", "fused_head",
 * "fused_f32", "jsplit", "tile_mma", "tile_tc", "tensor_decoupled", "tensor_chain", "tensor_tmem", "tensor_basic" ("" before the first).
 * Three of the paths of monarch_attn.h have two sets each, chosen by size. */
const char* monarch_attn_last_kernels(void);

#ifdef __cplusplus
}
#endif
#endif /* MONARCH_ATTN_TEST_H_ */
