/*
 * koala_debug.h -- diagnostic exports of libkoala that are not part of its interface: kernel
 * tuning for A/B runs, a launch counter, a self-test of the bounded-wait error path and a check
 * of the guard words between workspace buffers.  Used by the test-suite and the measurement
 * scripts; nothing here is needed to run the draft-then-verify step.
 */
#ifndef KOALA_DEBUG_H_
#define KOALA_DEBUG_H_

#include "../../include/koala.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Process-wide tuning of the tensor-core matrix multiply (the defaults are chosen for B200):
 * key 1 = shared-memory pipeline stages per CTA (0 = as many as fit, at most 8); key 2 = upper
 * bound on the automatic split-K factor (0 = default); key 3 = 1 switches stream-K off (every CTA
 * stays inside one weight tile); key 6 = 1 delays the weight stream until the previous kernel has finished;
 * key 7 = divisor of the split-K partial-sum traffic bound (default 8); key 8 = how many pipeline
 * stages request their weight tile at once, before that wait (< 0, the default: two behind programmatic
 * launch, else all; the ring's length or more = all in either case); key 9 = fewest query
 * rows per sequence for which the tcgen05 attention kernel is used (default 16); key 10 = 1 keeps
 * the one-wave split-K factor when a launch has several token tiles (more than 128 rows);
 * key 11 = 1 keeps 128 weight rows per CTA also for the widest token tiles (MMA N = 256);
 * key 12 = key chunks per (sequence, head) of the tcgen05 attention kernel (0 = chosen from the shape);
 * key 13 = 1 runs pairs of more than 128 tokens as 128-token tiles with the residual rows as extra
 * accumulator columns (the form used up to 128 tokens) instead of 256-token tiles with two accumulating
 * MMAs; keys 15 (256-row weight tiles) and 16 (128-row tiles) = 1, 2 or 4: that many epilogue warps per
 * 32 accumulator lanes instead of the default; key 17 = 1: no CTA-pair GEMM kernel, 2: not up to 128
 * rows; key 18 = fewest rows for it (default 113); key 20 = 0: no dry pass over its
 * tile loop before the dependency wait; key 21 = 0: no dry pass of the GEMM epilogue warps; key 22 =
 * key chunks of the mma.sync attention kernel (0 = by rule); key 23 = 1: pairs of more than 64 rows always
 * summed in short chains (as in prompt forwards); key 24 = SM cycles between the requests of the stages past those of key 8
 * (default 1600; 0 or less = they come with their activations). */
void koala_set_tuning(int key, int value);

/* Kernels launched by the library in this process so far (all contexts). */
uint64_t koala_launch_count(void);

/* Exercises the path a bounded device-side wait takes when it runs out, without anything else in
 * flight: a one-thread kernel on the context's stream initialises an mbarrier that nothing ever
 * arrives at, waits for it for `limit_cycles` SM clock cycles (1 .. 10^8), and on expiry records
 * KOALA_E_TIMEOUT in the context's device status word exactly as the matrix-multiply and
 * attention kernels do.  koala_poll() then reports it.  The status word keeps the code: use a
 * context made for this purpose. */
int koala_selftest_timeout(koala_ctx *ctx, int limit_cycles);

/* Every buffer carved from the workspace is followed by a 256-byte guard that koala_init fills
 * with a fixed pattern and nothing ever writes.  Waits for the context's stream, reads the guards
 * back and counts those that changed (a write past the end of the buffer before it).  n_guards /
 * n_damaged: host ints. */
int koala_debug_check_guards(koala_ctx *ctx, int *n_guards, int *n_damaged);

/* How koala_ingest deals the blocks of B prompts of len[b] tokens to forwards of at most ingest_rows rows,
 * without enqueueing anything: *n_blocks and *n_tokens handed out until the forward with index fail_at
 * (< 0: none) reports KOALA_E_CUDA, which ends the dealing and is returned.  Host memory only. */
int koala_debug_deal_blocks(int B, const int32_t *len, int ingest_rows, int fail_at, int *n_blocks, int *n_tokens);

/* The ring of a CTA of the one-CTA multiply for stages of stage_bytes on a device with smem_optin bytes of shared memory per
 * block: *stages, how many of their weight tiles are requested at once (*early) and the cycles between the others' requests
 * (*pace; 0: they come with the activations).  wide: 256 weight rows per CTA; pdl: programmatic launch.  Host logic only. */
int koala_debug_gemm_ring(int stage_bytes, int smem_optin, int wide, int pdl, int *stages, int *early, int *pace);

/* Rows that a thread of the rotary kernel takes for R rows of a bf16 model of hidden size H whose Q/K/V product left up to n
 * partial sums per column, its `tiles` tiles of kblocks K blocks dealt to `ctas` CTAs or clusters (0: not dealt).  Host logic only. */
int koala_debug_rope_rows(int R, int H, int ctas, int tiles, int kblocks, int n);

#ifdef __cplusplus
}
#endif
#endif /* KOALA_DEBUG_H_ */
