/*
 * lsp_tuning.h -- internal knobs of the B200 LSP decode library, for the micro-benchmarks and the kernel tests.
 *
 * Not part of the public contract (include/lsp.h): the keys name tile shapes, grids and benchmark aids of the current
 * kernels and change with them.  None of them changes what the library computes, except keys 3-5, which change how
 * lsp_op_linear behaves as a timing harness.
 */
#ifndef LSP_TUNING_H_
#define LSP_TUNING_H_

#include "../../include/lsp.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Benchmark aids:
 *   3  lsp_op_linear returns without synchronising or checking the device status (1) or not (0)
 *   4  lsp_op_linear enqueues the operation this many times
 *   5  repetition r reads its weights at W + (r mod value) * N * K elements, so a buffer of several weight copies keeps
 *      the L2 cold
 * tcgen05 GEMM, up to 128 rows (the persistent kernel k_gemm_stream):
 *   10 CTAs a launch whose tiles are split is dealt to (0 = by the tile count)          11 maximum pipeline stages
 *   17 its grid (1: one CTA per SM with even shares; else, the default, a multiple of the tile count)
 *   21 64-element K atoms per pipeline stage (0 = automatic, 1, 2)   22 fewest two-atom stages the automatic choice accepts
 *   23 its tile width (0 = automatic, 128, 256)
 *   25 launch the step's kernels with programmatic dependent launch (1, default) or plainly (0)
 *   29 the K slices of a split tile run as one thread block cluster, reduced through distributed shared memory (1,
 *      default), or through global scratch by the last CTA to arrive (0)
 *   32 tile width of the dual (SwiGLU) GEMM: 0 = automatic (default), 192 or 256
 *   43 a SwiGLU tile's weights come by one copy per half and K atom even where one copy can bring them all (0, default)
 *   33 a cluster of 2 exchanges half tiles (1, default) or publishes whole partial tiles like larger clusters (0)
 *   44 ... from this many rows on (default 64)
 * GEMM on pairs of SMs, more than 128 rows (k_gemm_pair):
 *   41 its tile width (0 = automatic, 64 ... 256 in steps of 32; the rotary projection ignores a width that is no
 *      multiple of 64)   42 most row groups of 256 per band (0 = automatic)
 *   46 its K slices (0 = automatic, 1 = never split, 2 or 3 where they fit)
 * tcgen05 attention:
 *   28 fewest (query row x group head) rows of a (sequence, KV head) for which the tcgen05 kernel is used (default 0)
 *   30 it splits a row tile's keys over a thread block cluster when there are few CTAs (1, default)
 *   47 two row tiles per CTA (k_attn_rows): 0 = where that gives every SM a CTA and saves rounds
 *      (default), 1 = never, 2 = always
 * decode loop:
 *   31 with device-resident block lengths (lsp_set_option key 4), lsp_generate reads every step before sizing the next
 *      once at most this many masked positions per sequence remain (default 8)
 * Accepted without effect (they tuned kernel variants that no longer exist): 18, 19, 20, 24, 26, 27, 36 to 39.
 * Unknown key, or a value outside the range of key 41, 46 or 47: LSP_ERR_ARG. */
int lsp_debug_set(lsp_ctx* ctx, int key, int value);

/* Exercises the bounded-wait recovery path without touching any data: launches one thread that waits, for limit_us
 * microseconds, on a barrier nothing arrives at, and then records the expiry in the context's status word the way the
 * GEMM and attention kernels do.  Returns what a step would return in that situation: LSP_ERR_DEVICE_TIMEOUT (site 99
 * in lsp_last_error), with the status word and the split-K counters cleared again, so that the next call runs normally. */
int lsp_debug_wait_selftest(lsp_ctx* ctx, int limit_us);

#ifdef __cplusplus
}
#endif
#endif /* LSP_TUNING_H_ */
