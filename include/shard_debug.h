/*
 * shard_debug.h -- test exports of libshard (not part of the serving path).
 *
 * They expose single pieces of the step so tests can check them bit by bit:
 * the private weight layout read back in natural order, and one projection
 * (the same GEMV kernel the step runs, with a plain fp32 store instead of the
 * fused epilogue).  The fused projections are numbered
 *   0 = q|k|v  (rows: the q rows, then k, then v; inputs H)
 *   1 = o      (rows H; inputs Hq*d)
 *   2 = gate|up (rows: the F gate rows, then the F up rows; inputs H)
 *   3 = down   (rows H; inputs F)
 * Same conventions as shard.h (0 / negative SHARD_E* codes, fp16 as uint16_t).
 */
#ifndef GB300_SHARD_DEBUG_H
#define GB300_SHARD_DEBUG_H

#include <stdint.h>

#include "shard.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Natural row count, input count K, and private-layout bytes of a fused
 * projection of one layer. */
int shard_debug_op_info(shard_t shard, int layer, int op, int* rows, int* K, long long* bytes);

/* Dequantises a fused projection from the library's private layout:
 * out (dev fp32, [rows][ld], ld >= K) receives (q - z) * s in natural order
 * (Section 3.2, Step 4).  Synchronous. */
int shard_debug_unpack(shard_t shard, int layer, int op, float* out, int ld);

/* y[m][r] = sum_k W[r][k] * x[m][k] for m < M (1..16) with the step's GEMV
 * kernel.  x: dev fp16 [M][K]; y: dev fp32 [M][y_ld], y_ld >= rows.  Uses the
 * shard's work buffers: do not overlap with shard_step.  Asynchronous on
 * cuda_stream. */
int shard_debug_gemv(shard_t shard, int layer, int op, const uint16_t* x, int M, float* y, int y_ld,
                     void* cuda_stream);

/* y[n][r] = sum_k W[r][k] * x[n][k] for n < S (any S >= 1) with the
 * many-token tensor-core projection (tcgen05; the prefill path): x dev fp16
 * [S][x_ld], 16-byte aligned, x_ld a multiple of 128 and >= K rounded up to
 * 128, columns K .. x_ld - 1 zero; y dev fp32 [S][y_ld], y_ld >= rows,
 * natural row order.  Same W4A16 arithmetic as the step's projections (exact
 * q - z, fp32 sums, the fp16 group scale applied in fp32).  All of K in one
 * part.  x is first copied into the kernel's order of inputs, in a buffer that the
 * shard keeps and a first or larger call allocates (not under stream capture).
 * Asynchronous on cuda_stream. */
int shard_debug_gemm(shard_t shard, int layer, int op, const uint16_t* x, int x_ld, int S, float* y, int y_ld,
                     void* cuda_stream);

/* The many-token projection as shard_prefill launches it.  x dev fp16 [S][x_ld] as
 * for shard_debug_gemm, but each block of 32 inputs in the kernel's order: input k
 * at 16 ((k >> 2) & 1) + 4 ((k >> 3) & 3) + (k & 3).  Either y: dev fp32, K in
 * `parts` parts (1..4, at most K / 128 rounded up; 0: as many as a prefill of S
 * tokens takes), part p's sums at y + p * y_part, [S][y_ld], natural rows.  Or h
 * (op 2, parts 0 or 1): dev fp16 [S][h_ld], silu(gate) * up in the same order of
 * inputs, h_ld a multiple of 8 and >= F rounded up to 128; values past F are left as
 * they are.  Nothing is allocated.  Asynchronous on cuda_stream.  Returns the parts
 * (1..4), or a negative error. */
int shard_debug_gemm_stage(shard_t shard, int layer, int op, const uint16_t* x, int x_ld, int S, int parts, float* y,
                           int y_ld, long long y_part, uint16_t* h, int h_ld, void* cuda_stream);

/* The many-token projection's token tile for S tokens and its rings, for a
 * model of its barriers: rings[0..5] = stages of weight units, of token tiles
 * and of the dequantised A operand, accumulators, MMA-issuing threads,
 * dequantise sets.  Host only: needs no shard and no GPU. */
int shard_debug_gemm_rings(int S, int group, int* tile, int* rings);

/* Phase durations of the last completed shard_step, from the GPU's global
 * timer read by one thread at the end of each grid-barrier wait of the step
 * kernel: us[i] is the time between the end of wait i and the end of wait
 * i + 1 (time 0 = kernel start).  Order, 4 * n_layers + 1 values: the
 * prologue with the first RMSNorm and q|k|v projection; then per layer:
 * attention, o, RMSNorm + gate|up, down, and (except after the last layer)
 * the next layer's RMSNorm + q|k|v projection merged into its attention.
 * Returns the number of values written (at most n), or a negative error.
 * Synchronises the device. */
int shard_debug_phase_times(shard_t shard, double* us, int n);

/* Test knob for kv_state_load's staging buffer: gives the present one back and
 * makes later loads behave as if no more than `bytes` of device memory could be
 * had for it (0: none, so the load makes strided copies; -1: no limit). */
int shard_debug_set_load_stage(shard_t shard, long long bytes);

/* Test knob for the step kernel's bounded waits (they must never hang the
 * GPU; the paper has no counterpart): limit = polls before a cross-CTA wait
 * gives up (default 2^22); skip_arrival >= 0 makes CTA 1 leave out its arrival at that grid barrier of every following
 * step (0 = the prologue's), so the other CTAs' waits run out; -1 = off.  A
 * wait that runs out makes the step report "pipeline wait timed out" (EINVAL)
 * through shard_sync_status or the next shard_step, and the KV states stay
 * rejected until kv_state_reset.  Takes effect at the next shard_step. */
int shard_debug_set_wait(shard_t shard, unsigned limit, int skip_arrival);

#ifdef __cplusplus
}
#endif

#endif /* GB300_SHARD_DEBUG_H */
