/*
 * lbm_bench.h -- measurement helpers of libmrtlbm.so that are not part of the
 * method: arithmetic-throughput probes that give the ALU rooflines of the
 * step kernels a measured denominator, and the launches that lbm_step makes
 * (the paper has no counterpart).
 *
 * Same conventions as lbm.h: 0 on success, a negative LBM_* code otherwise.
 */
#ifndef LBM_BENCH_H
#define LBM_BENCH_H

#include "lbm.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Throughput of dependent-free fused multiply-adds on device `device`
 * (-1: the current one), timed with CUDA events over `reps` launches after
 * one warm-up launch; each launch covers every SM with independent FMA
 * chains.  kind 0: FP64 (fma.rn.f64), 1: FP32 (fma.rn.f32), 2: packed
 * FP32x2 (fma.rn.f32x2, two FMAs per instruction).  *fma_per_s receives
 * thread-level FMA operations per second (a packed instruction counts two;
 * FLOP/s = 2 x this) and *inst_per_s (may be NULL) thread-level
 * instructions per second.  Allocates and frees a small device buffer; runs
 * on the legacy default stream and synchronises the device.
 * Errors: LBM_ERR_ARG (kind, reps < 1 or NULL output), LBM_ERR_CUDA. */
int lbm_bench_fma_peak(int kind, int device, int reps, double *fma_per_s, double *inst_per_s);

/* Time steps that one launch of lbm_step takes, where that many are due, on a
 * cavity of nx x ny nodes with these options: 1, 2 or 4 in *steps, and in
 * *kernel (may be NULL) which kernel takes them: the one-step kernel of the
 * storage and layout, a window held by each SM (small grids) or strips (large
 * ones).  sms: the SMs of the GPU; 0 asks the device of the options.  Makes no
 * CUDA call with sms > 0.  Errors: LBM_ERR_ARG (NULL, a size below 2, sms < 0),
 * LBM_ERR_CUDA. */
enum { LBM_LAUNCH_STEP = 0, LBM_LAUNCH_TILE = 1, LBM_LAUNCH_STRIPS = 2 };
int lbm_bench_steps_per_launch(int nx, int ny, const lbm_opts *opts, int sms, int *steps, int *kernel);

#ifdef __cplusplus
}
#endif
#endif
