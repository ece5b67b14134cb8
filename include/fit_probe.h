/*
 * fit_probe.h -- measurement and test probes of libfit (C ABI).
 *
 * Not part of the fit.  fit_probe_fp32 measures the FP32 ceiling that the
 * fused kernel's rate is compared with: it is derived from unit counts (SMs x
 * 128 FP32 lanes x 2 flops x clock), and the probe checks it on the device the
 * fit runs on, with scalar and with packed (two-lane) fused multiply-adds.
 * The others let tests see what no entry point shows: the FP64 arithmetic by
 * itself, whether host buffers are taken in place, a training whose blocks do
 * not meet.  The paper has no counterpart.
 */
#ifndef FIT_PROBE_H
#define FIT_PROBE_H

#include <stdint.h>

#include "fit.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Threads per block of the probe. */
#define FIT_PROBE_THREADS 256

/*
 * fit_probe_fp32: launches an FP32 throughput kernel on the CURRENT device,
 * on `stream` (a cudaStream_t; NULL = the default stream), and returns at
 * once; time it with events on the same stream.
 *
 *   packed  0: every thread runs 16 independent chains of scalar fused
 *           multiply-adds (fma.rn.f32); 1: 16 chains of packed two-lane
 *           fused multiply-adds (fma.rn.f32x2), i.e. 32 FP32 FMAs per round.
 *   blocks  grid size (>= 1), FIT_PROBE_THREADS threads each.
 *   iters   rounds per thread (>= 1).
 *   out     DEVICE buffer of at least blocks x FIT_PROBE_THREADS floats
 *           (caller-owned); each thread writes the sum of its chains there
 *           so that no chain can be optimised away.
 *   flops   HOST pointer; receives the FP32 flops the launch performs
 *           (an FMA counts as 2): blocks x threads x iters x 16 x 2
 *           (x 2 again when packed).
 *
 * Returns FIT_OK (0), FIT_ERR_ARG (-1) on a bad argument, FIT_ERR_CUDA (-2)
 * if the launch fails (message in fit_last_error()).
 */
int fit_probe_fp32(int packed, int blocks, int iters, float* out, void* stream, double* flops);

/*
 * fit_probe_f64: the FP64 fit's arithmetic, out[i] = op(x[i], y[i]) for i < n
 * (DEVICE arrays of n doubles), asynchronous on `stream`:
 *   FIT_PROBE_RCP 1 / x, _DIV x / y, _RSQRT 1 / sqrt(x), _SQRT sqrt(x), _TAN
 *   x / y and _SLOPE x / (y y) as the plane propagation forms them, _ATAN
 *   atan(x) / x for |x| < 1/4.
 * Returns FIT_OK, FIT_ERR_ARG or FIT_ERR_CUDA.
 */
#define FIT_PROBE_RCP 0
#define FIT_PROBE_DIV 1
#define FIT_PROBE_RSQRT 2
#define FIT_PROBE_SQRT 3
#define FIT_PROBE_TAN 4
#define FIT_PROBE_SLOPE 5
#define FIT_PROBE_ATAN 6
#define FIT_PROBE_OPS 7
int fit_probe_f64(int op, const double* x, const double* y, int64_t n, double* out, void* stream);

/*
 * fit_probe_host_in_place: whether fit_propagate_update_host would take these
 * buffers of n tracks in place (1) or stage them (0) on the current device; a
 * question to the driver, nothing runs.  FIT_ERR_ARG on a bad argument.
 */
int fit_probe_host_in_place(const fit_tracks_in* in, const fit_tracks_out* out,
                            const fit_hits* hits, int64_t n, int nlayer);

/*
 * fit_probe_train_limits: for the tests of fit_mlp_train, how often a block of
 * its kernel looks at the barrier before it gives up (as created: 2^22), and
 * the most blocks it may count on to run together (0: as many as the device
 * holds).  FIT_ERR_ARG if m is NULL or blocks < 0.
 */
int fit_probe_train_limits(fit_mlp* m, uint32_t looks, int blocks);

#ifdef __cplusplus
}
#endif

#endif /* FIT_PROBE_H */
