/* Probes of the dynamic quantizers' grid-wide maximum: the quantizer kernels
 * with chosen wait limits, and a kernel that holds SMs, so that tests see the
 * path of a grid whose CTAs are not all resident.  Part of libqlin_probe.so. */
#ifndef QLIN_GRID_PROBE_H
#define QLIN_GRID_PROBE_H

#ifdef __cplusplus
extern "C" {
#endif

/* The dynamic-scale quantizer of x (bf16 [M, K]) with its own limits.
 *   fmt      1 = NVFP4 (out: a qlin_nvfp4_t), 2 = FP8 (out: a qlin_fp8_t)
 *   sync     five device words, 8-byte aligned: the grid's scratch (zero, or
 *            word 3 set to the number of 64 KB pieces of x or more, so that no
 *            piece is left to take); left zero
 *   help_ns  wait for the grid before reading x in the missing CTAs' place
 *            (0: every CTA does so at once), at most 1 ms
 *   stop_ns  wait for the last pieces, at most 1 ms (0: every CTA that finds no
 *            piece left reads all of x for itself)
 *   counts   host array of 3: CTAs that gave up the first wait, pieces they read,
 *            CTAs that read all of x
 * Synchronises the device.  Returns 0, 1 for an invalid argument, 4 for a CUDA
 * error. */
int qlin_probe_grid_max(int fmt, const void *x, long long M, long long K, void *out,
                        unsigned *sync, unsigned long long help_ns, unsigned long long stop_ns,
                        unsigned *counts, void *stream);

/* Occupy `ctas` SMs (a CTA with all of an SM's shared memory each) for `ns`
 * nanoseconds, at most 5 ms.  Asynchronous.  Returns as above. */
int qlin_probe_hold_sms(int ctas, unsigned long long ns, void *stream);

#ifdef __cplusplus
}
#endif

#endif /* QLIN_GRID_PROBE_H */
