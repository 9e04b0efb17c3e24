/*
 * cc3_debug.h -- diagnostic entry points of libcc3 (not part of the hot path).
 *
 * cc3_debug_split_gemm runs ONE plain contraction C[m][n] = sum_k A[m][k] B[n][k]
 * (row-major float64 host arrays A[M][K], B[N][K], C[M][N]) through the split
 * precision tensor-core engine that the CC3 triples kernels use: both operands
 * are cut into `slices` integer-valued BF16 slices with one power-of-two scale
 * each, the slice-product triangle runs on tcgen05 tensor cores with exact
 * FP32 accumulation of the leading levels, and the result is recombined in
 * double-float and accumulated in FP64.  It exists to test the engine in
 * isolation against a plain FP64 product.  Allocates and frees its own device
 * memory; synchronous; returns a cc3 status (CC3_ERR_ARG for sizes < 1 or
 * slices outside 3..7).
 */
#ifndef CC3_DEBUG_H
#define CC3_DEBUG_H
#include <stddef.h>
#ifdef __cplusplus
extern "C" {
#endif
int cc3_debug_split_gemm(int M, int N, int K, const double *A, const double *B, double *C,
                         int slices);

/* Runs one bounded device wait that cannot succeed (one thread of one CTA
 * waits on an mbarrier nothing arrives on, nothing else in flight) with a
 * limit of limit_s seconds (1e-6 <= limit_s <= 1), the same bounded-wait
 * primitive every spin of the library's kernels uses.  Returns
 * CC3_ERR_TIMEOUT once the kernel has recorded the give-up in its status word
 * and returned (the CUDA context stays usable), CC3_ERR_ARG for a limit out
 * of range.  Synchronous, on the legacy default stream of the current device.
 * Exists to test the failure path without a GPU fault. */
int cc3_debug_wait_timeout(double limit_s);

/* The split densities' D_oo kernel alone: D_oo[l][k] (row-major, no x no) of
 * given double-float tensors tau and L3~, host arrays [T][a][b][c][2] (high part,
 * low part) over the triples i >= j >= k in loop order, i = j = k included:
 *   D_oo[l][k] = -1/2 sum_{i >= j} (2 - delta_ij) sum_{abc} L3~^{abc}_{ijk} tau^{abc}_{ijl},
 * L3~ taken as zero at i = j = k; each tensor read in the order of (i, j, k) that
 * its triple stores.  blocks_per_pair: thread blocks that share a pair's sum (0:
 * as in cc3_density_triples); fewer give each thread longer sums.  Exists to
 * measure the sums' rounding.  Synchronous, on the legacy default stream. */
int cc3_debug_doo_pairs(int no, int nv, const float *tau, const float *lt, double *D_oo,
                        int blocks_per_pair);

/* Bytes that the library's pool on the current device holds, those in use, and
 * the most in use since the last call (which starts that count anew).  Waits for
 * the device.  CC3_ERR_UNSUPPORTED where the device has no pools. */
int cc3_debug_memory(size_t *held, size_t *used, size_t *peak);
#ifdef __cplusplus
}
#endif
#endif
