/*
 * rsb_probe.h — one inner step of librsb on its own, for tests: the eigenpairs of a
 * cycle's projected matrix, which the solvers compute on the device and no call of rsb.h
 * returns.  Not part of the method.
 */
#ifndef RSB_PROBE_H
#define RSB_PROBE_H

#ifdef __cplusplus
extern "C" {
#endif

/*
 * The keep + 1 smallest eigenpairs of the symmetric K x K matrix S, by the kernel that ends
 * a Lanczos cycle (f32 != 0: the FP32 solves' form).  Host arrays: S[K * K] row by row,
 * theta[keep + 1] ascending, Y[K * (keep + 1)] row by row (column i belongs to theta[i]).
 * 1 <= K <= 40, 0 <= keep < K, keep <= 16; RSB_EINVAL otherwise.
 */
int rsb_probe_ritz(int f32, int K, int keep, const double *S, double *theta, double *Y);

#ifdef __cplusplus
}
#endif

#endif /* RSB_PROBE_H */
