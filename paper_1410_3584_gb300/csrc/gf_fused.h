// Fused passes of the gradient flow's inner iteration (gf_fused.cuh), for grids whose last axis
// has a compile-time FFT length.
#pragma once
#include "common.cuh"

namespace nlp {

// device scalars of a gradient-flow step
enum { S_MIN = 0, S_MAX, S_DIFF, S_NORM, S_CHANGE, S_EPOT, S_EINT, S_EKIN,
       S_CHEB_Q, S_CHEB_R0, S_CHEB_R1, S_CHEB_C1, S_CHEB_C2, S_COUNT = 16 };

// flag: [0] first converged inner iteration, [1] first non-finite one (either set: the passes do
// nothing), [2] blocks done, [4..5] the largest update so far (bits of a double)
constexpr int kInnerFlags = 6;

template <typename T>
cudaError_t launch_gf_r2c(const T *phi, const T *b, const T *x, T inv_tau, const double *scal, const int *flag,
                          const DevPlan<T> &P, cudaStream_t st);
template <typename T>
cudaError_t launch_gf_c2r(T *x, T *d, const DevPlan<T> &P, double *scal, int *flag, int it, double tol,
                          cudaStream_t st);

__device__ __forceinline__ bool cheb_ok(double q) { return q > 1e-300 && q < 1.0; }

// inner-iteration bookkeeping: records the first iteration whose update max|x^(m+1) - x^(m)| is <= tol
// (flag[0]) or non-finite (flag[1]); advances the Chebyshev coefficients for the next iteration
__device__ __forceinline__ void inner_check(double *scal, double diff, double tol, int it, int *flag) {
    const double q = scal[S_CHEB_Q];
    if (cheb_ok(q)) {
        const double r0 = it > 1 ? scal[S_CHEB_R1] : q, r1 = 1.0 / (2.0 / q - r0);   // rho_{k-1}, rho_k
        scal[S_CHEB_R0] = r0;
        scal[S_CHEB_R1] = r1;
        scal[S_CHEB_C1] = r1 * r0;
        scal[S_CHEB_C2] = 2.0 * r1 / q;
    }
    scal[S_DIFF] = diff;
    if (flag[0] || flag[1]) return;
    if (!isfinite(diff)) flag[1] = it;
    else if (diff <= tol) flag[0] = it;
}

}  // namespace nlp
