// The two real-grid ends of the gradient flow's inner iteration, fused into the last-axis FFT
// passes.  The iteration is bound by the FP64 rate of its transforms; as separate kernels the
// right-hand side, the update with its reduction, the convergence test and the capture of the
// converged iterate added 48 us and seven launches to 130 us of transforms at 96^3 FP64.
//   - the R2C reads phi^n, b and x and transforms r = phi^n/tau + (alpha - b) x;
//   - the C2R ends in the Chebyshev update d = c1 d + c2 (G(x) - x), x += d; the largest |d| is
//     folded through integer maxima of its bits (order independent, no FP64 operations), and
//     the last block to finish runs the convergence test for the next iteration.
// Iterations past convergence find the flag set and do nothing, so x stays the first converged
// iterate.
#pragma once
#include "fft_launch.cuh"
#include "gf_fused.h"

namespace nlp {

template <typename T> struct RhsSrc {
    const T *__restrict__ phi, *__restrict__ b, *__restrict__ x;
    T inv_tau, alpha;
    __device__ __forceinline__ T operator()(int64_t i) const { return phi[i] * inv_tau + (alpha - b[i]) * x[i]; }
};

template <typename T, int NBC, int TPC, class FL>
__global__ void __launch_bounds__(NBC * TPC, line_blocks<FL, T>()) k_gf_r2c(const T *phi, const T *b, const T *x, T inv_tau,
                                                         const double *scal, const int *flag, DevPlan<T> P) {
    extern __shared__ __align__(16) unsigned char smraw[];
    if (flag[0] | flag[1]) return;
    const RhsSrc<T> src{phi, b, x, inv_tau, (T)(0.5 * (scal[S_MIN] + scal[S_MAX]))};
    fwd_r2c_reg_block<T, NBC, true, TPC, FL>(src, P, blockIdx.x, smraw);
}

template <typename T> struct ChebOut {
    T *__restrict__ x, *__restrict__ d;
    double c1, c2;
    unsigned long long m;   // bits of the largest |update| (a NaN is larger than any number)
    __device__ __forceinline__ void operator()(int64_t i, T g) {
        const T xi = x[i];
        const double r = (double)g - (double)xi;
        const T dn = (T)(c1 == 0.0 ? c2 * r : c1 * (double)d[i] + c2 * r);   // c1 = 0: d is not set yet
        d[i] = dn;
        x[i] = xi + dn;
        const unsigned long long u = (unsigned long long)__double_as_longlong((double)dn) & 0x7fffffffffffffffull;
        m = u > m ? u : m;
    }
};

template <typename T, int NBC, int TPC, class FL>
__global__ void __launch_bounds__(NBC * TPC, line_blocks<FL, T>()) k_gf_c2r(T *x, T *d, DevPlan<T> P, double *scal, int *flag, int it,
                                                         double tol) {
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned long long s_max;
    if (flag[0] | flag[1]) return;   // (set by earlier launches only, or by this one after every block is done)
    if (threadIdx.x == 0) s_max = 0;
    __syncthreads();
    ChebOut<T> out{x, d, scal[S_CHEB_C1], scal[S_CHEB_C2], 0ull};
    inv_c2r_reg_block<T, NBC, TPC, FL>(out, P, blockIdx.x, smraw);
    atomicMax(&s_max, out.m);
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long *gmax = reinterpret_cast<unsigned long long *>(flag + 4);
        atomicMax(gmax, s_max);
        __threadfence();
        if (atomicAdd(flag + 2, 1) == (int)gridDim.x - 1) {
            __threadfence();
            const unsigned long long u = atomicExch(gmax, 0ull);
            flag[2] = 0;
            inner_check(scal, __longlong_as_double((long long)u), tol, it, flag);
        }
    }
}

template <typename T>
cudaError_t launch_gf_r2c(const T *phi, const T *b, const T *x, T inv_tau, const double *scal, const int *flag,
                          const DevPlan<T> &P, cudaStream_t st) {
    cudaError_t e = cudaErrorInvalidValue;
    with_fixed_len(P.len[2], [&](auto fl) {
        using FL = decltype(fl);
        constexpr int TPC = line_threads<FL, T>(), NBC = line_count<FL, T>();
        const int64_t npairs = (int64_t)P.n[0] * P.n[1] / 2;
        const size_t sm = sizeof(cpx<T>) * (size_t)NBC * line_ld(P.len[2].N) * r2c_buffers<FL>();
        if ((e = allow_smem<k_gf_r2c<T, NBC, TPC, FL>>()) != cudaSuccess) return;
        k_gf_r2c<T, NBC, TPC, FL><<<(unsigned)((npairs + NBC - 1) / NBC), NBC * TPC, sm, st>>>(phi, b, x, inv_tau, scal,
                                                                                              flag, P);
        e = cudaGetLastError();
    });
    return e;
}

template <typename T>
cudaError_t launch_gf_c2r(T *x, T *d, const DevPlan<T> &P, double *scal, int *flag, int it, double tol,
                          cudaStream_t st) {
    cudaError_t e = cudaErrorInvalidValue;
    with_fixed_len(P.len[2], [&](auto fl) {
        using FL = decltype(fl);
        constexpr int TPC = line_threads<FL, T>(), NBC = line_count<FL, T>();
        const int64_t npairs = (int64_t)P.n[0] * P.n[1] / 2;
        const size_t sm = sizeof(cpx<T>) * (size_t)NBC * line_ld(P.len[2].N) * fixed_buffers<FL>();
        if ((e = allow_smem<k_gf_c2r<T, NBC, TPC, FL>>()) != cudaSuccess) return;
        k_gf_c2r<T, NBC, TPC, FL><<<(unsigned)((npairs + NBC - 1) / NBC), NBC * TPC, sm, st>>>(x, d, P, scal, flag, it,
                                                                                              tol);
        e = cudaGetLastError();
    });
    return e;
}

}  // namespace nlp
