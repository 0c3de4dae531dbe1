// Host-side launchers of the device kernels (one per kernel family).
#pragma once
#include "common.cuh"

namespace nlp {

// Dynamic shared-memory opt-in limit of the current device.  Every kernel that may take more
// than the default 48 KB is given, once, the whole opt-in limit minus its static shared
// memory (not the size of the launch at hand), so launches of different sizes from several
// host threads never change a limit that another thread's launch relies on.  The setup runs
// on the device current at the first call.
int max_dyn_smem();
template <auto Kernel> inline cudaError_t allow_smem() {
    static const cudaError_t status = [] {
        cudaFuncAttributes a{};
        cudaError_t e = cudaFuncGetAttributes(&a, Kernel);
        if (e != cudaSuccess) return e;
        return cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    max_dyn_smem() - (int)a.sharedSizeBytes);
    }();
    return status;
}

// A host table to device memory on the stream whose kernels read it; it is there on return, and `src` may
// go.  (A plain cudaMemcpy or cudaMemset runs on the legacy stream, may return before the data has
// arrived, and a stream created non-blocking does not wait for it.)
inline cudaError_t copy_in(void *dst, const void *src, size_t bytes, cudaStream_t st) {
    const cudaError_t e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st);
    return e != cudaSuccess ? e : cudaStreamSynchronize(st);
}

// One strided C2C FFT pass (see k_fft_strided).
struct StridedDesc {
    int n_in, n_out;      // input / output windows (>= N means the whole line)
    int64_t es;           // element stride along the transformed axis (complex units)
    int ncol;             // contiguous columns per outer line
    int nouter;           // outer lines
    int64_t os;           // stride between outer lines
    int outer_map_n;      // > 0: outer index o addresses line (o - outer_map_n/2) mod outer_map_N
    int outer_map_N;
    void *out;            // null: in place; else the output array (same layout as the input)
    const int *skip;      // null, or two flags: the pass is left out if one is set (fixed lengths only)
};

// The passes along axis 1 and axis 0 of an evaluation, restricted to what the nodes reach
// (DevPlan::kz, span): forward a1 then a0 (3D only), inverse b0 (3D only) then b1.
struct EvalPasses {
    StridedDesc a1, a0, b0, b1;
};
template <typename T> inline EvalPasses eval_passes(const DevPlan<T> &D) {
    EvalPasses E{};
    const bool three = D.dim == 3;
    const int kz = D.kz > 0 ? D.kz : D.nh, w0 = D.span[0] > 0 ? D.span[0] : D.nf[0], w1 = D.span[1] > 0 ? D.span[1] : D.nf[1];
    E.a1.n_in = D.n[1];
    E.a1.n_out = w1;
    E.a1.es = D.nh;
    E.a1.ncol = kz;
    E.a1.nouter = three ? D.n[0] : 1;
    E.a1.os = (int64_t)D.nf[1] * D.nh;
    E.a1.outer_map_n = three ? D.n[0] : 0;
    E.a1.outer_map_N = D.nf[0];
    if (three) {
        E.a0.n_in = D.n[0];
        E.a0.n_out = w0;
        E.a0.es = (int64_t)D.nf[1] * D.nh;
        E.a0.ncol = kz;
        E.a0.nouter = w1;
        E.a0.os = D.nh;
        E.a0.outer_map_n = w1 < D.nf[1] ? w1 : 0;
        E.a0.outer_map_N = D.nf[1];
        E.b0 = E.a0;
        E.b0.n_in = w0;
        E.b0.n_out = D.n[0];
    }
    E.b1 = E.a1;
    E.b1.n_in = w1;
    E.b1.n_out = D.n[1];
    return E;
}

template <typename T> cudaError_t launch_fwd_r2c(const T *rho, const DevPlan<T> &P, cudaStream_t st);
template <typename T> cudaError_t launch_inv_c2r(T *phi, const DevPlan<T> &P, cudaStream_t st);
template <typename T>
cudaError_t launch_fft_strided(cpx<T> *data, const StridedDesc &d, const FftLen<T> &L, int sign, cudaStream_t st);
template <typename T>
cudaError_t launch_fft_four(const cpx<T> *in, cpx<T> *out, const StridedDesc &d, const DevPlan<T> &D, int sign,
                            cudaStream_t st);
template <typename T> bool cols_on_reg_engine(const FftLen<T> &L);

// Whether a length has the compile-time kernels that the fused passes need.
bool fft_fixed_len(int N);
// passes of the lengths of fft_other.cuh: true when N is one of them (e: the launch's status)
template <typename T> bool r2c_other(const T *rho, const DevPlan<T> &P, cudaStream_t st, cudaError_t &e);
template <typename T> bool c2r_other(T *phi, const DevPlan<T> &P, cudaStream_t st, cudaError_t &e);
template <typename T>
bool cols_other(cpx<T> *data, const StridedDesc &d, const FftLen<T> &L, int sign, cudaStream_t st, cudaError_t &e);
// y = IFFT(m FFT(x)) along the axis of d (a fixed length), in place; m: an array of the data's
// layout, real or complex, or the product of one factor per axis (a: the axis, o: outer, c: columns).
template <typename T, class V>
cudaError_t launch_fft_mul(cpx<T> *data, const StridedDesc &d, const FftLen<T> &L, const V *m, cudaStream_t st);
template <typename T>
cudaError_t launch_fft_mul3(cpx<T> *data, const StridedDesc &d, const FftLen<T> &L, const cpx<double> *a,
                            const cpx<double> *o, const cpx<double> *c, cudaStream_t st);

template <typename T>
cudaError_t launch_fft_contig(cpx<T> *data, int64_t nlines, const FftLen<T> &L, int sign, T post, cudaStream_t st);

// Fused interpolate -> scale -> spread over all node chunks (see spread.cu): each chunk's
// tile window goes to its slot of P.win; launch_combine then writes every cell of G.
template <typename T> cudaError_t launch_interp_spread(const DevPlan<T> &P, cudaStream_t st);
template <typename T> int generic_warps(const DevPlan<T> &P, size_t smem_limit);
template <typename T> size_t interp_spread_smem(const DevPlan<T> &P, int nwarps);
// 3D ring kernels (see ring_dev.cuh): columns -> strips, nodes, strips -> columns, columns -> G.
template <typename T> cudaError_t launch_ring_cols(const DevPlan<T> &P, cudaStream_t st);
template <typename T> cudaError_t launch_ring_nodes(const DevPlan<T> &P, cudaStream_t st);
template <typename T> cudaError_t launch_ring_inv(const DevPlan<T> &P, cudaStream_t st);
template <typename T> cudaError_t launch_ring_gather(const DevPlan<T> &P, cudaStream_t st);
// 2D ring kernels: nodes (launch_ring_nodes, strips from F), then strips -> G.  FP32 at the default width
// (tolerance 1e-6) only: other tolerances run the generic kernel there, as fast as before the 2D rings
// (64^2 at 1e-5 and 1e-8: 49 and 53 us an evaluation; 37 at 1e-6, 49 with the generic kernel), and each
// more width is another pair of kernels to compile and to test.
template <typename T> cudaError_t launch_ring_gather2(const DevPlan<T> &P, cudaStream_t st);
template <typename T> constexpr bool ring_2d(int w) { return sizeof(T) == 8 ? w >= 8 && w <= 15 : w == 7; }
template <typename T> int ring_xy_stride(int w);                          // a node's row of DevPlan::rg_xy
template <typename T> size_t ring_smem(const DevPlan<T> &P, int warps);   // largest block of `warps` warps
template <typename T> int ring_psi_stride(int w);                         // 0: no ring kernels for this width
template <typename T> cudaError_t launch_window_sum(const DevPlan<T> &P, cudaStream_t st);   // tiles of several chunks
template <typename T> cudaError_t launch_combine(const DevPlan<T> &P, cudaStream_t st);

// 2D Poisson (Algorithm 1) FP64 parts (see poisson2d.cu).  L, h: collapsed 3D view.
template <typename T>
cudaError_t launch_poisson_moments(const T *rho, const DevPlan<T> &P, const double *L, const double *h,
                                   double *part, int nblocks, double *mom, cudaStream_t st);
template <typename T> cudaError_t launch_poisson_origin(const DevPlan<T> &P, double *mom, cudaStream_t st);
template <typename T>
cudaError_t launch_poisson_u1(T *phi, const DevPlan<T> &P, const double *L, const double *h, cudaStream_t st);
// plan time: the u_{1,1}, u_{1,2} table of the grid (3 doubles per point)
cudaError_t launch_u1_table(double *tab, int nx, int ny, const double *L, const double *h, double sigma,
                            cudaStream_t st);

// precomputed-kernel method: F *= K-hat (toeplitz.cu)
template <typename T> cudaError_t launch_mul_spec(cpx<T> *F, const cpx<T> *K, int64_t M, cudaStream_t st);


}  // namespace nlp
