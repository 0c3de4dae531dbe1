// 1D Poisson potential (Sec. 2.2, the 1D case): phi = U * rho with U(x) = -|x|/2.
//
// The Gaussian G_1 = rho-hat(0) G - (x rho)-hat(0) G' (G of width sigma, unit mass) carries
// the mass and the first moment of rho; its potential u_1 = rho-hat(0) u_{1,1} - (x rho)-hat(0)
// u_{1,2} solves Eq. (1DPois) in closed form.  The rest, u_2 = U * (rho - G_1), has the
// Fourier integrand W(k) = (rho-hat(k) - G_1-hat(k)) / k^2, smooth at k = 0 with
// W(0) = -(x^2 rho)-hat(0)/2 + sigma^2 rho-hat(0)/2, so u_2 is a regular FFT quadrature:
//   rho-hat(k_l) = h e^{i k_l L} sum_m rho_m e^{-2 pi i l m / 2n}      (trapezoid, zero padded)
//   u_2(x_m)     = (dk / 2 pi) sum_l W(k_l) e^{-i k_l L} e^{+2 pi i l m / 2n}
// with k_l = l dk, dk = pi / (n h), l = -n..n-1 (e^{i k_l L} = i^l on this grid), terms with
// |k_l| > P dropped, sigma = 6 sqrt(2) / P.  FP64 throughout (the grids have at most 1024 points).
//
// One evaluation: two launches.  An FFT of 2n points is too small to split over SMs and
// bound by the two FP64 FMAs per clock of the one it runs on (38 us each for 2048 points, 90 us
// the evaluation with five launches), so both transforms are direct sums over all SMs, halved by
// symmetry, with the twiddles e^{-i pi k/n} and what the grid alone decides from plan-time tables
// (21 to 29 us the evaluation at n = 1024, from run to run: the sums take 2 x 1700 clocks of every
// FP64 unit, the rest is latency):
//   k_p1d_forward: a warp per l <= n/2; a lane's m = lane + 32 i all have its parity, so the even
//     and the odd half of the sum, E and O, come from the even and odd lanes: F_l = E + O,
//     F_{n-l} = conj(E - O).  Every block takes the moments of rho itself.
//   k_p1d_inverse: a warp per point m; u_2 is real, so the terms l and n - l join as
//     Re(e) (a_l + s a_{n-l}) + Im(e) (s b_{n-l} - b_l), e = e^{i pi l m/n}, s = (-1)^m.
#include <algorithm>
#include <cmath>
#include <vector>

#include "launch.h"
#include "plan.h"

namespace nlp {

// plan-time tables of an n-point grid, in doubles: twiddles (2n complex), g and s of l = 0..n,
// u_{1,1} and u_{1,2} of the points; then the coefficients of the evaluation at hand (a and b for
// s = +1, a and b for s = -1, l = 0..n/2 each) and its moments {C0, M1}
struct P1dTables {
    const double *tw, *g, *s, *u11, *u12;
    double *coef, *mom;
};
__host__ __device__ static P1dTables p1d_tables(double *base, int n) {
    P1dTables t;
    t.tw = base;
    t.g = base + 4 * n;
    t.s = t.g + n + 1;
    t.u11 = t.s + n + 1;
    t.u12 = t.u11 + n;
    t.coef = base + 4 * n + 2 * (n + 1) + 2 * n;
    t.mom = t.coef + 4 * (n / 2 + 1);
    return t;
}
static size_t p1d_table_size(int n) { return 4 * (size_t)n + 2 * (n + 1) + 2 * (size_t)n + 4 * (n / 2 + 1) + 2; }

constexpr int kP1dBlock = 128;

// n16 16-byte pieces to shared memory, asynchronously (all in flight at once); cp_wait before a barrier
__device__ __forceinline__ void cp_all(void *dst, const void *src, int n16) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    for (int i = threadIdx.x; i < n16; i += kP1dBlock)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16u * i), "l"((const char *)src + 16 * (size_t)i)
                     : "memory");
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// i^q for integer q, times v
__device__ __forceinline__ cpx<double> mul_ipow(cpx<double> v, int q) {
    switch (q & 3) {
        case 0: return v;
        case 1: return mk<double>(-v.y, v.x);
        case 2: return mk<double>(-v.x, -v.y);
        default: return mk<double>(v.y, -v.x);
    }
}

__global__ void __launch_bounds__(kP1dBlock) k_p1d_forward(const double *__restrict__ rho, int n, double L, double h,
                                                           double sigma, double *base) {
    extern __shared__ __align__(16) unsigned char smraw[];
    cpx<double> *tw = (cpx<double> *)smraw;      // [2n]
    double *r = (double *)(tw + 2 * n);          // [n]
    __shared__ double part[3][kP1dBlock / 32];
    const P1dTables T = p1d_tables(base, n);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    cp_all(tw, T.tw, 2 * n);
    double c0 = 0.0, m1 = 0.0, m2 = 0.0;
#pragma unroll 8
    for (int m = threadIdx.x; m < n; m += kP1dBlock) {
        const double v = rho[m], x = -L + m * h;
        r[m] = v;
        c0 += v;
        m1 += x * v;
        m2 += x * x * v;
    }
    for (int o = 16; o > 0; o >>= 1) {
        c0 += __shfl_xor_sync(0xffffffffu, c0, o);
        m1 += __shfl_xor_sync(0xffffffffu, m1, o);
        m2 += __shfl_xor_sync(0xffffffffu, m2, o);
    }
    if (lane == 0) {
        part[0][warp] = c0;
        part[1][warp] = m1;
        part[2][warp] = m2;
    }
    cp_wait();
    __syncthreads();
    double mom[3];
    for (int q = 0; q < 3; ++q) {
        mom[q] = part[q][0];
        for (int u = 1; u < kP1dBlock / 32; ++u) mom[q] += part[q][u];
        mom[q] *= h;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        T.mom[0] = mom[0];
        T.mom[1] = mom[1];
    }
    const int l = blockIdx.x * (kP1dBlock / 32) + warp;
    if (2 * l > n) return;
    const int N = 2 * n, step = (int)((32ll * l) % N);
    int k = (l * lane) % N;
    double fx = 0.0, fy = 0.0;
#pragma unroll 4
    for (int m = lane; m < n; m += 32) {
        const cpx<double> e = tw[k];
        const double v = r[m];
        fx = fma(v, e.x, fx);
        fy = fma(v, e.y, fy);
        k += step;
        k -= k >= N ? N : 0;
    }
    // even and odd lanes apart; the upper half warp continues with the imaginary part
    {
        const bool up = lane & 16;
        const double keep = up ? fy : fx, send = up ? fx : fy;
        fx = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
    for (int o = 8; o > 1; o >>= 1) fx += __shfl_xor_sync(0xffffffffu, fx, o);
    const double ex = __shfl_sync(0xffffffffu, fx, 0), ox = __shfl_sync(0xffffffffu, fx, 1);
    const double ey = __shfl_sync(0xffffffffu, fx, 16), oy = __shfl_sync(0xffffffffu, fx, 17);
    if (lane > 1) return;
    // lane 0: l, lane 1: n - l.  y = (dk / 2 pi) W(k_l) e^{-i k_l L}, e^{i k_l L} = i^l
    const int q = lane == 0 ? l : n - l;
    const cpx<double> F = lane == 0 ? mk<double>(ex + ox, ey + oy) : mk<double>(ex - ox, oy - ey);
    const double dk = M_PI / (n * h), g = T.g[q], s = T.s[q];
    cpx<double> y;
    if (q == 0) {
        y = mk<double>((-0.5 * mom[2] + 0.5 * sigma * sigma * mom[0]) * (dk / (2.0 * M_PI)), 0.0);
    } else {
        const cpx<double> g1 = mul_ipow(mk<double>(mom[0] * g, -(q * dk) * mom[1] * g), -q);
        y = scale(scale(F, h) - g1, s);
    }
    const double py = __shfl_down_sync(0x3u, y.x, 1), pi = __shfl_down_sync(0x3u, y.y, 1);
    if (lane == 0) {
        // the terms l and n - l of the sum: once for l = 0 (and n), twice for the others, n/2 has no partner
        const double c = l == 0 ? 1.0 : 2.0;
        const double px = 2 * l == n ? 0.0 : py, pq = 2 * l == n || l == 0 ? 0.0 : pi;
        const int H = n / 2 + 1;
        T.coef[l] = c * (y.x + px);
        T.coef[H + l] = c * (pq - y.y);
        T.coef[2 * H + l] = c * (y.x - px);
        T.coef[3 * H + l] = c * (-pq - y.y);
    }
}

__global__ void __launch_bounds__(kP1dBlock) k_p1d_inverse(double *__restrict__ phi, int n, double *base) {
    extern __shared__ __align__(16) unsigned char smraw[];
    cpx<double> *tw = (cpx<double> *)smraw;      // [2n]
    double *co = (double *)(tw + 2 * n);         // [4][n/2 + 1]
    const P1dTables T = p1d_tables(base, n);
    const int H = n / 2 + 1, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    cp_all(tw, T.tw, 2 * n);
    cp_all(co, T.coef, 2 * H);
    cp_wait();
    __syncthreads();
    const double C0 = T.mom[0], M1 = T.mom[1];
    const int N = 2 * n;
    for (int m = blockIdx.x * (kP1dBlock / 32) + warp; m < n; m += gridDim.x * (kP1dBlock / 32)) {
        const double *a = co + (m & 1) * 2 * H, *b = a + H;
        const int step = (int)((32ll * m) % N);
        int k = (m * lane) % N;
        double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
        for (int l = lane; l < H; l += 32) {
            const cpx<double> e = tw[k];   // e^{-i pi l m / n}
            s0 = fma(a[l], e.x, s0);
            s1 = fma(-b[l], e.y, s1);
            k += step;
            k -= k >= N ? N : 0;
        }
        s0 += s1;
        for (int o = 16; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        if (lane == 0) phi[m] = s0 + C0 * T.u11[m] - M1 * T.u12[m];
    }
}

nlp_status plan_build_1d(nlp_plan_s *p) {
    if (p->prec != NLP_FP64) return NLP_ERR_UNSUPPORTED;
    const int n = p->grid.n[0];
    const double L = p->grid.L[0];
    const double h = 2.0 * L / n;
    double P = M_PI / h;
    if (p->opts.kmax > 0) P = std::min(P, p->opts.kmax);
    p->p1d_n = n;
    p->p1d_P = P;
    p->sigma = 6.0 * std::sqrt(2.0) / P;
    p->n3[0] = p->n3[1] = 1;
    p->n3[2] = n;
    p->L3[2] = L;
    p->h[2] = h;
    nlp_status s;
    void *d;
    std::vector<double> t(p1d_table_size(n), 0.0);
    const double dk = M_PI / (n * h), sg = p->sigma;
    for (int k = 0; k < 2 * n; ++k) {
        t[2 * k] = std::cos(M_PI * k / n);
        t[2 * k + 1] = -std::sin(M_PI * k / n);
    }
    const P1dTables T = p1d_tables(t.data(), n);
    for (int l = 0; l <= n; ++l) {
        const double k = l * dk;
        const_cast<double *>(T.g)[l] = std::exp(-0.5 * k * k * sg * sg);
        const_cast<double *>(T.s)[l] = l == 0 || k > P ? 0.0 : dk / (2.0 * M_PI) / (k * k);
    }
    for (int m = 0; m < n; ++m) {
        const double x = -L + m * h, e = std::erf(x / (M_SQRT2 * sg));
        const_cast<double *>(T.u11)[m] = -sg / std::sqrt(2.0 * M_PI) * std::exp(-x * x / (2.0 * sg * sg)) - 0.5 * x * e;
        const_cast<double *>(T.u12)[m] = -0.5 * e;
    }
    if ((s = alloc_dev(p, &d, sizeof(double) * t.size()))) return s;
    if (copy_in(d, t.data(), sizeof(double) * t.size(), p->stream) != cudaSuccess) return NLP_ERR_CUDA;
    p->p1d_tab = (double *)d;
    p->info.dim = 1;
    p->info.kernel = p->kernel;
    p->info.precision = p->prec;
    p->info.n[0] = p->info.n[1] = 1;
    p->info.n[2] = n;
    p->info.nf[0] = p->info.nf[1] = 1;
    p->info.nf[2] = 2 * n;
    p->info.kmax = P;
    p->info.sigma_poisson = p->sigma;
    p->info.workspace_bytes = p->bytes;
    return NLP_OK;
}

nlp_status eval_1d(nlp_plan_s *p, const double *rho, double *phi) {
    const int n = p->p1d_n;
    cudaStream_t st = p->stream;
    const size_t fwd = sizeof(double) * 5 * (size_t)n, inv = sizeof(double) * (4 * (size_t)n + 4 * (n / 2 + 1));
    if (allow_smem<k_p1d_forward>() != cudaSuccess || allow_smem<k_p1d_inverse>() != cudaSuccess) return NLP_ERR_CUDA;
    constexpr int per = kP1dBlock / 32;
    k_p1d_forward<<<(n / 2 + per) / per, kP1dBlock, fwd, st>>>(rho, n, p->grid.L[0], p->h[2], p->sigma, p->p1d_tab);
    if (cudaGetLastError() != cudaSuccess) return NLP_ERR_CUDA;
    k_p1d_inverse<<<std::min((n + per - 1) / per, 152), kP1dBlock, inv, st>>>(phi, n, p->p1d_tab);
    return cudaGetLastError() == cudaSuccess ? NLP_OK : NLP_ERR_CUDA;
}

}  // namespace nlp
