// Interpolation/spreading device code of the generic kernel, shared by the single-plan kernel
// (spread.cu) and the batched persistent kernel (batch.cu): per-block bodies with the
// block index passed explicitly.  Each body processes one chunk and writes the chunk's tile
// window to its scratch slot (the combine pass of spread_common.cuh folds the slots into G).
#pragma once
#include "common.cuh"
#include "spread_common.cuh"

namespace nlp {

// ======================================================================= generic kernel
// One warp per node (lanes over the taps of the last two axes, a loop over the first), for
// 2D plans and for 3D plans the ring kernels do not cover.  Each warp spreads into its
// own copy of the tile window (plain read-modify-write: within a node the lanes own distinct
// cells, and a warp's nodes follow each other), and the copies are summed in warp order
// when the chunk's window is written out.
//
// Shared memory: F window, nwin warp windows, kernel values of nwin warps, row tables.
template <typename T> __host__ __device__ constexpr size_t generic_win_table_offset(size_t WW, int nwin) {
    return align16((size_t)(1 + nwin) * WW * sizeof(cpx<T>) + (size_t)nwin * 3 * kMaxWidth * sizeof(T));
}
template <typename T> __host__ __device__ constexpr size_t generic_smem_bytes(size_t WW, size_t rows, int nwin) {
    return generic_win_table_offset<T>(WW, nwin) + 2 * rows * sizeof(int64_t);
}

template <typename T>
__device__ __forceinline__ void spread_generic_block(const DevPlan<T> &P, int bid, unsigned char *smraw) {
    const int w = P.w;
    const int w0 = P.dim == 3 ? w : 1;
    const int W0 = P.win_n[0], W1 = P.win_n[1], W2 = P.win_n[2];
    const int WW = W0 * W1 * W2;
    const int nw = blockDim.x >> 5;
    cpx<T> *sF = (cpx<T> *)smraw;
    cpx<T> *sGall = sF + WW;
    T *spsi = (T *)(sGall + (size_t)nw * WW);
    const int rows = W0 * W1;
    int64_t *rowoff = (int64_t *)(smraw + generic_win_table_offset<T>(WW, nw)), *rowmir = rowoff + rows;
    const Chunk ch = P.chunks[bid];

    window_row_table(P, ch, W0, W1, rowoff, rowmir);
    const WinCol wc = window_col(P, ch, W2, rows);
    __syncthreads();
    if (!P.ones_mode) window_fill(P, wc, rowoff, rowmir, rows, W2, sF);
    for (int q = threadIdx.x; q < nw * WW; q += blockDim.x) sGall[q] = mk<T>(0, 0);
    __syncthreads();

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T *ps = spsi + warp * 3 * kMaxWidth;
    cpx<T> *sG = sGall + (size_t)warp * WW;
    const T two_w = (T)2 / (T)w;
    const int sa = W1 * W2;
    for (int j = ch.j0 + warp; j < ch.j1; j += nw) {
        const T d0 = P.nd[4 * (int64_t)j + 0], d1 = P.nd[4 * (int64_t)j + 1];
        const T d2 = P.nd[4 * (int64_t)j + 2], om = P.nd[4 * (int64_t)j + 3];
        const uint32_t o = P.no[j];
        const int o0 = o & 0xff, o1 = (o >> 8) & 0xff, o2 = (o >> 16) & 0xff;
        for (int t = lane; t < 3 * kMaxWidth; t += 32) {
            const int ax = t / kMaxWidth, tt = t % kMaxWidth;
            T v = (T)0;
            if (ax == 0) v = (w0 == 1) ? (tt == 0 ? (T)1 : (T)0) : (tt < w ? es_kernel<T>(((T)tt - d0) * two_w, P.beta) : (T)0);
            else if (tt < w) v = P.psi_gen ? P.psi_gen[((int64_t)j * 3 + ax) * w + tt]
                                           : es_kernel<T>(((T)tt - (ax == 1 ? d1 : d2)) * two_w, P.beta);
            ps[t] = v;
        }
        __syncwarp();
        // interpolation
        cpx<T> acc = mk<T>(0, 0);
        if (!P.ones_mode)
            for (int p = lane; p < w * w; p += 32) {
                const int b = p / w, c = p % w;
                const T wbc = ps[kMaxWidth + b] * ps[2 * kMaxWidth + c];
                const cpx<T> *col = sF + (o0 * W1 + (o1 + b)) * W2 + (o2 + c);
                T sx = 0, sy = 0;
                for (int a = 0; a < w0; ++a) {
                    const T wa = ps[a];
                    const cpx<T> f = col[a * sa];
                    sx += wa * f.x;
                    sy += wa * f.y;
                }
                acc.x += wbc * sx;
                acc.y += wbc * sy;
            }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
        }
        cpx<T> cj;
        if (P.ones_mode) {
            cj = mk<T>(om, (T)0);
        } else if (P.pois == nullptr) {
            cj = scale(acc, om);
        } else {
            // Algorithm 1: W(k) = (rho-hat(k) - (C0 - i k.M1) e^{-sigma^2 |k|^2/2}) / |k| in FP64
            // (om already holds (2pi)^-2 w_r w_phi / |k|)
            const double kx = P.pois[3 * (int64_t)j], ky = P.pois[3 * (int64_t)j + 1], kr = P.pois[3 * (int64_t)j + 2];
            const double g = exp(-0.5 * P.sigma * P.sigma * kr * kr);
            const double re = P.hvol * (double)acc.x - P.mom[0] * g;
            const double im = P.hvol * (double)acc.y + (kx * P.mom[1] + ky * P.mom[2]) * g;
            cj = mk<T>((T)((double)om * re), (T)((double)om * im));
        }
        // spreading into this warp's window
        for (int p = lane; p < w * w; p += 32) {
            const int b = p / w, c = p % w;
            const T wbc = ps[kMaxWidth + b] * ps[2 * kMaxWidth + c];
            const cpx<T> v = scale(cj, wbc);
            cpx<T> *col = sG + (o0 * W1 + (o1 + b)) * W2 + (o2 + c);
            for (int a = 0; a < w0; ++a) {
                const T wa = ps[a];
                cpx<T> g = col[a * sa];
                g.x += v.x * wa;
                g.y += v.y * wa;
                col[a * sa] = g;
            }
        }
        __syncwarp();
    }
    __syncthreads();
    cpx<T> *out = P.win + (int64_t)bid * P.win_cells;
    for (int q = threadIdx.x; q < WW; q += blockDim.x) {
        cpx<T> s = sGall[q];
        for (int k = 1; k < nw; ++k) s = s + sGall[(size_t)k * WW + q];
        out[q] = s;
    }
}

}  // namespace nlp
