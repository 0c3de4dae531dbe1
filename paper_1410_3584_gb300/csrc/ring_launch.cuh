// Kernels and launchers of the ring decomposition (included once per precision by ring_f32.cu
// and ring_f64.cu).
#pragma once
#include "common.cuh"
#include "launch.h"
#include "ring_dev.cuh"

namespace nlp {

constexpr int kItemBlock = 128;   // a warp per item
template <typename T> constexpr int ring_node_block() { return sizeof(T) == 4 ? 64 : 32; }

template <typename T, int W> __global__ void __launch_bounds__(kItemBlock) k_ring_cols(DevPlan<T> P) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int warp = threadIdx.x >> 5, item = blockIdx.x * (kItemBlock / 32) + warp;
    if (item < P.rg_nitem) ring_cols_warp<T, W>(P, item, smraw + warp * RingStage<T, W>::bytes, threadIdx.x & 31);
}

template <typename T, int W> __global__ void __launch_bounds__(kItemBlock) k_ring_inv(DevPlan<T> P) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int warp = threadIdx.x >> 5, item = blockIdx.x * (kItemBlock / 32) + warp;
    if (item < P.rg_nitem) ring_inv_warp<T, W>(P, item, smraw + warp * RingStage<T, W>::bytes, threadIdx.x & 31);
}

template <typename T> __global__ void __launch_bounds__(256) k_ring_gather(DevPlan<T> P) {
    __shared__ cpx<T> tile[32][33];
    __shared__ RingGatherSmem S;
    ring_gather_block<T>(P, blockIdx.x, 32 * blockIdx.y, tile, S);
}

template <typename T, int W, int DIM>
__global__ void __launch_bounds__(ring_node_block<T>()) k_ring_nodes(DevPlan<T> P, int first, RingClass cl) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int warp = threadIdx.x >> 5, arc = first + blockIdx.x * (ring_node_block<T>() / 32) + warp;
    if (arc < cl.end) ring_node_warp<W, DIM>(P, arc, smraw + warp * ring_node_smem<T, W>(cl), cl, threadIdx.x & 31);
}

// calls fn(std::integral_constant<int, w>) for the widths the ring kernels are built for
template <typename T, class Fn> static bool ring_width_switch(int w, Fn &&fn) {
#define NLP_W(X) case X: fn(std::integral_constant<int, X>{}); return true;
    if constexpr (sizeof(T) == 4) {
        switch (w) { NLP_W(4) NLP_W(5) NLP_W(6) NLP_W(7) NLP_W(8) NLP_W(9) NLP_W(10) }
    } else {
        switch (w) { NLP_W(8) NLP_W(9) NLP_W(10) NLP_W(11) NLP_W(12) NLP_W(13) NLP_W(14) NLP_W(15) }
    }
#undef NLP_W
    return false;
}

template <typename T> size_t ring_smem(const DevPlan<T> &P, int warps) {
    size_t b = 0;
    ring_width_switch<T>(P.w, [&](auto w) {
        b = warps * RingStage<T, decltype(w)::value>::bytes;
        for (const RingClass &c : P.rg_cls) b = std::max(b, warps * ring_node_smem<T, decltype(w)::value>(c));
    });
    return b;
}

template <typename T> int ring_xy_stride(int w) {
    int r = 0;
    ring_width_switch<T>(w, [&](auto c) { r = RingGeo<T, decltype(c)::value>::XY; });
    return r;
}

template <typename T> int ring_psi_stride(int w) {
    int r = 0;
    ring_width_switch<T>(w, [&](auto c) { r = RingGeo<T, decltype(c)::value>::PS; });
    return r;
}

template <typename T> cudaError_t launch_ring_cols(const DevPlan<T> &P, cudaStream_t st) {
    cudaError_t e = cudaErrorInvalidValue;
    if (P.rg_nitem == 0) return cudaSuccess;
    ring_width_switch<T>(P.w, [&](auto w) {
        constexpr int W = decltype(w)::value, per = kItemBlock / 32;
        k_ring_cols<T, W><<<(P.rg_nitem + per - 1) / per, kItemBlock, per * RingStage<T, W>::bytes, st>>>(P);
        e = cudaGetLastError();
    });
    return e;
}

template <typename T, int W, int DIM> static cudaError_t ring_nodes(const DevPlan<T> &P, cudaStream_t st) {
    constexpr int per = ring_node_block<T>() / 32;
    cudaError_t e = allow_smem<k_ring_nodes<T, W, DIM>>();
    int first = 0;
    for (const RingClass &c : P.rg_cls) {
        if (e == cudaSuccess && c.end > first) {
            k_ring_nodes<T, W, DIM><<<(c.end - first + per - 1) / per, ring_node_block<T>(),
                                      per * ring_node_smem<T, W>(c), st>>>(P, first, c);
            e = cudaGetLastError();
        }
        first = c.end;
    }
    return e;
}
template <typename T> cudaError_t launch_ring_nodes(const DevPlan<T> &P, cudaStream_t st) {
    cudaError_t e = cudaErrorInvalidValue;
    ring_width_switch<T>(P.w, [&](auto w) {
        constexpr int W = decltype(w)::value;
        if (P.ring == 3) e = ring_nodes<T, W, 3>(P, st);
        else if constexpr (ring_2d<T>(W)) e = ring_nodes<T, W, 2>(P, st);
    });
    return e;
}

template <typename T> cudaError_t launch_ring_inv(const DevPlan<T> &P, cudaStream_t st) {
    cudaError_t e = cudaErrorInvalidValue;
    if (P.rg_nitem == 0) return cudaSuccess;
    ring_width_switch<T>(P.w, [&](auto w) {
        constexpr int W = decltype(w)::value, per = kItemBlock / 32;
        k_ring_inv<T, W><<<(P.rg_nitem + per - 1) / per, kItemBlock, per * RingStage<T, W>::bytes, st>>>(P);
        e = cudaGetLastError();
    });
    return e;
}

template <typename T> __global__ void __launch_bounds__(256) k_ring_gather2(DevPlan<T> P) {
    __shared__ cpx<T> part[8][32];
    ring_gather2_block<T>(P, blockIdx.x, part);
}
template <typename T> cudaError_t launch_ring_gather2(const DevPlan<T> &P, cudaStream_t st) {
    if (P.rg_npat == 0) return cudaSuccess;
    k_ring_gather2<T><<<P.rg_npat, 256, 0, st>>>(P);
    return cudaGetLastError();
}

template <typename T> cudaError_t launch_ring_gather(const DevPlan<T> &P, cudaStream_t st) {
    if (P.rg_npat == 0 || P.rg_zlen == 0) return cudaSuccess;
    k_ring_gather<T><<<dim3(P.rg_npat, (P.rg_zlen + 31) / 32), 256, 0, st>>>(P);
    return cudaGetLastError();
}

}  // namespace nlp
