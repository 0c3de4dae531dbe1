// Learned initial guess for the normalized gradient flow of Sec. 3.1 (not part of the paper):
// a small network maps (beta, trap anisotropy gamma, kernel type) to a ground-state
// amplitude sampled on a 48^3 grid; the gradient flow started from it finishes the solve.
//
//   features : [log10(beta)/3, (gamma-1)/3, is Coulomb, is dipolar]        (padded to 64)
//   MLP      : 64 -> 512 -> 512 -> 512 -> 512, SiLU; dense layers as BF16 tcgen05 GEMMs with
//              FP32 accumulation (FP32 master weights, BF16 copies refreshed after updates)
//   head     : 512 -> 1728 (padded to 1792), linear, read as 8 channels x 6^3
//   decoder  : [nearest x2 -> 3^3 conv 8->8 -> SiLU] at 12^3 and 24^3, nearest x2 -> 3^3 conv
//              8->1 at 48^3 (zero padding)
//   loss     : mean squared error against the target amplitude; AdamW.
// Every forward and backward step is a kernel of this file; the decoder and elementwise
// work run on CUDA cores in FP32.  Mode 1 runs the dense layers on an FP32 CUDA-core GEMM
// instead (used to check the gradients against an FP64 host computation).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <random>
#include <vector>

#include "common.cuh"
#include "gemm_tc.cuh"
#include "launch.h"

namespace nlp {

constexpr int kFeat = 4, kFeatPad = 64, kHid = 512, kHeadOut = 8 * 216, kHeadPad = 1792;
constexpr int kC = 8;
constexpr int kGout = 48;
constexpr int64_t kOut = (int64_t)kGout * kGout * kGout;
constexpr int kBP = 128;   // padded batch = GEMM M of the forward layers
constexpr int kConv = 3;   // conv layers: (8->8 @ 12^3), (8->8 @ 24^3), (8->1 @ 48^3)
constexpr int kConvCi[kConv] = {kC, kC, kC}, kConvCo[kConv] = {kC, kC, 1}, kConvG[kConv] = {12, 24, 48};

// flat FP32 parameter vector: W_l [out][in] row-major then b_l, for l = 0..4; then for each
// conv layer w [co][ci][27] (tap d = 9 dz + 3 dy + dx, offsets -1..1) then bias [co]
struct Layout {
    size_t W[5], b[5], cw[kConv], cb[kConv], total;
    int nin[5], nout[5];
    Layout() {
        const int ins[5] = {kFeatPad, kHid, kHid, kHid, kHid}, outs[5] = {kHid, kHid, kHid, kHid, kHeadPad};
        size_t o = 0;
        for (int l = 0; l < 5; ++l) {
            nin[l] = ins[l];
            nout[l] = outs[l];
            W[l] = o;
            o += (size_t)ins[l] * outs[l];
            b[l] = o;
            o += outs[l];
        }
        for (int c = 0; c < kConv; ++c) {
            cw[c] = o;
            o += (size_t)kConvCo[c] * kConvCi[c] * 27;
            cb[c] = o;
            o += kConvCo[c];
        }
        total = o;
    }
};

#define GS(q, N) \
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < (int64_t)(N); q += (int64_t)gridDim.x * blockDim.x)

__device__ __forceinline__ float sig(float x) { return 1.f / (1.f + expf(-x)); }

// element q of a GEMM result that is still in S split-K parts of kBP x N, added in order (a sum
// kernel of its own cost 4 to 5 us a layer)
__device__ __forceinline__ float split_sum(const float *C, int S, int64_t q, int N) {
    float t = C[q];
#pragma unroll 8
    for (int z = 1; z < S; ++z) t += C[q + (int64_t)z * kBP * N];
    return t;
}

// Y = act(C + b) on rows < B (rows >= B stay zero), C in S parts; keeps the pre-activation; BF16
// copies of Y and of its transpose for the GEMMs that read it
__global__ void k_bias_act(const float *C, int S, const float *b, float *pre, float *Y, __nv_bfloat16 *Ybf,
                           __nv_bfloat16 *Ytbf, int B, int N, int act) {
    GS(q, (int64_t)kBP * N) {
        const int r = (int)(q / N), c = (int)(q % N);
        float v = 0.f, y = 0.f;
        if (r < B) {
            v = split_sum(C, S, q, N) + b[c];
            y = act ? v * sig(v) : v;
        }
        pre[q] = v;
        Y[q] = y;
        const __nv_bfloat16 yb = __float2bfloat16(y);
        if (Ybf) Ybf[q] = yb;
        if (Ytbf) Ytbf[(size_t)c * kBP + r] = yb;
    }
}

// dPre = dY * act'(pre) on rows < B, dY in S parts; BF16 copies of dPre and of its transpose
__global__ void k_act_back(const float *dY, int S, const float *pre, float *dP, __nv_bfloat16 *dPbf, __nv_bfloat16 *dPtbf,
                           int B, int N, int act) {
    GS(q, (int64_t)kBP * N) {
        const int r = (int)(q / N), c = (int)(q % N);
        float g = 0.f;
        if (r < B) {
            const float v = pre[q], s = sig(v), d = split_sum(dY, S, q, N);
            g = act ? d * (s * (1.f + v * (1.f - s))) : d;
        }
        dP[q] = g;
        const __nv_bfloat16 gb = __float2bfloat16(g);
        dPbf[q] = gb;
        dPtbf[(size_t)c * kBP + r] = gb;
    }
}

// db[c] = sum over rows of dP (fixed order): 32 columns a block, the rows in 8 runs of 16 side by
// side (128 rows in a chain per thread, on 2 blocks, took 7.3 us a layer; this 2.9 us)
__global__ void __launch_bounds__(256) k_colsum(const float *dP, float *db, int N) {
    __shared__ float sh[8][32];
    const int x = threadIdx.x & 31, u = threadIdx.x >> 5, c = blockIdx.x * 32 + x;
    float s = 0.f;
    if (c < N) {
#pragma unroll
        for (int r = 0; r < kBP / 8; ++r) s += dP[(size_t)(u * (kBP / 8) + r) * N + c];
    }
    sh[u][x] = s;
    __syncthreads();
    if (u == 0 && c < N) {
        for (int k = 1; k < 8; ++k) s += sh[k][x];
        db[c] = s;
    }
}

// BF16 copy and/or BF16 transpose and/or FP32 transpose of a row-major FP32 matrix [R x Cc]
__global__ void k_convert(const float *X, __nv_bfloat16 *Xb, __nv_bfloat16 *Xtb, float *Xt, int R, int Cc) {
    GS(q, (int64_t)R * Cc) {
        const int r = (int)(q / Cc), c = (int)(q % Cc);
        const float x = X[q];
        const __nv_bfloat16 v = __float2bfloat16(x);
        if (Xb) Xb[q] = v;
        if (Xtb) Xtb[(size_t)c * R + r] = v;
        if (Xt) Xt[(size_t)c * R + r] = x;
    }
}

// features [B x 4] -> padded input rows [kBP x 64] (FP32, BF16, BF16 transposed)
__global__ void k_input(const float *feat, int B, float *X, __nv_bfloat16 *Xbf, __nv_bfloat16 *Xtbf) {
    GS(q, (int64_t)kBP * kFeatPad) {
        const int r = (int)(q / kFeatPad), c = (int)(q % kFeatPad);
        const float v = (r < B && c < kFeat) ? feat[r * kFeat + c] : 0.f;
        X[q] = v;
        Xbf[q] = __float2bfloat16(v);
        Xtbf[(size_t)c * kBP + r] = __float2bfloat16(v);
    }
}

// head rows [kBP x 1792] -> z0 [B][1728]; and the reverse for the gradient (zeros elsewhere)
__global__ void k_head_unpack(const float *Y, float *z0, int B) {
    GS(q, (int64_t)B * kHeadOut) z0[q] = Y[(q / kHeadOut) * kHeadPad + q % kHeadOut];
}
__global__ void k_head_pack(const float *dz0, float *dY, int B) {
    GS(q, (int64_t)kBP * kHeadPad) {
        const int64_t r = q / kHeadPad, c = q % kHeadPad;
        dY[q] = (r < B && c < kHeadOut) ? dz0[r * kHeadOut + c] : 0.f;
    }
}

static dim3 grid_for(int64_t n) {
    return dim3((unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16)));
}

// ---- decoder layers: nearest x2, then a 3^3 convolution with zero padding 1, tap
// d = 9 dz + 3 dy + dx (offsets -1..1).  The upsampled grid (edge g) is never stored: every
// kernel below reads the coarse one (edge h = g / 2) or writes it.  At 64 samples the stored
// form moved 226 MB four times a pass at 48^3 and its halo staging took more instructions than
// the convolution itself.
//
// Forward and input gradient are bound by their 27 FP32 multiply-adds per channel pair and fine
// point (1.5 G at 24^3 and at 48^3: 41 us of the FP32 pipes).  A thread owns 2 x 2 fine points
// in x and y, kUpZ in z and CO_T channels: 32 sums in registers, so that the taps of a channel
// (27 CO_T registers) and each plane read from shared memory feed 864 multiply-adds, two an
// instruction (one each: 15 to 30 % slower).  What is left over the floor is the halo staging
// and its latency.  A block covers the full width, `nyp` pairs of rows and one z slab of one sample.
constexpr int kUpThreads = 128;   // at most, so that four blocks an SM have 128 registers a thread

template <int CO_T> constexpr int kUpZ = 8 / CO_T;   // fine z points of a thread

// a.x += w.x v, a.y += w.y v: both channels of a pair in one instruction, each rounded as fmaf
__device__ __forceinline__ void fma2(float2 &a, float2 w, float v) {
    asm("{\n .reg .b64 A, W, V;\n mov.b64 A, {%0, %1};\n mov.b64 W, {%2, %3};\n mov.b64 V, {%4, %4};\n"
        " fma.rn.f32x2 A, W, V, A;\n mov.b64 {%0, %1}, A;\n}\n"
        : "+f"(a.x), "+f"(a.y)
        : "f"(w.x), "f"(w.y), "f"(v));
}

// row pairs of a block: the largest divisor of h that fits
__host__ __device__ constexpr int up_pairs(int h, int groups) {
    int n = kUpThreads / (h * groups);
    while (h % n) --n;
    return n;
}

// pre[b][oc](p) = bias[oc] + sum_ic sum_d w[oc][ic][d] in[b][ic]((p + d - 1) >> 1), act = SiLU(pre)
// when given.  The input channels are summed in GRP groups whose sums are added in order.
// At 64 samples, upsampling and SiLU included: 8 -> 8 at 24^3 78 us (288 before), 8 -> 1 at
// 48^3 84 us (574 before).
template <int OC, int h>
__global__ void __launch_bounds__(kUpThreads, 4)
    k_up_conv(const float *__restrict__ in, const float *__restrict__ w, const float *__restrict__ bias,
              float *__restrict__ pre, float *__restrict__ act) {
    // eight output channels: pairs of channels, 4 z; one: pairs of y, 8 z, in groups of two inputs
    constexpr int CO_T = OC == 1 ? 1 : 2, GRP = OC == 1 ? 4 : 1;
    constexpr int Z = kUpZ<CO_T>, HZ = Z / 2 + 2;   // coarse planes a slab reaches
    constexpr int nyp = up_pairs(h, OC / CO_T), NT = h * nyp * (OC / CO_T);
    extern __shared__ float4 up_sm[];
    float *sw = (float *)up_sm;                     // [kC][OC / CO_T][28][CO_T] taps
    float *sh = sw + kC * OC * 28;                  // [kC][HZ][nyp + 2][h + 2]
    constexpr int g = 2 * h, HX = h + 2, HP = (nyp + 2) * HX, nty = h / nyp, ntz = g / Z;
    static_assert(h % nyp == 0 && g % Z == 0, "whole tiles");
    const int ty = blockIdx.x % nty, tz = (blockIdx.x / nty) % ntz, b = blockIdx.x / (nty * ntz);
    const int Y0 = ty * nyp - 1, Z0 = tz * (Z / 2) - 1;
    for (int i = threadIdx.x; i < kC * OC * 27; i += NT) {
        const int oc = i / (kC * 27), r = i - oc * (kC * 27), ic = r / 27, d = r - ic * 27;
        sw[(ic * OC + oc / CO_T * CO_T) * 28 + CO_T * d + oc % CO_T] = w[i];
    }
    const float *src = in + (int64_t)b * kC * h * h * h;
#pragma unroll 8
    for (int i = threadIdx.x; i < kC * HZ * HP; i += NT) {
        const int row = i / HX, x = i - row * HX - 1;
        const int pl = row / (nyp + 2), y = Y0 + row - pl * (nyp + 2);
        const int ic = pl / HZ, z = Z0 + pl - ic * HZ;
        float v = 0.f;
        if ((unsigned)z < (unsigned)h && (unsigned)y < (unsigned)h && (unsigned)x < (unsigned)h)
            v = src[((ic * h + z) * h + y) * h + x];
        sh[i] = v;
    }
    __syncthreads();
    const int xp = threadIdx.x % h, yp = (threadIdx.x / h) % nyp, oc0 = threadIdx.x / (h * nyp) * CO_T;
    float2 acc[16], tot[GRP > 1 ? 16 : 1];   // CO_T = 2: [z][y][x] of (channel 0, 1); 1: [z][x] of (y 0, 1)
#pragma unroll 1
    for (int gr = 0; gr < GRP; ++gr) {
        const float b0 = gr == 0 ? bias[oc0] : 0.f, b1 = CO_T == 2 ? bias[oc0 + CO_T - 1] : b0;
#pragma unroll
        for (int q = 0; q < 16; ++q) acc[q] = make_float2(b0, b1);
#pragma unroll 1
        for (int ic = gr * (kC / GRP); ic < (gr + 1) * (kC / GRP); ++ic) {
            float wt[28 * CO_T];
#pragma unroll
            for (int k = 0; k < 7 * CO_T; ++k) {
                const float4 f = *(const float4 *)(sw + (ic * OC + oc0) * 28 + 4 * k);
                wt[4 * k] = f.x, wt[4 * k + 1] = f.y, wt[4 * k + 2] = f.z, wt[4 * k + 3] = f.w;
            }
            const float *hb = sh + ic * HZ * HP + yp * HX + xp;
#pragma unroll
            for (int cz = 0; cz < HZ; ++cz) {
                float v[3][3];
#pragma unroll
                for (int e = 0; e < 9; ++e) v[e / 3][e % 3] = hb[cz * HP + (e / 3) * HX + e % 3];
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    const int hz = 2 * cz - 1 + f;   // fine plane, 0 = one below the slab
                    if (hz < 0 || hz > Z + 1) continue;
#pragma unroll
                    for (int dz = 0; dz < 3; ++dz) {
                        const int zo = hz - dz;
                        if (zo < 0 || zo >= Z) continue;
#pragma unroll
                        for (int k = 0; k < 9; ++k) {
                            const int d = dz * 9 + k, dy = k / 3, dx = k % 3;
                            if constexpr (CO_T == 2) {
#pragma unroll
                                for (int q = 0; q < 4; ++q)
                                    fma2(acc[zo * 4 + q], make_float2(wt[2 * d], wt[2 * d + 1]),
                                         v[((q >> 1) + dy + 1) >> 1][((q & 1) + dx + 1) >> 1]);
                            } else {
#pragma unroll
                                for (int q = 0; q < 2; ++q)
                                    fma2(acc[zo * 2 + q],
                                         make_float2(v[(dy + 1) >> 1][(q + dx + 1) >> 1],
                                                     v[(dy + 2) >> 1][(q + dx + 1) >> 1]), wt[d]);
                            }
                        }
                    }
                }
            }
        }
        if constexpr (GRP > 1) {
#pragma unroll
            for (int q = 0; q < 16; ++q)
                tot[q] = gr == 0 ? acc[q] : make_float2(tot[q].x + acc[q].x, tot[q].y + acc[q].y);
        }
    }
#pragma unroll
    for (int c = 0; c < CO_T; ++c)
#pragma unroll
        for (int q = 0; q < 2 * Z; ++q) {
            const int zo = q >> 1, yy = q & 1, z = tz * Z + zo, y = 2 * (ty * nyp + yp) + yy;
            float r[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float2 f = CO_T == 2 ? acc[CO_T == 2 ? zo * 4 + yy * 2 + u : 0] : tot[CO_T == 1 ? zo * 2 + u : 0];
                r[u] = (CO_T == 2 ? c : yy) ? f.y : f.x;
            }
            const int64_t o = (((int64_t)b * OC + oc0 + c) * g + z) * g * g + (int64_t)y * g + 2 * xp;
            *(float2 *)(pre + o) = make_float2(r[0], r[1]);
            if (act) *(float2 *)(act + o) = make_float2(r[0] * sig(r[0]), r[1] * sig(r[1]));
        }
}

// gradient with respect to the layer's coarse input, times SiLU'(pre) of the layer that made it
// (pre null: not): din[b][ci](P) = sum over the 8 fine points p of P of
// sum_co sum_d w[co][ci][26 - d] dout[b][co](p + d - 1).
// At 64 samples, with the sum over children and SiLU': 24^3 106 us (216 before), 48^3
// 100 us (282 before).
// With one output channel a thread takes the four channel pairs in turn, so that a block stages
// its plane once and has four times the work; with eight the pairs are side by side.
__host__ __device__ constexpr int back_groups(int Co) { return Co == 1 ? 1 : kC / 2; }

template <int Co, int h>
__global__ void __launch_bounds__(kUpThreads, 3)
    k_up_conv_back(const float *__restrict__ dout, const float *__restrict__ w, const float *__restrict__ pre,
                   float *__restrict__ din) {
    constexpr int Z = kUpZ<2>, HZ = Z + 2, GT = back_groups(Co), nyp = up_pairs(h, GT), NT = h * nyp * GT;
    extern __shared__ float4 up_sm[];
    float *sw = (float *)up_sm;        // [Co][kC / 2][28][2] flipped taps of channel pairs
    float *sh = sw + Co * kC * 28;     // [Co][HZ][2 nyp + 2][g + 2]
    constexpr int g = 2 * h, HX = g + 2, NY = 2 * nyp + 2, HP = NY * HX, nty = h / nyp, ntz = g / Z;
    static_assert(h % nyp == 0 && g % Z == 0, "whole tiles");
    const int ty = blockIdx.x % nty, tz = (blockIdx.x / nty) % ntz, b = blockIdx.x / (nty * ntz);
    const int y0 = 2 * ty * nyp - 1, z0 = tz * Z - 1;
    for (int i = threadIdx.x; i < Co * kC * 27; i += NT) {
        const int r = i / 27, d = i - r * 27;
        sw[(r >> 1) * 56 + 2 * d + (r & 1)] = w[r * 27 + 26 - d];
    }
    const float *src = dout + (int64_t)b * Co * g * g * g;
#pragma unroll 8
    for (int i = threadIdx.x; i < Co * HZ * HP; i += NT) {
        const int row = i / HX, x = i - row * HX - 1;
        const int pl = row / NY, y = y0 + row - pl * NY;
        const int co = pl / HZ, z = z0 + pl - co * HZ;
        float v = 0.f;
        if ((unsigned)z < (unsigned)g && (unsigned)y < (unsigned)g && (unsigned)x < (unsigned)g)
            v = src[((co * g + z) * g + y) * g + x];
        sh[i] = v;
    }
    __syncthreads();
    const int xp = threadIdx.x % h, yp = (threadIdx.x / h) % nyp, gq = threadIdx.x / (h * nyp);
    const int Y = ty * nyp + yp;
#pragma unroll 1
    for (int c0 = 2 * gq; c0 < kC; c0 += 2 * GT) {
        float2 acc[Z][2][2];
        float pv[Z];   // the SiLU arguments of the epilogue, on their way meanwhile
        const int64_t o0 = (((int64_t)b * kC + c0) * h + tz * (Z / 2)) * h * h + Y * h + xp;
#pragma unroll
        for (int q = 0; q < Z; ++q) pv[q] = pre ? pre[o0 + (q & 1) * h * h * h + (q >> 1) * h * h] : 0.f;
#pragma unroll
        for (int q = 0; q < 4 * Z; ++q) acc[q / 4][(q / 2) & 1][q & 1] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int co = 0; co < Co; ++co) {
            float2 wt[28];
#pragma unroll
            for (int k = 0; k < 14; ++k) {
                const float4 f = *(const float4 *)(sw + (co * kC + c0) * 28 + 4 * k);
                wt[2 * k] = make_float2(f.x, f.y), wt[2 * k + 1] = make_float2(f.z, f.w);
            }
            const float *hb = sh + co * HZ * HP + 2 * yp * HX + 2 * xp;
#pragma unroll
            for (int hz = 0; hz < HZ; ++hz) {
                float v[4][4];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float2 f = *(const float2 *)(hb + hz * HP + (e >> 1) * HX + 2 * (e & 1));
                    v[e >> 1][2 * (e & 1)] = f.x, v[e >> 1][2 * (e & 1) + 1] = f.y;
                }
#pragma unroll
                for (int dz = 0; dz < 3; ++dz) {
                    const int zo = hz - dz;
                    if (zo < 0 || zo >= Z) continue;
#pragma unroll
                    for (int k = 0; k < 9; ++k)
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            fma2(acc[zo][q >> 1][q & 1], wt[dz * 9 + k], v[(q >> 1) + k / 3][(q & 1) + k % 3]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < Z; ++q) {   // channel c0 + (q & 1), coarse plane q / 2 of the slab
            float s = 0.f;
#pragma unroll
            for (int d = 0; d < 8; ++d) {
                const float2 f = acc[(q & ~1) + (d >> 2)][(d >> 1) & 1][d & 1];
                s += q & 1 ? f.y : f.x;
            }
            if (pre) {
                const float v = pv[q], t = sig(v);
                s = s * (t * (1.f + v * (1.f - t)));
            }
            din[o0 + (q & 1) * h * h * h + (q >> 1) * h * h] = s;
        }
    }
}

template <int OC, int h>
static cudaError_t launch_up_conv(const float *in, const float *w, const float *bias, float *pre, float *act, int B,
                                  cudaStream_t st) {
    constexpr int ct = OC == 1 ? 1 : 2, z = kUpZ<ct>, nyp = up_pairs(h, OC / ct);
    constexpr size_t smem = sizeof(float) * (kC * OC * 28 + kC * (z / 2 + 2) * (nyp + 2) * (h + 2));
    static_assert(smem <= 48 * 1024, "fits without opting in");
    k_up_conv<OC, h><<<(unsigned)(B * (h / nyp) * (2 * h / z)), h * nyp * (OC / ct), smem, st>>>(
        in, w, bias, pre, act);
    return cudaGetLastError();
}

template <int Co, int h>
static cudaError_t launch_up_conv_back(const float *dout, const float *w, const float *pre, float *din, int B,
                                       cudaStream_t st) {
    constexpr int z = kUpZ<2>, gt = back_groups(Co), nyp = up_pairs(h, gt);
    constexpr size_t smem = sizeof(float) * (kC * Co * 28 + Co * (z + 2) * (2 * nyp + 2) * (2 * h + 2));
    static_assert(smem <= 48 * 1024, "fits without opting in");
    k_up_conv_back<Co, h><<<(unsigned)(B * (h / nyp) * (2 * h / z)), h * nyp * gt, smem, st>>>(dout, w, pre, din);
    return cudaGetLastError();
}

// ---- weight gradient: dw[co][ci][d] = sum_{b,p} dout[b][co](p) in[b][ci]((p + d - 1) >> 1),
// db[co] = sum_{b,p} dout[b][co](p).  A coarse point P meets tap d through the 8 fine points
// 2 P + c + 1 - d, c in {0,1}^3, so with the box sums S(q) = sum_c dout(q + c)
//   dw[co][ci][d] = sum_{b,P} in[b][ci](P) S[b][co](2 P + 1 - d),   db[co] = sum_{b,P} S(2 P):
// an eighth of the multiply-adds.  A block walks work items (sample, kWgY x kWgZ coarse rows of
// the full width) of one output channel in a fixed order: it forms the item's box sums in shared
// memory (columns along z, so that a plane's sum of four serves two boxes; even and odd x apart,
// so that neighbouring P read neighbouring words), then warp dz takes the points of tap plane dz
// with 8 x 9 sums in registers: 72 multiply-adds per 17 words read, and 128 registers a thread
// (half the channels a warp and twice the warps: 58 and 57 us instead of 56 and 48).  The sums
// of the lanes go to the block's slot part[co][block][8 x 27 + 1].  Bound by the latency of its
// loads (each item's box sums wait for dout).
// At 64 samples (with the fold over blocks): 24^3 55 us (330 before), 48^3 64 us (332).
constexpr int kWgY = 6, kWgZ = 2, kWgWarps = 3;
constexpr int kWgOut = kC * 27 + 1;     // a channel's sums: taps, then the bias
constexpr int kWgBlocks = 760;          // blocks of a launch, five an SM

template <int h>
__global__ void __launch_bounds__(32 * kWgWarps, 5)
    k_up_wgrad(const float *__restrict__ dout, const float *__restrict__ in, float *__restrict__ part, int B,
               int Co) {
    extern __shared__ float wg_sm[];
    constexpr int g = 2 * h, RP = g + 1, NR = 2 * kWgY + 1, HP = NR * RP, nty = h / kWgY, ntz = h / kWgZ;
    static_assert(h % kWgY == 0 && h % kWgZ == 0, "whole tiles");   // S: [2 kWgZ + 1][NR][RP]
    const int co = blockIdx.y, dz = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int npt = h * kWgY * kWgZ;
    const int items = B * nty * ntz;
    float acc[kC][9], accb = 0.f;
#pragma unroll
    for (int i = 0; i < kC * 9; ++i) acc[i / 9][i % 9] = 0.f;
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        const int ty = it % nty, tz = (it / nty) % ntz, b = it / (nty * ntz);
        const int y0 = 2 * ty * kWgY - 1, z0 = 2 * tz * kWgZ - 1;
        const float *src = dout + ((int64_t)b * Co + co) * g * g * g;
        __syncthreads();   // the previous item's sums are no longer read
        for (int i = threadIdx.x; i < HP; i += 32 * kWgWarps) {
            const int r = i / RP, xi = i - r * RP, x = xi - 1, y = y0 + r;
            const bool xa = x >= 0, xb = x + 1 < g, ya = y >= 0 && y < g, yb = y + 1 < g;
            float a[2 * kWgZ + 2];
#pragma unroll
            for (int k = 0; k < 2 * kWgZ + 2; ++k) {
                const int z = z0 + k;
                const bool zk = z >= 0 && z < g;
                const float *s = src + ((int64_t)z * g + y) * g + x;
                const float p0 = zk && ya && xa ? s[0] : 0.f, p1 = zk && ya && xb ? s[1] : 0.f;
                const float p2 = zk && yb && xa ? s[g] : 0.f, p3 = zk && yb && xb ? s[g + 1] : 0.f;
                a[k] = (p0 + p1) + (p2 + p3);
            }
            float *o = wg_sm + r * RP + ((xi & 1) ? h + 1 : 0) + (xi >> 1);
#pragma unroll
            for (int k = 0; k + 1 < 2 * kWgZ + 2; ++k) o[k * HP] = a[k] + a[k + 1];
        }
        __syncthreads();
        for (int p = lane; p < npt; p += 32) {
            const int row = p / h, X = p - row * h, yr = row % kWgY, zr = row / kWgY;
            const int Y = ty * kWgY + yr, Z = tz * kWgZ + zr;
            float f[kC], sv[9];
            const float *fi = in + (((int64_t)b * kC * h + Z) * h + Y) * h + X;
#pragma unroll
            for (int c = 0; c < kC; ++c) f[c] = fi[(int64_t)c * h * h * h];
            const float *bp = wg_sm + (2 * zr + 2 - dz) * HP + (2 * yr + 2) * RP + X;
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                sv[3 * dy] = bp[-dy * RP + 1];
                sv[3 * dy + 1] = bp[-dy * RP + h + 1];
                sv[3 * dy + 2] = bp[-dy * RP];
            }
            if (dz == 1) accb += sv[4];
#pragma unroll
            for (int c = 0; c < kC; ++c)
#pragma unroll
                for (int k = 0; k < 9; ++k) acc[c][k] = fmaf(f[c], sv[k], acc[c][k]);
        }
    }
    float *out = part + ((size_t)co * gridDim.x + blockIdx.x) * kWgOut;
#pragma unroll
    for (int i = 0; i < kC * 9 + 1; ++i) {
        float v = i < kC * 9 ? acc[(i / 9) % kC][i % 9] : accb;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0 && i < kC * 9) out[i / 9 * 27 + dz * 9 + i % 9] = v;
        if (lane == 0 && i == kC * 9 && dz == 1) out[kC * 27] = v;
    }
}

// the blocks' partials in a fixed order: one warp per weight
__global__ void k_up_wgrad_final(const float *part, int nblk, float *dw, float *db, int Co) {
    const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= Co * kWgOut) return;
    const int co = i / kWgOut, d = i - co * kWgOut;
    float t = 0.f;
    for (int u = lane; u < nblk; u += 32) t += part[((size_t)co * nblk + u) * kWgOut + d];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) {
        if (d < kC * 27) dw[co * kC * 27 + d] = t;
        else db[co] = t;
    }
}

template <int Co, int h>
static cudaError_t launch_up_wgrad(const float *dout, const float *in, float *part, float *dw, float *db, int B,
                                   cudaStream_t st) {
    const int nblk = std::min(kWgBlocks / Co, B * (h / kWgY) * (h / kWgZ));
    constexpr size_t sums = (size_t)(2 * kWgZ + 1) * (2 * kWgY + 1) * (2 * h + 1);
    constexpr size_t smem = sizeof(float) * sums;
    k_up_wgrad<h><<<dim3(nblk, Co), 32 * kWgWarps, smem, st>>>(dout, in, part, B, Co);
    k_up_wgrad_final<<<(Co * kWgOut + 7) / 8, 256, 0, st>>>(part, nblk, dw, db, Co);
    return cudaGetLastError();
}

// layer c of the decoder (kConvCo, kConvG)
static cudaError_t up_conv(int c, const float *in, const float *w, const float *bias, float *pre, float *act, int B,
                           cudaStream_t st) {
    auto f = c == 0 ? launch_up_conv<kConvCo[0], kConvG[0] / 2>
                    : c == 1 ? launch_up_conv<kConvCo[1], kConvG[1] / 2> : launch_up_conv<kConvCo[2], kConvG[2] / 2>;
    return f(in, w, bias, pre, act, B, st);
}
static cudaError_t up_conv_back(int c, const float *dout, const float *w, const float *pre, float *din, int B,
                                cudaStream_t st) {
    auto f = c == 0 ? launch_up_conv_back<kConvCo[0], kConvG[0] / 2>
                    : c == 1 ? launch_up_conv_back<kConvCo[1], kConvG[1] / 2>
                             : launch_up_conv_back<kConvCo[2], kConvG[2] / 2>;
    return f(dout, w, pre, din, B, st);
}
static cudaError_t up_wgrad(int c, const float *dout, const float *in, float *part, float *dw, float *db, int B,
                            cudaStream_t st) {
    auto f = c == 0 ? launch_up_wgrad<kConvCo[0], kConvG[0] / 2>
                    : c == 1 ? launch_up_wgrad<kConvCo[1], kConvG[1] / 2> : launch_up_wgrad<kConvCo[2], kConvG[2] / 2>;
    return f(dout, in, part, dw, db, B, st);
}

// squared-error partial sums per block and d out = 2 (out - t) / n
__global__ void k_mse(const float *out, const float *t, float *dout, int64_t n, double *part) {
    double s = 0.0;
    GS(q, n) {
        const float d = out[q] - t[q];
        s += (double)d * d;
        dout[q] = 2.f * d / (float)n;
    }
    __shared__ double sh[256];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// AdamW with bias-corrected moments and decoupled weight decay
__global__ void k_adamw(float *p, const float *g, float *m, float *v, int64_t n, float lr, float b1, float b2,
                        float eps, float wd, float c1, float c2) {
    GS(q, n) {
        const float gq = g[q];
        const float mq = b1 * m[q] + (1.f - b1) * gq;
        const float vq = b2 * v[q] + (1.f - b2) * gq * gq;
        m[q] = mq;
        v[q] = vq;
        p[q] -= lr * ((mq / c1) / (sqrtf(vq / c2) + eps) + wd * p[q]);
    }
}

// beta = 0 ground state of the trap V = (x^2 + y^2 + gamma^2 z^2)/2, normalised in the continuum:
// b(x) = gamma^{1/4} pi^{-3/4} exp(-(x^2 + y^2 + gamma z^2)/2).  The network learns the
// correction to it.
__device__ __forceinline__ double base_amp(double x, double y, double z, double gamma) {
    return pow(gamma, 0.25) * pow(M_PI, -0.75) * exp(-0.5 * (x * x + y * y + gamma * z * z));
}

// guess at the target grid points: b(x) + trilinear sample of the 48^3 network output (point j
// at -Ls + j hs; zero correction outside the sampled cube), clamped at zero
template <typename T>
__global__ void k_resample(const float *src, double Ls, double gamma, T *dst, int n0, int n1, int n2, double L0,
                           double L1, double L2) {
    const double hs = 2.0 * Ls / kGout;
    const int nn[3] = {n0, n1, n2};
    const double LL[3] = {L0, L1, L2};
    GS(q, (int64_t)n0 * n1 * n2) {
        const int64_t idx[3] = {q / ((int64_t)n1 * n2), (q / n2) % n1, q % n2};
        int lo[3];
        double f[3], x[3];
        bool inside = true;
        for (int a = 0; a < 3; ++a) {
            x[a] = -LL[a] + idx[a] * (2.0 * LL[a] / nn[a]);
            const double u = (x[a] + Ls) / hs;
            if (!(u >= 0.0 && u <= kGout - 1)) inside = false;
            lo[a] = min(max((int)floor(u), 0), kGout - 2);
            f[a] = u - lo[a];
        }
        double v = base_amp(x[0], x[1], x[2], gamma);
        if (inside) {
            for (int d = 0; d < 8; ++d) {
                const int dz = d >> 2, dy = (d >> 1) & 1, dx = d & 1;
                const double wgt = (dz ? f[0] : 1 - f[0]) * (dy ? f[1] : 1 - f[1]) * (dx ? f[2] : 1 - f[2]);
                v += wgt * src[((int64_t)(lo[0] + dz) * kGout + (lo[1] + dy)) * kGout + (lo[2] + dx)];
            }
        }
        dst[q] = (T)fmax(v, 0.0);
    }
}

// average over the 8 reflections x_a -> -x_a of the grid (index i -> (n - i) mod n on each axis),
// in place: one thread per orbit, representative indices 0..n/2 on every axis
template <typename T> __global__ void k_symmetrize(T *x, int n0, int n1, int n2) {
    const int h0 = n0 / 2 + 1, h1 = n1 / 2 + 1, h2 = n2 / 2 + 1;
    GS(q, (int64_t)h0 * h1 * h2) {
        const int i2 = (int)(q % h2), i1 = (int)((q / h2) % h1), i0 = (int)(q / ((int64_t)h1 * h2));
        const int a0[2] = {i0, (n0 - i0) % n0}, a1[2] = {i1, (n1 - i1) % n1}, a2[2] = {i2, (n2 - i2) % n2};
        double s = 0.0;
        for (int d = 0; d < 8; ++d)
            s += (double)x[((int64_t)a0[d >> 2] * n1 + a1[(d >> 1) & 1]) * n2 + a2[d & 1]];
        const T m = (T)(0.125 * s);
        for (int d = 0; d < 8; ++d) x[((int64_t)a0[d >> 2] * n1 + a1[(d >> 1) & 1]) * n2 + a2[d & 1]] = m;
    }
}

// FP64 partial sums of x^2 per block
template <typename T> __global__ void k_sumsq_part(const T *x, int64_t n, double *part) {
    double acc = 0.0;
    GS(q, n) {
        const double v = (double)x[q];
        acc += v * v;
    }
    __shared__ double sh[256];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// phi *= 1 / sqrt(hvol sum phi^2) (partials summed in order by every block)
template <typename T> __global__ void k_normalize(T *x, int64_t n, const double *part, int np, double hvol) {
    __shared__ double s;
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int i = 0; i < np; ++i) t += part[i];
        s = t > 0.0 ? 1.0 / sqrt(hvol * t) : 0.0;
    }
    __syncthreads();
    GS(q, n) x[q] = (T)((double)x[q] * s);
}

// the beta = 0 amplitude on the 48^3 cube (training targets are ground state minus this)
__global__ void k_base_cube(double Ls, const float *gamma, int B, float *out) {
    const double hs = 2.0 * Ls / kGout;
    GS(q, (int64_t)B * kOut) {
        const int64_t p = q % kOut;
        const int b = (int)(q / kOut);
        const int k = (int)(p % kGout), j = (int)((p / kGout) % kGout), i = (int)(p / ((int64_t)kGout * kGout));
        out[q] = (float)base_amp(-Ls + i * hs, -Ls + j * hs, -Ls + k * hs, (double)gamma[b]);
    }
}

constexpr int kRedBlocks = 512;
constexpr size_t kGemmWorkFloats = (size_t)16 * kBP * kHeadPad;   // split-K partials: 16 x 128 x 1792

}  // namespace nlp

using namespace nlp;

struct nlp_surrogate_s {
    Layout lay;
    cudaStream_t stream = nullptr;
    int mode = 0;          // 0: BF16 tensor-core GEMMs, 1: FP32 CUDA-core GEMMs
    double box_L = 10.0;   // output point j sits at -box_L + j * 2 box_L / 48 on each axis
    std::vector<void *> allocs;
    float *P = nullptr, *Gr = nullptr, *Mm = nullptr, *Vv = nullptr;   // params, grads, AdamW moments
    __nv_bfloat16 *Wbf[5] = {}, *Wtbf[5] = {};                         // W [out x in], W^T [in x out]
    float *Wt32[5] = {};                                               // W^T in FP32 (mode 1)
    float *X[6] = {}, *pre[5] = {}, *Cbuf = nullptr;                   // layer inputs/outputs [kBP x width]
    __nv_bfloat16 *Xbf[6] = {}, *Xtbf[6] = {};
    float *Xt32 = nullptr, *dPt32 = nullptr;                           // FP32 transposes (mode 1)
    float *dY = nullptr, *dP = nullptr;
    __nv_bfloat16 *dPbf = nullptr, *dPtbf = nullptr;
    // decoder: z0 -> [up -> conv -> (SiLU)] x 3; cpre[c] is conv c's output, cact[c] its SiLU
    float *z0 = nullptr, *cpre[kConv] = {}, *cact[kConv] = {};
    float *dz0 = nullptr, *dcpre[kConv] = {};
    float *wpart = nullptr, *dout = nullptr, *feat1 = nullptr;
    float *gemm_work = nullptr;   // split-K partials of the tensor-core GEMMs
    double *part = nullptr;
    int *err = nullptr;
    long long step = 0;
    // optional per-class kernel timers: an event after every launch, attributed to its class
    bool timing = false;
    static constexpr int kMaxEv = 160;
    cudaEvent_t ev[kMaxEv] = {};
    int ev_cls[kMaxEv] = {};
    int nev = 0;
    double cls_ms[NLP_SK_COUNT] = {};
    long long cls_n[NLP_SK_COUNT] = {};
};

// record the end of the launch just issued (class cls; -1 = the start mark)
static void mark(nlp_surrogate_s *s, int cls) {
    if (!s->timing || s->nev >= nlp_surrogate_s::kMaxEv) return;
    cudaEventRecord(s->ev[s->nev], s->stream);
    s->ev_cls[s->nev++] = cls;
}

// fold the recorded events into the per-class totals (waits for the last one)
static void collect(nlp_surrogate_s *s) {
    if (!s->timing || s->nev < 2) {
        s->nev = 0;
        return;
    }
    cudaEventSynchronize(s->ev[s->nev - 1]);
    for (int i = 1; i < s->nev; ++i) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, s->ev[i - 1], s->ev[i]) == cudaSuccess && s->ev_cls[i] >= 0) {
            s->cls_ms[s->ev_cls[i]] += ms;
            s->cls_n[s->ev_cls[i]]++;
        }
    }
    s->nev = 0;
}

static nlp_status sg_alloc(nlp_surrogate_s *s, void **p, size_t bytes) {
    if (cudaMalloc(p, bytes) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return NLP_ERR_OOM;
    }
    s->allocs.push_back(*p);
    return NLP_OK;
}

// split-K factor: the largest divisor of the K chunks that keeps the grid near 128 CTAs and the
// partials within `work_floats` (S = 1: no split)
static int gemm_splits(int M, int N, int K, size_t work_floats) {
    const int bn = N % 128 == 0 ? 128 : 64;
    const int tiles = (N / bn) * (M / 128), kch = K / 64;
    int best = 1;
    for (int S = 2; S <= kch; ++S)
        if (kch % S == 0 && tiles * S <= 128 && (size_t)S * M * N <= work_floats) best = S;
    return best;
}

// C = A B^T on the tensor cores; with S > 1 the K range is split over grid z, split z writing its
// partial product at C + z M N
static cudaError_t launch_gemm_tc(const __nv_bfloat16 *A, const __nv_bfloat16 *B, float *C, int M, int N, int K, int S,
                                  int *err, cudaStream_t st) {
    if (M % 128 || K % 64 || N % 64) return cudaErrorInvalidValue;
    cudaError_t e = allow_smem<k_gemm_bf16_tc<128>>();
    if (e == cudaSuccess) e = allow_smem<k_gemm_bf16_tc<64>>();
    if (e != cudaSuccess) return e;
    if (N % 128 == 0)
        k_gemm_bf16_tc<128><<<dim3(N / 128, M / 128, S), 128, kGemmSmemBytes, st>>>(A, B, C, M, N, K, K / S, err,
                                                                                    1ll << 22);
    else
        k_gemm_bf16_tc<64><<<dim3(N / 64, M / 128, S), 128, kGemmSmemBytes, st>>>(A, B, C, M, N, K, K / S, err,
                                                                                  1ll << 22);
    return cudaGetLastError();
}

// C[M x N] = A[M x K] B[N x K]^T, BF16 operands (mode 0) or FP32 operands (mode 1).  With `parts`
// the reader adds the product's *parts split-K parts, M N floats apart from *parts_at on; without,
// K is not split (the weight gradients: K = 128, two chunks, 4 to 56 tiles).
static nlp_status gemm(nlp_surrogate_s *s, const __nv_bfloat16 *A, const __nv_bfloat16 *B, const float *A32,
                       const float *B32, float *C, int M, int N, int K, const float **parts_at = nullptr,
                       int *parts = nullptr) {
    if (parts) *parts = 1, *parts_at = C;
    if (s->mode) {
        k_gemm_f32_simt<<<dim3((N + 15) / 16, (M + 15) / 16), 256, 0, s->stream>>>(A32, B32, C, M, N, K);
        mark(s, NLP_SK_GEMM);
        return cudaGetLastError() == cudaSuccess ? NLP_OK : NLP_ERR_CUDA;
    }
    const int S = parts ? gemm_splits(M, N, K, kGemmWorkFloats) : 1;
    if (S > 1) {
        C = s->gemm_work;
        *parts = S, *parts_at = C;
    }
    const bool ok = launch_gemm_tc(A, B, C, M, N, K, S, s->err, s->stream) == cudaSuccess;
    mark(s, NLP_SK_GEMM);
    return ok ? NLP_OK : NLP_ERR_CUDA;
}

static void refresh_weights(nlp_surrogate_s *s) {
    for (int l = 0; l < 5; ++l) {
        const int ni = s->lay.nin[l], no = s->lay.nout[l];
        k_convert<<<grid_for((int64_t)ni * no), 256, 0, s->stream>>>(s->P + s->lay.W[l], s->Wbf[l], s->Wtbf[l],
                                                                     s->mode ? s->Wt32[l] : nullptr, no, ni);
        mark(s, NLP_SK_ELEMENTWISE);
    }
}

static nlp_status forward(nlp_surrogate_s *s, const float *feat, int B) {
    cudaStream_t st = s->stream;
    const Layout &L = s->lay;
    nlp_status r;
    k_input<<<grid_for((int64_t)kBP * kFeatPad), 256, 0, st>>>(feat, B, s->X[0], s->Xbf[0], s->Xtbf[0]);
    mark(s, NLP_SK_ELEMENTWISE);
    for (int l = 0; l < 5; ++l) {
        const int ni = L.nin[l], no = L.nout[l];
        const float *Y;
        int S;
        if ((r = gemm(s, s->Xbf[l], s->Wbf[l], s->X[l], s->P + L.W[l], s->Cbuf, kBP, no, ni, &Y, &S))) return r;
        k_bias_act<<<grid_for((int64_t)kBP * no), 256, 0, st>>>(Y, S, s->P + L.b[l], s->pre[l], s->X[l + 1],
                                                                s->Xbf[l + 1], s->Xtbf[l + 1], B, no, l < 4);
        mark(s, NLP_SK_ELEMENTWISE);
    }
    k_head_unpack<<<grid_for((int64_t)B * kHeadOut), 256, 0, st>>>(s->X[5], s->z0, B);
    mark(s, NLP_SK_ELEMENTWISE);
    for (int c = 0; c < kConv; ++c) {
        if (up_conv(c, c ? s->cact[c - 1] : s->z0, s->P + L.cw[c], s->P + L.cb[c], s->cpre[c], s->cact[c], B, st) !=
            cudaSuccess)
            return NLP_ERR_CUDA;
        mark(s, NLP_SK_CONV_FWD);
    }
    return cudaGetLastError() == cudaSuccess ? NLP_OK : NLP_ERR_CUDA;
}

static nlp_status check_err(nlp_surrogate_s *s) {
    int h = 0;
    if (cudaMemcpyAsync(&h, s->err, sizeof(int), cudaMemcpyDeviceToHost, s->stream) != cudaSuccess ||
        cudaStreamSynchronize(s->stream) != cudaSuccess)
        return NLP_ERR_CUDA;
    return h ? NLP_ERR_TIMEOUT : NLP_OK;
}

// loss and every parameter gradient into s->Gr (flat layout)
static nlp_status backward(nlp_surrogate_s *s, const float *target, int B, double *loss) {
    cudaStream_t st = s->stream;
    const Layout &L = s->lay;
    const int64_t nout = (int64_t)B * kOut;
    k_mse<<<kRedBlocks, 256, 0, st>>>(s->cpre[kConv - 1], target, s->dout, nout, s->part);
    mark(s, NLP_SK_LOSS);
    const float *dnext = s->dout;   // gradient w.r.t. the current conv output (pre-activation)
    for (int c = kConv - 1; c >= 0; --c) {
        const float *cin = c ? s->cact[c - 1] : s->z0;
        float *din = c ? s->dcpre[c - 1] : s->dz0;
        if (up_wgrad(c, dnext, cin, s->wpart, s->Gr + L.cw[c], s->Gr + L.cb[c], B, st) != cudaSuccess)
            return NLP_ERR_CUDA;
        mark(s, NLP_SK_CONV_BWD_W);
        if (up_conv_back(c, dnext, s->P + L.cw[c], c ? s->cpre[c - 1] : nullptr, din, B, st) != cudaSuccess)
            return NLP_ERR_CUDA;
        mark(s, NLP_SK_CONV_BWD_IN);
        dnext = din;
    }
    k_head_pack<<<grid_for((int64_t)kBP * kHeadPad), 256, 0, st>>>(s->dz0, s->dY, B);
    mark(s, NLP_SK_ELEMENTWISE);
    nlp_status r;
    const float *dY = s->dY;
    int S = 1;
    for (int l = 4; l >= 0; --l) {
        const int ni = L.nin[l], no = L.nout[l];
        k_act_back<<<grid_for((int64_t)kBP * no), 256, 0, st>>>(dY, S, s->pre[l], s->dP, s->dPbf, s->dPtbf, B, no,
                                                                l < 4);
        mark(s, NLP_SK_ELEMENTWISE);
        k_colsum<<<(no + 31) / 32, 256, 0, st>>>(s->dP, s->Gr + L.b[l], no);
        mark(s, NLP_SK_ELEMENTWISE);
        // dW [no x ni] = dPre^T X : A = dPre^T [no x kBP], B = X^T [ni x kBP]
        if (s->mode) {
            k_convert<<<grid_for((int64_t)kBP * no), 256, 0, st>>>(s->dP, nullptr, nullptr, s->dPt32, kBP, no);
            k_convert<<<grid_for((int64_t)kBP * ni), 256, 0, st>>>(s->X[l], nullptr, nullptr, s->Xt32, kBP, ni);
            mark(s, NLP_SK_ELEMENTWISE);
        }
        if ((r = gemm(s, s->dPtbf, s->Xtbf[l], s->dPt32, s->Xt32, s->Gr + L.W[l], no, ni, kBP))) return r;
        // dX [kBP x ni] = dPre W : A = dPre [kBP x no], B = W^T [ni x no]; the next layer's dY
        if (l > 0 && (r = gemm(s, s->dPbf, s->Wtbf[l], s->dP, s->Wt32[l], s->dY, kBP, ni, no, &dY, &S))) return r;
    }
    if (cudaGetLastError() != cudaSuccess) return NLP_ERR_CUDA;
    if (loss) {
        double h[kRedBlocks];
        if (cudaMemcpyAsync(h, s->part, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess) return NLP_ERR_CUDA;
        if (cudaStreamSynchronize(st) != cudaSuccess) return NLP_ERR_CUDA;
        double t = 0;
        for (double x : h) t += x;
        *loss = t / (double)nout;
    }
    return NLP_OK;
}

extern "C" {

void nlp_surrogate_features(double beta, double gamma, nlp_kernel kernel, float *feat) {
    if (!feat) return;
    feat[0] = (float)(std::log10(beta > 0 ? beta : 1e-300) / 3.0);
    feat[1] = (float)((gamma - 1.0) / 3.0);
    feat[2] = kernel == NLP_COULOMB_3D ? 1.f : 0.f;
    feat[3] = kernel == NLP_DIPOLE_3D ? 1.f : 0.f;
}

void nlp_surrogate_destroy(nlp_surrogate s) {
    if (!s) return;
    cudaStreamSynchronize(s->stream);
    for (void *p : s->allocs) cudaFree(p);
    for (cudaEvent_t e : s->ev)
        if (e) cudaEventDestroy(e);
    delete s;
}

nlp_status nlp_surrogate_create(double box_L, unsigned long long seed, int mode, void *stream, nlp_surrogate *out) {
    if (!out) return NLP_ERR_INVALID_ARG;
    *out = nullptr;
    if (!(box_L > 0) || (mode != 0 && mode != 1)) return NLP_ERR_INVALID_ARG;
    nlp_surrogate_s *s = new (std::nothrow) nlp_surrogate_s();
    if (!s) return NLP_ERR_OOM;
    s->stream = (cudaStream_t)stream;
    s->mode = mode;
    s->box_L = box_L;
    const Layout &L = s->lay;
    nlp_status r = NLP_OK;
    auto A = [&](size_t bytes) -> void * {
        void *p = nullptr;
        if (r == NLP_OK) r = sg_alloc(s, &p, bytes);
        return p;
    };
    s->P = (float *)A(4 * L.total);
    s->Gr = (float *)A(4 * L.total);
    s->Mm = (float *)A(4 * L.total);
    s->Vv = (float *)A(4 * L.total);
    for (int l = 0; l < 5; ++l) {
        const size_t e = (size_t)L.nin[l] * L.nout[l];
        s->Wbf[l] = (__nv_bfloat16 *)A(2 * e);
        s->Wtbf[l] = (__nv_bfloat16 *)A(2 * e);
        s->Wt32[l] = (float *)A(4 * e);
    }
    const int widths[6] = {kFeatPad, kHid, kHid, kHid, kHid, kHeadPad};
    for (int l = 0; l < 6; ++l) {
        s->X[l] = (float *)A(4 * (size_t)kBP * widths[l]);
        s->Xbf[l] = (__nv_bfloat16 *)A(2 * (size_t)kBP * widths[l]);
        s->Xtbf[l] = (__nv_bfloat16 *)A(2 * (size_t)kBP * widths[l]);
        if (l < 5) s->pre[l] = (float *)A(4 * (size_t)kBP * widths[l + 1]);
    }
    const size_t wide = (size_t)kBP * kHeadPad;
    s->Cbuf = (float *)A(4 * wide);
    s->dY = (float *)A(4 * wide);
    s->dP = (float *)A(4 * wide);
    s->dPbf = (__nv_bfloat16 *)A(2 * wide);
    s->dPtbf = (__nv_bfloat16 *)A(2 * wide);
    s->Xt32 = (float *)A(4 * wide);
    s->dPt32 = (float *)A(4 * wide);
    s->z0 = (float *)A(4 * (size_t)kBP * kHeadOut);
    s->dz0 = (float *)A(4 * (size_t)kBP * kHeadOut);
    for (int c = 0; c < kConv; ++c) {
        const size_t G3 = (size_t)kConvG[c] * kConvG[c] * kConvG[c];
        s->cpre[c] = (float *)A(4 * kBP * kConvCo[c] * G3);
        if (c + 1 < kConv) {
            s->cact[c] = (float *)A(4 * kBP * kConvCo[c] * G3);
            s->dcpre[c] = (float *)A(4 * kBP * kConvCo[c] * G3);
        }
    }
    s->dout = (float *)A(4 * (size_t)kBP * kOut);
    s->wpart = (float *)A(4 * (size_t)kWgBlocks * kWgOut);
    s->gemm_work = (float *)A(4 * kGemmWorkFloats);
    s->feat1 = (float *)A(4 * kFeat);
    s->part = (double *)A(8 * kRedBlocks);
    s->err = (int *)A(sizeof(int));
    if (r) {
        nlp_surrogate_destroy(s);
        return r;
    }
    // initialisation: W ~ U(-1/sqrt(fan_in), 1/sqrt(fan_in)) over the real (unpadded) entries,
    // padding entries and biases zero
    std::vector<float> h(L.total, 0.f);
    std::mt19937_64 rng(seed);
    auto fill = [&](size_t off, int rows, int cols, int used_rows, int used_cols, double fan) {
        std::uniform_real_distribution<double> U(-1.0 / std::sqrt(fan), 1.0 / std::sqrt(fan));
        for (int i = 0; i < rows; ++i)
            for (int j = 0; j < cols; ++j)
                h[off + (size_t)i * cols + j] = (i < used_rows && j < used_cols) ? (float)U(rng) : 0.f;
    };
    fill(L.W[0], kHid, kFeatPad, kHid, kFeat, kFeat);
    for (int l = 1; l < 4; ++l) fill(L.W[l], kHid, kHid, kHid, kHid, kHid);
    fill(L.W[4], kHeadPad, kHid, kHeadOut, kHid, kHid);
    for (int c = 0; c < kConv; ++c)
        fill(L.cw[c], kConvCo[c] * kConvCi[c], 27, kConvCo[c] * kConvCi[c], 27, kConvCi[c] * 27.0);
    // everything on the network's stream (a stream created non-blocking does not order
    // against the legacy default stream)
    cudaStream_t st = s->stream;
    bool ok = cudaMemcpyAsync(s->P, h.data(), 4 * L.total, cudaMemcpyHostToDevice, st) == cudaSuccess &&
              cudaMemsetAsync(s->Mm, 0, 4 * L.total, st) == cudaSuccess &&
              cudaMemsetAsync(s->Vv, 0, 4 * L.total, st) == cudaSuccess &&
              cudaMemsetAsync(s->Gr, 0, 4 * L.total, st) == cudaSuccess &&
              cudaMemsetAsync(s->err, 0, sizeof(int), st) == cudaSuccess && cudaStreamSynchronize(st) == cudaSuccess;
    if (ok) {
        refresh_weights(s);
        ok = cudaStreamSynchronize(s->stream) == cudaSuccess;
    }
    if (!ok) {
        nlp_surrogate_destroy(s);
        return NLP_ERR_CUDA;
    }
    *out = s;
    return NLP_OK;
}

int64_t nlp_surrogate_num_params(nlp_surrogate s) { return s ? (int64_t)s->lay.total : 0; }

nlp_status nlp_surrogate_get_params(nlp_surrogate s, float *host) {
    if (!s || !host) return NLP_ERR_INVALID_ARG;
    if (cudaStreamSynchronize(s->stream) != cudaSuccess ||
        cudaMemcpy(host, s->P, 4 * s->lay.total, cudaMemcpyDeviceToHost) != cudaSuccess)
        return NLP_ERR_CUDA;
    return NLP_OK;
}

nlp_status nlp_surrogate_set_params(nlp_surrogate s, const float *host) {
    if (!s || !host) return NLP_ERR_INVALID_ARG;
    if (copy_in(s->P, host, 4 * s->lay.total, s->stream) != cudaSuccess) return NLP_ERR_CUDA;
    refresh_weights(s);
    return cudaStreamSynchronize(s->stream) == cudaSuccess ? NLP_OK : NLP_ERR_CUDA;
}

nlp_status nlp_surrogate_forward(nlp_surrogate s, const float *feat_dev, int B, float *out_dev) {
    if (!s || !feat_dev || !out_dev || B < 1 || B > kBP) return NLP_ERR_INVALID_ARG;
    nlp_status r = forward(s, feat_dev, B);
    if (r) return r;
    if (cudaMemcpyAsync(out_dev, s->cpre[kConv - 1], 4 * (size_t)B * kOut, cudaMemcpyDeviceToDevice, s->stream) !=
        cudaSuccess)
        return NLP_ERR_CUDA;
    return check_err(s);
}

nlp_status nlp_surrogate_gradients(nlp_surrogate s, const float *feat_dev, const float *target_dev, int B,
                                   double *loss, float *grads_host) {
    if (!s || !feat_dev || !target_dev || B < 1 || B > kBP) return NLP_ERR_INVALID_ARG;
    nlp_status r = forward(s, feat_dev, B);
    if (r || (r = backward(s, target_dev, B, loss)) || (r = check_err(s))) return r;
    if (grads_host && cudaMemcpy(grads_host, s->Gr, 4 * s->lay.total, cudaMemcpyDeviceToHost) != cudaSuccess)
        return NLP_ERR_CUDA;
    return NLP_OK;
}

nlp_status nlp_surrogate_train_step(nlp_surrogate s, const float *feat_dev, const float *target_dev, int B, float lr,
                                    float weight_decay, double *loss) {
    if (!s || !feat_dev || !target_dev || B < 1 || B > kBP || !(lr > 0) || !(weight_decay >= 0))
        return NLP_ERR_INVALID_ARG;
    s->nev = 0;   // drop marks of calls outside a training step
    mark(s, -1);
    nlp_status r = forward(s, feat_dev, B);
    if (r || (r = backward(s, target_dev, B, loss))) {
        s->nev = 0;
        return r;
    }
    s->step++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = (float)(1.0 - std::pow((double)b1, (double)s->step));
    const float c2 = (float)(1.0 - std::pow((double)b2, (double)s->step));
    k_adamw<<<grid_for((int64_t)s->lay.total), 256, 0, s->stream>>>(s->P, s->Gr, s->Mm, s->Vv, (int64_t)s->lay.total,
                                                                     lr, b1, b2, 1e-8f, weight_decay, c1, c2);
    mark(s, NLP_SK_ADAMW);
    refresh_weights(s);
    collect(s);
    if (cudaGetLastError() != cudaSuccess) return NLP_ERR_CUDA;
    return loss ? check_err(s) : NLP_OK;
}

nlp_status nlp_surrogate_initial_guess(nlp_surrogate s, double beta, double gamma, nlp_kernel kernel,
                                       const nlp_grid *grid, nlp_precision prec, void *phi_dev) {
    if (!s || !grid || !phi_dev || grid->dim != 3 || !(beta > 0) || !(gamma > 0) ||
        (kernel != NLP_COULOMB_3D && kernel != NLP_DIPOLE_3D) || (prec != NLP_FP64 && prec != NLP_FP32))
        return NLP_ERR_INVALID_ARG;
    for (int a = 0; a < 3; ++a)
        if (grid->n[a] < 2 || !(grid->L[a] > 0)) return NLP_ERR_INVALID_ARG;
    float f[kFeat];
    nlp_surrogate_features(beta, gamma, kernel, f);
    if (cudaMemcpyAsync(s->feat1, f, sizeof(f), cudaMemcpyHostToDevice, s->stream) != cudaSuccess ||
        cudaStreamSynchronize(s->stream) != cudaSuccess)
        return NLP_ERR_CUDA;
    nlp_status r = forward(s, s->feat1, 1);
    if (r) return r;
    const int n0 = grid->n[0], n1 = grid->n[1], n2 = grid->n[2];
    const int64_t N = (int64_t)n0 * n1 * n2, H = (int64_t)(n0 / 2 + 1) * (n1 / 2 + 1) * (n2 / 2 + 1);
    const double hvol = (2.0 * grid->L[0] / n0) * (2.0 * grid->L[1] / n1) * (2.0 * grid->L[2] / n2);
    const float *src = s->cpre[kConv - 1];
    cudaStream_t st = s->stream;
    if (prec == NLP_FP64) {
        double *phi = (double *)phi_dev;
        k_resample<double><<<grid_for(N), 256, 0, st>>>(src, s->box_L, gamma, phi, n0, n1, n2, grid->L[0], grid->L[1],
                                                        grid->L[2]);
        k_symmetrize<double><<<grid_for(H), 256, 0, st>>>(phi, n0, n1, n2);
        k_sumsq_part<double><<<kRedBlocks, 256, 0, st>>>(phi, N, s->part);
        k_normalize<double><<<grid_for(N), 256, 0, st>>>(phi, N, s->part, kRedBlocks, hvol);
    } else {
        float *phi = (float *)phi_dev;
        k_resample<float><<<grid_for(N), 256, 0, st>>>(src, s->box_L, gamma, phi, n0, n1, n2, grid->L[0], grid->L[1],
                                                       grid->L[2]);
        k_symmetrize<float><<<grid_for(H), 256, 0, st>>>(phi, n0, n1, n2);
        k_sumsq_part<float><<<kRedBlocks, 256, 0, st>>>(phi, N, s->part);
        k_normalize<float><<<grid_for(N), 256, 0, st>>>(phi, N, s->part, kRedBlocks, hvol);
    }
    if (cudaGetLastError() != cudaSuccess) return NLP_ERR_CUDA;
    return check_err(s);
}

nlp_status nlp_surrogate_base(nlp_surrogate s, const float *gamma_dev, int B, float *out_dev) {
    if (!s || !gamma_dev || !out_dev || B < 1) return NLP_ERR_INVALID_ARG;
    k_base_cube<<<grid_for((int64_t)B * kOut), 256, 0, s->stream>>>(s->box_L, gamma_dev, B, out_dev);
    return cudaGetLastError() == cudaSuccess ? NLP_OK : NLP_ERR_CUDA;
}

nlp_status nlp_surrogate_set_timing(nlp_surrogate s, int on) {
    if (!s) return NLP_ERR_INVALID_ARG;
    if (on && !s->ev[0])
        for (cudaEvent_t &e : s->ev)
            if (cudaEventCreate(&e) != cudaSuccess) return NLP_ERR_CUDA;
    s->timing = on != 0;
    s->nev = 0;
    for (int c = 0; c < NLP_SK_COUNT; ++c) {
        s->cls_ms[c] = 0.0;
        s->cls_n[c] = 0;
    }
    return NLP_OK;
}

nlp_status nlp_surrogate_get_kernel_times(nlp_surrogate s, double *ms, int64_t *launches) {
    if (!s || !ms) return NLP_ERR_INVALID_ARG;
    for (int c = 0; c < NLP_SK_COUNT; ++c) {
        ms[c] = s->cls_ms[c];
        if (launches) launches[c] = s->cls_n[c];
    }
    return NLP_OK;
}

nlp_status nlp_gemm_bf16(const void *A, const void *B, float *C, int M, int N, int K, void *stream) {
    if (!A || !B || !C || M <= 0 || N <= 0 || K <= 0 || M % 128 || K % 64 || N % 64) return NLP_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    int *err = nullptr;
    float *work = nullptr;
    const size_t wf = (size_t)16 * M * N;   // split-K partials, as the network's GEMMs use them
    if (cudaMalloc(&err, sizeof(int)) != cudaSuccess) return NLP_ERR_OOM;
    if (cudaMalloc(&work, sizeof(float) * wf) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(err);
        return NLP_ERR_OOM;
    }
    int h = 0;
    const int S = gemm_splits(M, N, K, wf);
    bool ok = cudaMemsetAsync(err, 0, sizeof(int), st) == cudaSuccess &&
              launch_gemm_tc((const __nv_bfloat16 *)A, (const __nv_bfloat16 *)B, S > 1 ? work : C, M, N, K, S, err,
                             st) == cudaSuccess;
    if (ok && S > 1) {
        const int64_t MN = (int64_t)M * N;
        k_splitk_sum<<<(unsigned)std::min<int64_t>((MN + 255) / 256, 1024), 256, 0, st>>>(work, S, MN, C);
        ok = cudaGetLastError() == cudaSuccess;
    }
    ok = ok && cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, st) == cudaSuccess &&
         cudaStreamSynchronize(st) == cudaSuccess;
    cudaFree(work);
    cudaFree(err);
    if (!ok) return NLP_ERR_CUDA;
    return h ? NLP_ERR_TIMEOUT : NLP_OK;
}

}  // extern "C"
