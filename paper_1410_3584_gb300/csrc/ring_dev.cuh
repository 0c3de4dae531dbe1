// Interpolation and spreading of the 3D node set by rings (device bodies, block index passed
// explicitly: the single-plan kernels of ring_launch.cuh and the batched persistent kernel run
// the same code).  rings.h builds the decomposition; with A_arc the strip of an arc,
//
//   columns -> strips   A_arc(x, y) = sum_i psi_z,i F(x, y, s + i)            (per ring: w taps)
//   nodes               c_j = omega_j sum_(x,y) psi_x psi_y A_arc(x, y),
//                       B_arc(x, y) = sum_j psi_x psi_y c_j  (over A_arc)     (per node: w^2 taps)
//   strips -> columns   G(x, y, z) = sum over arcs and images of psi_z,(z - s) B_arc(x, y).
//
// Operation count per node: w^2 taps, and w taps for each cell of its share of the strip (9.5
// cells at w = 7, 17 at w = 13 for the 144 x 144 x 240 nodes of a 128^3 grid), instead of w^3
// taps in each direction.  At 128^3, against one register-column kernel per 2^3 sub-tile of
// nodes (w^3 taps): FP64 65 -> 9.5 ms (FP64 FMA bound: 26 FMAs a cell and direction, 70% of the
// lanes of a patch on a strip), FP32 0.57 -> 0.43 ms (issue slots and shared-memory wavefronts:
// the node stage takes 0.22 of it).
//
// 2D plans (polar nodes, half turns) run the node stage with strips read from the spectrum and a gather
// of the strips into G: at 640 x 768 FP64 972 + 74 + 14 us (one warp per node on tile windows, window
// sum, combine) -> 239 + 20 with arcs of 128 nodes (an evaluation 579 us; 554 with arcs of 32), at
// 1024^2 FP32 53 + 12 + 8 -> 24 + 14.
//
// A warp owns a patch of 8 x 4 columns and marches along z through the patch's arcs in the
// order of their first tap, holding the w values of each column around it in registers, so F is
// read and G written once and the arcs' strips are read and written in 8-cell runs.  Every sum
// has one owner and a fixed order: results are bit-identical from run to run.
#pragma once
#include "common.cuh"
#include "es_dev.cuh"

namespace nlp {

// node footprint along x (rings.h): FP32 the even-aligned window (16-byte pairs), FP64 the taps
template <typename T, int W> struct RingGeo {
    static constexpr bool kPad = sizeof(T) == 4;
    static constexpr int WX = kPad ? 2 * ((W + 2) / 2) : W;   // footprint edge along x
    static constexpr int WP = kPad ? 2 * ((W + 1) / 2) : W;   // last-axis taps (FP32: in pairs)
    // kernel-value row: the w values, zeros, and the first tap in the last slot
    static constexpr int PS = kPad ? 4 * ((W + 4) / 4) : 2 * ((W + 2) / 2);
    static constexpr int NE = kPad ? 32 : 16;                 // entries staged together
    static constexpr int XY = kPad ? 4 * ((WX + W + 3) / 4) : 2 * W;   // a node's row of the table rg_xy
    // FP32 spreading: staged psi_y (a zero after the w rows) and psi_x of a node, in strides that the
    // lanes' 8-byte stores reach without bank conflicts
    static constexpr int WR = (W + 1) | 1, SX = WX + 2;
};

// a kernel-value row from shared memory (16-byte loads), without its first tap
template <typename T, int W> struct RingRow {
    static constexpr int PS = RingGeo<T, W>::PS;
    T v[PS];
    __device__ __forceinline__ void load(const T *p) {
        if constexpr (sizeof(T) == 4) {
#pragma unroll
            for (int i = 0; i < PS / 4; ++i) {
                const float4 q = reinterpret_cast<const float4 *>(p)[i];
                v[4 * i] = q.x;
                v[4 * i + 1] = q.y;
                v[4 * i + 2] = q.z;
                v[4 * i + 3] = q.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < PS / 2; ++i) {
                const double2 q = reinterpret_cast<const double2 *>(p)[i];
                v[2 * i] = q.x;
                v[2 * i + 1] = q.y;
            }
        }
        v[PS - 1] = (T)0;   // (the padding of the last pair where w + 1 = PS)
    }
};

// The w values of one column around the march position, FP32 as pairs along z (packed FMAs).
template <typename T, int W> struct RingCol;
template <int W> struct RingCol<float, W> {
    static constexpr int NP = RingGeo<float, W>::WP / 2;
    float2 re[NP], im[NP];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < NP; ++i) re[i] = im[i] = make_float2(0.f, 0.f);
    }
    // drop the lowest plane, take v as the highest tap
    __device__ __forceinline__ void shift(float vx, float vy) {
#pragma unroll
        for (int i = 0; i + 1 < NP; ++i) {
            re[i] = make_float2(re[i].y, re[i + 1].x);
            im[i] = make_float2(im[i].y, im[i + 1].x);
        }
        re[NP - 1] = W % 2 ? make_float2(vx, 0.f) : make_float2(re[NP - 1].y, vx);
        im[NP - 1] = W % 2 ? make_float2(vy, 0.f) : make_float2(im[NP - 1].y, vy);
    }
    __device__ __forceinline__ cpx<float> low() const { return mk<float>(re[0].x, im[0].x); }
    __device__ __forceinline__ cpx<float> at(int i) const {
        cpx<float> v = mk<float>(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < W; ++k)
            if (k == i) v = (k & 1) ? mk<float>(re[k / 2].y, im[k / 2].y) : mk<float>(re[k / 2].x, im[k / 2].x);
        return v;
    }
    __device__ __forceinline__ cpx<float> dot(const float *psi) const {
        float2 sx = make_float2(0.f, 0.f), sy = sx;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const float2 p = make_float2(psi[2 * i], psi[2 * i + 1]);
            sx = __ffma2_rn(re[i], p, sx);
            sy = __ffma2_rn(im[i], p, sy);
        }
        return mk<float>(sx.x + sx.y, sy.x + sy.y);
    }
    __device__ __forceinline__ void axpy(const float *psi, cpx<float> b) {
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const float2 p = make_float2(psi[2 * i], psi[2 * i + 1]);
            re[i] = __ffma2_rn(make_float2(b.x, b.x), p, re[i]);
            im[i] = __ffma2_rn(make_float2(b.y, b.y), p, im[i]);
        }
    }
};
template <int W> struct RingCol<double, W> {
    double re[W], im[W];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < W; ++i) re[i] = im[i] = 0.0;
    }
    __device__ __forceinline__ void shift(double vx, double vy) {
#pragma unroll
        for (int i = 0; i + 1 < W; ++i) {
            re[i] = re[i + 1];
            im[i] = im[i + 1];
        }
        re[W - 1] = vx;
        im[W - 1] = vy;
    }
    __device__ __forceinline__ cpx<double> low() const { return mk<double>(re[0], im[0]); }
    __device__ __forceinline__ cpx<double> at(int i) const {
        cpx<double> v = mk<double>(0.0, 0.0);
#pragma unroll
        for (int k = 0; k < W; ++k)
            if (k == i) v = mk<double>(re[k], im[k]);
        return v;
    }
    __device__ __forceinline__ cpx<double> dot(const double *psi) const {
        double sx = 0.0, sy = 0.0;
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const double p = psi[i];
            sx = fma(re[i], p, sx);
            sy = fma(im[i], p, sy);
        }
        return mk<double>(sx, sy);
    }
    __device__ __forceinline__ void axpy(const double *psi, cpx<double> b) {
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const double p = psi[i];
            re[i] = fma(b.x, p, re[i]);
            im[i] = fma(b.y, p, im[i]);
        }
    }
};

// fine-grid column (wrapped) of a lane of patch p
struct RingLane {
    int x, y;
    bool ok;
};
template <typename T> __device__ __forceinline__ RingLane ring_lane(const DevPlan<T> &P, int patch, int lane) {
    const int py_n = (P.nf[1] + 3) / 4;
    const int px = patch / py_n, py = patch - px * py_n;
    RingLane r;
    r.x = px * 8 + (lane & 7);
    r.y = py * 4 + (lane >> 3);
    r.ok = r.x < P.nf[0] && r.y < P.nf[1];
    return r;
}

// The entries of an item and their kernel-value rows, staged NE at a time in a warp's shared
// memory by asynchronous copies: while batch k is worked on, the rows of batch k + 1 (whose
// entries have arrived) and the entries of batch k + 2 are in flight.
__device__ __forceinline__ void ring_cp16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void ring_cp8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void ring_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void ring_cp_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

template <typename T, int W> struct RingStage {
    static constexpr int NE = RingGeo<T, W>::NE, PS = RingGeo<T, W>::PS;
    static constexpr size_t bytes = 3 * NE * sizeof(RingEnt) + 2 * NE * PS * sizeof(T);   // a warp
    T *psi;           // [2][NE][PS]
    uint32_t *ent;    // [3][NE][6]
    const DevPlan<T> &P;
    int e0, n, lane;
    __device__ __forceinline__ RingStage(const DevPlan<T> &P_, unsigned char *sm, int e0_, int n_, int lane_)
        : psi((T *)sm), ent((uint32_t *)(sm + 2 * NE * PS * sizeof(T))), P(P_), e0(e0_), n(n_), lane(lane_) {}
    __device__ __forceinline__ void issue_ent(int k) {
        const int c = 3 * min(NE, n - k * NE);   // 8-byte pieces
        uint32_t *dst = ent + (k % 3) * (NE * 6);
        const uint32_t *src = P.rg_ent + 6 * (int64_t)(e0 + k * NE);
        for (int i = lane; i < c; i += 32) ring_cp8(dst + 2 * i, src + 2 * i);
    }
    __device__ __forceinline__ void issue_psi(int k) {
        constexpr int Q = PS * (int)sizeof(T) / 16;   // 16-byte pieces of a row
        const int c = Q * min(NE, n - k * NE);
        const uint32_t *e = ent + (k % 3) * (NE * 6);
        T *dst = psi + (k & 1) * (NE * PS);
        for (int i = lane; i < c; i += 32) {
            const int u = i / Q, q = i - u * Q;
            const T *row = P.rg_psi + (int64_t)(e[6 * u + 1] & kEntRow) * PS;
            ring_cp16(dst + u * PS + q * (16 / (int)sizeof(T)), row + q * (16 / (int)sizeof(T)));
        }
    }
    __device__ __forceinline__ void start() {
        __syncwarp();   // the buffers may have been read before (several items a warp)
        issue_ent(0);
        if (n > NE) issue_ent(1);
        ring_cp_commit();
        ring_cp_wait();
        __syncwarp();
        issue_psi(0);
        ring_cp_commit();
    }
    // first tap of the lane's entry of batch k, and the entries where it changes (entry 0 among them)
    __device__ __forceinline__ uint32_t runs(int k, int &s) const {
        const int m = min(NE, n - k * NE);
        s = 0;
        if (lane < m) {
            const T v = psi[(k & 1) * (NE * PS) + lane * PS + PS - 1];
            if constexpr (sizeof(T) == 4) s = __float_as_int(v);
            else s = __double2loint(v);
        }
        const int before = __shfl_up_sync(0xffffffffu, s, 1);
        return __ballot_sync(0xffffffffu, lane < m && (lane == 0 || s != before));
    }
    // batch k becomes readable, the next copies start
    __device__ __forceinline__ void next(int k) {
        ring_cp_wait();
        __syncwarp();
        if ((k + 1) * NE < n) issue_psi(k + 1);
        if ((k + 2) * NE < n) issue_ent(k + 2);
        ring_cp_commit();
    }
};

// ------------------------------------------------------------------ columns -> strips
// One warp per item.  The window moves when the first tap does, its next plane loaded one step
// ahead.
template <typename T, int W>
__device__ __forceinline__ void ring_cols_warp(const DevPlan<T> &P, int item, unsigned char *sm, int lane) {
    constexpr int NE = RingGeo<T, W>::NE, PS = RingGeo<T, W>::PS;
    const RingItem I = P.rg_item[item];
    RingStage<T, W> S(P, sm, I.e0, I.e1 - I.e0, lane);
    S.start();
    const RingLane ln = ring_lane(P, I.patch, lane);
    const int N0 = P.nf[0], N1 = P.nf[1], N2 = P.nf[2];
    const int x = ln.ok ? ln.x : 0, y = ln.ok ? ln.y : 0;
    const cpx<T> *fd = P.F + ((int64_t)x * N1 + y) * P.nh;
    const cpx<T> *fm = P.F + ((int64_t)(x ? N0 - x : 0) * N1 + (y ? N1 - y : 0)) * P.nh;
    auto load = [&](int z) -> cpx<T> {   // F on the whole z axis (Hermitian half stored)
        if ((unsigned)z < (unsigned)P.nh) return fd[z];
        int l = z % N2;
        if (l < 0) l += N2;
        return 2 * l <= N2 ? fd[l] : conj(fm[N2 - l]);
    };
    RingCol<T, W> col;
    col.zero();
    int cur = INT32_MIN / 2;
    cpx<T> nxt = mk<T>(0, 0);
    cpx<T> *out = P.rg_strip + (lane & 7);
    const int row = 2 + (lane >> 3);
    for (int k = 0; k * NE < S.n; ++k) {
        S.next(k);
        const uint32_t *E = S.ent + (k % 3) * (NE * 6);
        const T *R = S.psi + (k & 1) * (NE * PS);
        int s;
        uint32_t runs = S.runs(k, s);   // entries whose first tap differs from the one before
        while (runs) {
            const int i0 = __ffs(runs) - 1;
            runs &= runs - 1;
            const int i1 = runs ? __ffs(runs) - 1 : min(NE, S.n - k * NE);
            const int to = __shfl_sync(0xffffffffu, s, i0);
            if (to - cur >= W) {
                cur = to - W;
                nxt = load(cur + W);
            }
            while (cur < to) {
                col.shift(nxt.x, nxt.y);
                ++cur;
                nxt = load(cur + W);
            }
#pragma unroll 4
            for (int i = i0; i < i1; ++i) {
                const uint2 h = *reinterpret_cast<const uint2 *>(E + 6 * i);
                const int off = (int)E[6 * i + row];
                RingRow<T, W> pz;
                pz.load(R + i * PS);
                const cpx<T> v = col.dot(pz.v);
                if (((h.x >> lane) & 1u) && !(h.y & kEntSpread)) out[off] = v;
            }
        }
    }
}

// ------------------------------------------------------------------ strips -> columns
// One warp per item: the transpose of the march above.  Planes that the march has passed are
// final for the item and go to its scratch planes (32 columns each); the strip values of the
// next 8 entries load while 8 are worked on.
template <typename T, int W>
__device__ __forceinline__ void ring_inv_warp(const DevPlan<T> &P, int item, unsigned char *sm, int lane) {
    constexpr int NE = RingGeo<T, W>::NE, PS = RingGeo<T, W>::PS, NB = sizeof(T) == 4 ? 8 : 4;
    const RingItem I = P.rg_item[item];
    RingStage<T, W> S(P, sm, I.e0, I.e1 - I.e0, lane);
    S.start();
    RingCol<T, W> col;
    col.zero();
    const int row = 2 + (lane >> 3), lx = lane & 7, nz = I.z1 - I.z0;
    cpx<T> *out = P.rg_scr + (int64_t)I.plane0 * 32 + lane;
    int cur = 0;
    auto emit = [&](cpx<T> v) {
        const int z = cur - I.z0;
        if ((unsigned)z < (unsigned)nz) out[z * 32] = v;
    };
    // strip values of entries [i0, i0 + NB) (NB divides NE: one batch), signs: their conjugations
    auto fetch = [&](int i0, cpx<T> (&b)[NB], uint32_t &mir) {
        const uint32_t *E = S.ent + ((i0 / NE) % 3) * (NE * 6) + (i0 % NE) * 6;
        mir = 0;
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            b[u] = mk<T>(0, 0);
            if (i0 + u < S.n) {
                const uint2 h = *reinterpret_cast<const uint2 *>(E + 6 * u);
                const int off = (int)E[6 * u + row];
                const bool m = (h.y & kEntMirror) != 0;
                mir |= m ? 1u << u : 0u;
                if ((h.x >> lane) & 1u) b[u] = P.rg_strip[m ? off - lx : off + lx];
            }
        }
    };
    cpx<T> bn[NB];
    uint32_t mn;
    fetch(0, bn, mn);
    for (int k = 0; k * NE < S.n; ++k) {
        S.next(k);
        int s;
        const uint32_t runs = S.runs(k, s);
        if (k == 0) cur = __shfl_sync(0xffffffffu, s, 0);
        const int m = min(NE, S.n - k * NE);
        for (int g = 0; g < m; g += NB) {
            cpx<T> b[NB];
            const uint32_t mb = mn;
#pragma unroll
            for (int u = 0; u < NB; ++u) b[u] = bn[u];
            if (k * NE + g + NB < S.n) fetch(k * NE + g + NB, bn, mn);   // (the next batch's entries have arrived)
            const T *R = S.psi + (k & 1) * (NE * PS) + g * PS;
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                if (g + u >= m) break;
                if ((runs >> (g + u)) & 1u) {
                    const int to = __shfl_sync(0xffffffffu, s, g + u);
                    for (int steps = 0; cur < to && steps < W; ++steps) {
                        emit(col.low());
                        col.shift((T)0, (T)0);
                        ++cur;
                    }
                    while (cur < to) {   // a gap wider than the window
                        emit(mk<T>(0, 0));
                        ++cur;
                    }
                }
                RingRow<T, W> pz;
                pz.load(R + u * PS);
                if ((mb >> u) & 1u) b[u].y = -b[u].y;
                col.axpy(pz.v, b[u]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < W; ++i) {
        emit(col.low());
        col.shift((T)0, (T)0);
        ++cur;
    }
}

// One block (256 threads) per patch and 32 planes: the items' planes added in item order (a
// warp holds four planes of the 32 columns, the loads of NI items in flight), written to G
// contiguous along z.
struct RingGatherSmem {
    int z0[64], z1[64], plane0[64];
};
template <typename T>
__device__ __forceinline__ void ring_gather_block(const DevPlan<T> &P, int pat, int zc, cpx<T> (*tile)[33], RingGatherSmem &S) {
    constexpr int NI = sizeof(T) == 4 ? 4 : 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int patch = P.rg_pat[3 * pat], i0 = P.rg_pat[3 * pat + 1], i1 = P.rg_pat[3 * pat + 2];
    const int zw = zc + 4 * warp;
    cpx<T> v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = mk<T>(0, 0);
    for (int ib = i0; ib < i1; ib += 64) {
        const int ni = min(64, i1 - ib);
        __syncthreads();
        for (int i = threadIdx.x; i < ni; i += blockDim.x) {
            const RingItem I = P.rg_item[ib + i];
            S.z0[i] = I.z0;
            S.z1[i] = I.z1;
            S.plane0[i] = I.plane0;
        }
        __syncthreads();
        // items ascend in z0 and in z1: those that meet the warp's planes are consecutive
        int a = 0, b = 0;
        for (int i = lane; i < ni; i += 32) {
            a += S.z1[i] <= zw;
            b += S.z0[i] < zw + 4;
        }
        a = __reduce_add_sync(0xffffffffu, a);
        b = __reduce_add_sync(0xffffffffu, b);
        for (int i = a; i < b; i += NI) {
            cpx<T> t[NI][4];
#pragma unroll
            for (int k = 0; k < NI; ++k) {
                const int q = min(i + k, b - 1);
                const int z0 = S.z0[q], z1 = i + k < b ? S.z1[q] : 0;
                const cpx<T> *src = P.rg_scr + ((int64_t)S.plane0[q] + (zw - z0)) * 32 + lane;
#pragma unroll
                for (int u = 0; u < 4; ++u) t[k][u] = (zw + u >= z0 && zw + u < z1) ? src[u * 32] : mk<T>(0, 0);
            }
#pragma unroll
            for (int k = 0; k < NI; ++k)
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = v[u] + t[k][u];
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) tile[4 * warp + u][lane] = v[u];
    __syncthreads();
    const int m = min(32, P.rg_zlen - zc);
    for (int c = warp; c < 32; c += 8) {
        const RingLane r = ring_lane(P, patch, c);
        if (r.ok && lane < m) P.G[((int64_t)r.x * P.nf[1] + r.y) * P.nh + zc + lane] = tile[lane][c];
    }
}

// ------------------------------------------------------------------ nodes
// One warp per arc, its strip in shared memory: the interpolation takes one node per lane (w^2
// taps from shared memory), then the strip is cleared and the spreading takes one node at a
// time with the lanes over its footprint, and the strip goes back to where it came from.
//
// In the spreading the footprint's cells belong to lanes by their position modulo the
// footprint: a lane keeps its cells in registers and exchanges only those that leave the
// footprint as it moves along the arc (a few per step) with the strip, whose cells no other lane
// ever touches.
constexpr int kRingStage = 32;   // FP32: nodes staged together by the spreading
constexpr int kRingBatch = 8;    // FP64

// shared memory of a warp for strips of c.cells cells and c.rows rows, arcs of c.nodes nodes
template <typename T, int W> __host__ __device__ inline size_t ring_node_smem(const RingClass &c) {
    size_t b = (size_t)c.cells * sizeof(cpx<T>) + (size_t)c.nodes * sizeof(cpx<T>);
    if (sizeof(T) == 4) b += kRingStage * (RingGeo<T, W>::SX * sizeof(float) + RingGeo<T, W>::WR * sizeof(float2) + sizeof(int));
    else b += (size_t)kRingBatch * 3 * W * sizeof(double) + kRingBatch * sizeof(int);
    b += (size_t)c.rows * sizeof(int);
    return (b + 15) / 16 * 16;
}

template <typename T> __device__ __forceinline__ void ring_strip_load(const DevPlan<T> &P, const RingArc &A, cpx<T> *sm, int lane) {
    const float4 *src = reinterpret_cast<const float4 *>(P.rg_strip + A.cell0);
    const int n16 = (int)(((size_t)A.ncell * sizeof(cpx<T>) + 15) / 16);
    for (int i = lane; i < n16; i += 32) ring_cp16(reinterpret_cast<float4 *>(sm) + i, src + i);
    ring_cp_commit();
}

// 2D: the strip straight from the forward spectrum, by the plan's index of every cell (bit 31: the
// conjugate, where a row leaves the stored half).
template <typename T>
__device__ __forceinline__ void ring_strip_spectrum(const DevPlan<T> &P, const RingArc &A, cpx<T> *sm, int lane) {
#pragma unroll 4
    for (int i = lane; i < A.ncell; i += 32) {
        const uint32_t s = P.rg_src[A.cell0 + i];
        const cpx<T> v = P.F[s & 0x7fffffffu];
        sm[i] = s >> 31 ? conj(v) : v;
    }
}

// c_j from the interpolated spectrum: times omega_j, or for 2D Poisson W(k_j) of Algorithm 1 in FP64
// (omega_j holds (2 pi)^-2 w_r w_phi / |k|)
template <typename T> __device__ __forceinline__ cpx<T> ring_node_value(const DevPlan<T> &P, int64_t j, cpx<T> f, T om) {
    if (P.pois == nullptr) return scale(f, om);
    const double kx = P.pois[3 * j], ky = P.pois[3 * j + 1], kr = P.pois[3 * j + 2];
    const double g = exp(-0.5 * P.sigma * P.sigma * kr * kr);
    const double re = P.hvol * (double)f.x - P.mom[0] * g;
    const double im = P.hvol * (double)f.y + (kx * P.mom[1] + ky * P.mom[2]) * g;
    return mk<T>((T)((double)om * re), (T)((double)om * im));
}

// FP32: the kernel values of a node are evaluated in registers (3D, in both halves) or read from the
// plan's FP64-evaluated table (2D); a lane owns pairs of adjacent cells.
template <int W, int DIM = 3>
__device__ __forceinline__ void ring_node_warp(const DevPlan<float> &P, int arc, unsigned char *sm, const RingClass &cl, int lane) {
    constexpr int WX = RingGeo<float, W>::WX, NP = WX / 2;
    constexpr int RPI = 32 / NP, NIT = (W + RPI - 1) / RPI, NR = RPI * NIT;   // row slots: NR >= W
    constexpr int WR = RingGeo<float, W>::WR, SX = RingGeo<float, W>::SX;
    const RingArc A = P.rg_arc[arc];
    cpx<float> *strip = (cpx<float> *)sm;
    float2 *cb = (float2 *)(strip + cl.cells);
    float2 *scw = cb + cl.nodes;                       // [stage][WR]: c psi_y, zero in the rows past w
    float *swx = (float *)(scw + kRingStage * WR);     // [stage][SX]: psi_x
    int *sbase = (int *)(swx + kRingStage * SX);       // [stage]: footprint origin
    int *srow = (int *)(sbase + kRingStage);
    if constexpr (DIM == 3) ring_strip_load(P, A, strip, lane);
    else ring_strip_spectrum(P, A, strip, lane);
    for (int r = lane; r < A.nrow; r += 32) srow[r] = P.rg_rows[A.row0 + r];
    const float c2w = 2.0f / (float)W, nbl2 = -P.beta * 1.44269504f;
    const float4 *rec = reinterpret_cast<const float4 *>(P.rg_node);
    auto values_x = [&](float d, float2 (&v)[NP]) {   // kernel values of the footprint's WX cells
#pragma unroll
        for (int i = 0; i < NP; ++i) v[i] = es_fast2(f2(2.0f * i, 2.0f * i + 1.0f), f2(d, d), c2w, nbl2);
    };
    auto values_y = [&](float d, float (&v)[W]) {     // and of its W rows
#pragma unroll
        for (int i = 0; i + 1 < W; i += 2) {
            const float2 e = es_fast2(f2((float)i, (float)(i + 1)), f2(d, d), c2w, nbl2);
            v[i] = e.x;
            v[i + 1] = e.y;
        }
        if (W % 2) v[W - 1] = es_fast((float)(W - 1), d, c2w, nbl2);
    };
    // node j: kernel values, weight, packed footprint origin
    auto node = [&](int j, float2 (&wx)[NP], float (&wy)[W], float &om, int &base) {
        if constexpr (DIM == 3) {
            const float4 nd = rec[j];
            values_x(nd.x, wx);
            values_y(nd.y, wy);
            om = nd.z;
            base = __float_as_int(nd.w);
        } else {
            constexpr int XY = RingGeo<float, W>::XY;
            float v[XY];
#pragma unroll
            for (int i = 0; i < XY / 4; ++i) {
                const float4 q = reinterpret_cast<const float4 *>(P.rg_xy + (int64_t)j * XY)[i];
                v[4 * i] = q.x;
                v[4 * i + 1] = q.y;
                v[4 * i + 2] = q.z;
                v[4 * i + 3] = q.w;
            }
#pragma unroll
            for (int i = 0; i < NP; ++i) wx[i] = f2(v[2 * i], v[2 * i + 1]);
#pragma unroll
            for (int i = 0; i < W; ++i) wy[i] = v[WX + i];
            om = P.rg_om[j];
            base = P.rg_pos[j];
        }
    };
    ring_cp_wait();
    __syncwarp();
    for (int j = A.j0 + lane; j < A.j1; j += 32) {
        float2 wx[NP];
        float wy[W], om;
        int base;
        node(j, wx, wy, om, base);
        const int xa = base & 0xffff, ya = base >> 16;
        float2 acc = f2(0.f, 0.f);
#pragma unroll
        for (int r = 0; r < W; ++r) {
            const float4 *p = reinterpret_cast<const float4 *>(strip + srow[ya + r] + xa);
            float2 s = f2(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const float4 f = p[i];
                s = __ffma2_rn(f2(f.x, f.y), f2(wx[i].x, wx[i].x), s);
                s = __ffma2_rn(f2(f.z, f.w), f2(wx[i].y, wx[i].y), s);
            }
            acc = __ffma2_rn(s, f2(wy[r], wy[r]), acc);
        }
        const cpx<float> c = ring_node_value<float>(P, j, mk<float>(acc.x, acc.y), om);
        cb[j - A.j0] = f2(c.x, c.y);
    }
    __syncwarp();
    for (int i = lane; i < A.ncell / 2; i += 32) reinterpret_cast<float4 *>(strip)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp();
    const int row = min(lane / NP, RPI - 1), pr = lane % NP;
    const bool lane_ok = lane < NP * RPI;   // (the lanes past it work on a copy that they never store)
    int at[NIT], dy[NIT], dx = 0, cur = -1;   // cells held, and their place in the footprint
    float4 g[NIT];
#pragma unroll
    for (int k = 0; k < NIT; ++k) {
        at[k] = -1;
        dy[k] = W;
        g[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int jb = A.j0; jb < A.j1; jb += kRingStage) {
        const int nb = min(kRingStage, A.j1 - jb);
        __syncwarp();
        if (lane < nb) {
            const float2 c = cb[jb + lane - A.j0];
            float2 wx[NP];
            float wy[W], om;
            int base;
            node(jb + lane, wx, wy, om, base);
            float2 *wr = reinterpret_cast<float2 *>(swx + lane * SX);
#pragma unroll
            for (int i = 0; i < NP; ++i) wr[i] = wx[i];
#pragma unroll
            for (int i = 0; i < W; ++i) scw[lane * WR + i] = f2(c.x * wy[i], c.y * wy[i]);
            scw[lane * WR + W] = f2(0.f, 0.f);
            sbase[lane] = base;
        }
        __syncwarp();
        const float2 *pw = scw;
        const float *px = swx;
        for (int q = 0; q < nb; ++q, pw += WR, px += SX) {
            const int base = sbase[q];
            if (base != cur) {
                cur = base;
                const int xa = cur & 0xffff, ya = cur >> 16;
                dx = pr - (xa / 2) % NP;
                dx = 2 * (dx + (dx < 0 ? NP : 0));
#pragma unroll
                for (int k = 0; k < NIT; ++k) {
                    dy[k] = row + k * RPI - ya % NR;
                    dy[k] = min(dy[k] + (dy[k] < 0 ? NR : 0), W);
                    if (dy[k] < W) {
                        const int to = srow[ya + dy[k]] + xa + dx;
                        if (to != at[k]) {
                            if (at[k] >= 0 && lane_ok) *reinterpret_cast<float4 *>(strip + at[k]) = g[k];
                            g[k] = *reinterpret_cast<const float4 *>(strip + to);
                            at[k] = to;
                        }
                    }
                }
            }
            const float2 wx = *reinterpret_cast<const float2 *>(px + dx);
#pragma unroll
            for (int k = 0; k < NIT; ++k) {
                const float2 cw = pw[dy[k]];   // zero weights for a cell outside the footprint
                g[k].x = fmaf(cw.x, wx.x, g[k].x);
                g[k].y = fmaf(cw.y, wx.x, g[k].y);
                g[k].z = fmaf(cw.x, wx.y, g[k].z);
                g[k].w = fmaf(cw.y, wx.y, g[k].w);
            }
        }
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < NIT; ++k)
        if (at[k] >= 0 && lane_ok) *reinterpret_cast<float4 *>(strip + at[k]) = g[k];
    __syncwarp();
    float4 *dst = reinterpret_cast<float4 *>(P.rg_strip + A.cell0);
    for (int i = lane; i < A.ncell / 2; i += 32) dst[i] = reinterpret_cast<const float4 *>(strip)[i];
}

// FP64 (bound by the FP64 FMA rate, 2 per clock and SM): kernel values from the plan's table
// [node][psi_x w, psi_y w]; in the spreading the w^2 cells of the footprint are dealt flat over
// the lanes, with c psi_x formed once per node, so a node costs ceil(w^2 / 32) + 1 FMA pairs a lane.
template <int W, int DIM = 3>
__device__ __forceinline__ void ring_node_warp(const DevPlan<double> &P, int arc, unsigned char *sm, const RingClass &cl, int lane) {
    constexpr int NB = kRingBatch, NIT = (W * W + 31) / 32;
    const RingArc A = P.rg_arc[arc];
    cpx<double> *strip = (cpx<double> *)sm;
    cpx<double> *cb = strip + cl.cells;
    cpx<double> *scx = cb + cl.nodes;              // [NB][W]: c psi_x
    double *swy = (double *)(scx + NB * W);        // [NB][W]
    int *sbase = (int *)(swy + NB * W);            // [NB]
    int *srow = sbase + NB;
    if constexpr (DIM == 3) ring_strip_load(P, A, strip, lane);
    else ring_strip_spectrum(P, A, strip, lane);
    for (int r = lane; r < A.nrow; r += 32) srow[r] = P.rg_rows[A.row0 + r];
    ring_cp_wait();
    __syncwarp();
    for (int j = A.j0 + lane; j < A.j1; j += 32) {
        const double *tab = P.rg_xy + (int64_t)j * (2 * W);
        const int base = P.rg_pos[j], xa = base & 0xffff, ya = base >> 16;
        double wx[W];
#pragma unroll
        for (int i = 0; i < W; ++i) wx[i] = tab[i];
        double ax = 0.0, ay = 0.0;
#pragma unroll 1
        for (int r = 0; r < W; ++r) {
            const cpx<double> *p = strip + srow[ya + r] + xa;
            double sx = 0.0, sy = 0.0;
#pragma unroll
            for (int i = 0; i < W; ++i) {
                const cpx<double> f = p[i];
                sx = fma(f.x, wx[i], sx);
                sy = fma(f.y, wx[i], sy);
            }
            const double wr = tab[W + r];
            ax = fma(sx, wr, ax);
            ay = fma(sy, wr, ay);
        }
        cb[j - A.j0] = ring_node_value<double>(P, j, mk<double>(ax, ay), P.rg_om[j]);
    }
    __syncwarp();
    for (int i = lane; i < A.ncell; i += 32) strip[i] = mk<double>(0.0, 0.0);
    // the lane's cells by slot t = lane + 32 k: row slot t / W, column slot t mod W (both modulo W)
    int at[NIT], sd[NIT], cur = -1;   // cells held; their footprint row and column (x | y << 8)
    cpx<double> g[NIT];
#pragma unroll
    for (int k = 0; k < NIT; ++k) {
        at[k] = -1;
        sd[k] = 0;
        g[k] = mk<double>(0.0, 0.0);
    }
    for (int jb = A.j0; jb < A.j1; jb += NB) {
        const int nb = min(NB, A.j1 - jb);
        __syncwarp();
        for (int t = lane; t < nb * W; t += 32) {
            const int k = t / W, i = t - k * W;
            const double *tab = P.rg_xy + (int64_t)(jb + k) * (2 * W);
            const cpx<double> c = cb[jb + k - A.j0];
            const double wx = tab[i];
            scx[t] = mk<double>(c.x * wx, c.y * wx);
            swy[t] = tab[W + i];
        }
        if (lane < nb) sbase[lane] = P.rg_pos[jb + lane];
        __syncwarp();
        for (int q = 0; q < nb; ++q) {
            const int base = sbase[q];
            if (base != cur) {
                cur = base;
                const int xa = cur & 0xffff, ya = cur >> 16, xm = xa % W, ym = ya % W;
#pragma unroll
                for (int k = 0; k < NIT; ++k) {
                    const int t = lane + 32 * k;
                    int dy = t / W - ym, dx = t % W - xm;
                    dy += dy < 0 ? W : 0;
                    dx += dx < 0 ? W : 0;
                    sd[k] = dx | dy << 8;
                    if (t < W * W) {
                        const int to = srow[ya + dy] + xa + dx;
                        if (to != at[k]) {
                            if (at[k] >= 0) strip[at[k]] = g[k];
                            g[k] = strip[to];
                            at[k] = to;
                        }
                    } else {
                        sd[k] = 0;
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < NIT; ++k) {
                const cpx<double> cx = scx[q * W + (sd[k] & 0xff)];
                const double wy = swy[q * W + (sd[k] >> 8)];
                g[k].x = fma(cx.x, wy, g[k].x);
                g[k].y = fma(cx.y, wy, g[k].y);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < NIT; ++k)
        if (at[k] >= 0) strip[at[k]] = g[k];
    __syncwarp();
    cpx<double> *dst = P.rg_strip + A.cell0;
    for (int i = lane; i < A.ncell; i += 32) dst[i] = strip[i];
}

// 2D: strips -> G, one block per patch (x: the last axis, y: axis 1): the arcs and mirror images that
// reach it in equal runs over the warps, eight loads in flight, the warps' sums added in order.
// (One warp a patch was bound by the patch at k = 0, which every small ring reaches: 39 us at
// 1024^2 FP32, 14 with eight.)
template <typename T> __device__ __forceinline__ void ring_gather2_block(const DevPlan<T> &P, int pat, cpx<T> (*part)[32]) {
    constexpr int NB = 8;
    const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int patch = P.rg_pat[3 * pat], b0 = P.rg_pat[3 * pat + 1], n = P.rg_pat[3 * pat + 2] - b0;
    const int e0 = b0 + (int)((int64_t)n * warp / nw), e1 = b0 + (int)((int64_t)n * (warp + 1) / nw);
    const int lx = lane & 7, row = 2 + (lane >> 3);
    cpx<T> s = mk<T>(0, 0);
    for (int e = e0; e < e1; e += NB) {
        cpx<T> v[NB];
        uint32_t mir = 0;
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const uint32_t *E = P.rg_ent + 6 * (int64_t)min(e + u, e1 - 1);
            const uint2 h = *reinterpret_cast<const uint2 *>(E);
            const int off = (int)E[row];
            const bool m = (h.y & kEntMirror) != 0;
            mir |= m ? 1u << u : 0u;
            v[u] = e + u < e1 && ((h.x >> lane) & 1u) ? P.rg_strip[m ? off - lx : off + lx] : mk<T>(0, 0);
        }
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            if (e + u >= e1) break;   // (uniform: an FP64 addition of zeros costs as much as any)
            s.x += v[u].x;
            s.y += (mir >> u) & 1u ? -v[u].y : v[u].y;
        }
    }
    part[warp][lane] = s;
    __syncthreads();
    if (warp == 0) {
        for (int u = 1; u < nw; ++u) s = s + part[u][lane];
        const int PY = (P.nf[1] + kPatchY - 1) / kPatchY;
        const int x = patch / PY * kPatchX + lx, y = patch % PY * kPatchY + (lane >> 3);
        if (x < P.nh && y < P.nf[1]) P.G[(int64_t)y * P.nh + x] = s;
    }
}

}  // namespace nlp
