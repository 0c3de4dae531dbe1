// Compile-time kernels for the other lengths 48 ... 360 that upsampled grids of even 2-3-5 sizes
// have (plain passes; the fused ones take the run-time engine there).  Radices and threads a line
// by the rule of line_threads: a divisor of N / R for every pass, or nearly so where 2, 3 and 5 meet
// (60, 100, 120, 180, 200, 240, 300: up to a fifth of the lanes' turns idle).  FP64 takes enough
// threads to fill the warps of its 8 lines a block: 4 threads on 60 points and 5 on 100 took 116
// instead of 64 and 232 instead of 158 us for an evaluation at 30^3 and 50^3.  Against the run-time
// engine (16 threads a line, up to 10 of them idle in a pass, radix dispatched at run time), an
// evaluation with the precomputed kernel at n^3, us: FP32 n = 54 66 -> 46, 72 80 -> 54, 108 174 -> 113,
// 162 641 -> 390, no length below 1.05x; FP64 40 121 -> 86, 72 388 -> 284, 108 1090 -> 944, 150
// 3167 -> 3099 (the least).
#pragma once
#include "fft_launch.cuh"

namespace nlp {
template <typename T> struct OtherLens {
    template <class D, class S> using Pick = typename std::conditional<sizeof(T) == 8, D, S>::type;
    template <class Fn> static bool with(int N, Fn &&fn) {
        switch (N) {
            case 48: fn(Radices<4, 12>{}); return true;
            case 60: fn(Radices<5, 3, 4>{}); return true;
            case 72: fn(Pick<Radices<3, 8, 3>, Radices<6, 12>>{}); return true;
            case 80: fn(Pick<Radices<4, 5, 4>, Radices<4, 20>>{}); return true;
            case 100: fn(Pick<Radices<5, 4, 5>, Radices<5, 20>>{}); return true;
            case 108: fn(Radices<6, 3, 6>{}); return true;
            case 120: fn(Radices<5, 4, 6>{}); return true;
            case 144: fn(Radices<12, 12>{}); return true;
            case 180: fn(Radices<5, 6, 6>{}); return true;
            case 200: fn(Pick<Radices<5, 8, 5>, Radices<10, 20>>{}); return true;
            case 216: fn(Radices<6, 6, 6>{}); return true;
            case 240: fn(Pick<Radices<4, 12, 5>, Radices<12, 20>>{}); return true;
            case 288: fn(Radices<6, 8, 6>{}); return true;
            case 300: fn(Radices<5, 6, 10>{}); return true;
            case 324: fn(Radices<6, 3, 3, 6>{}); return true;
            case 360: fn(Radices<6, 10, 6>{}); return true;
        }
        return false;
    }
};
template <typename T> bool r2c_other(const T *rho, const DevPlan<T> &P, cudaStream_t st, cudaError_t &e) {
    return r2c_fixed<T, OtherLens<T>>(rho, P, st, e);
}
template <typename T> bool c2r_other(T *phi, const DevPlan<T> &P, cudaStream_t st, cudaError_t &e) {
    return c2r_fixed<T, OtherLens<T>>(phi, P, st, e);
}
template <typename T>
bool cols_other(cpx<T> *data, const StridedDesc &d, const FftLen<T> &L, int sign, cudaStream_t st, cudaError_t &e) {
    return cols_fixed<T, OtherLens<T>>(data, d, L, sign, st, e);
}
}  // namespace nlp
