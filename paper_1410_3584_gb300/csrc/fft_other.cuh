// Compile-time kernels for the other lengths 48 ... 360 that upsampled grids of even 2-3-5 sizes
// have (plain passes; the fused ones take the run-time engine there).  Radices and threads a line
// as line_threads says.  Against the run-time engine (16 threads a line, up to 10 of them idle in a pass,
// radix dispatched at run time), us a pass at 16 and at 2000 blocks: FP32 C2R 60 6.3 / 6.3, 23 / 15;
// 240 11 / 11, 63 / 51; 300 15 / 10, 123 / 78; 360 17 / 11, 146 / 94; FP64 R2C 60 11.9 / 10.4, 78 / 72;
// 120 19 / 15, 162 / 119; 200 27 / 23, 283 / 242; 300 39 / 35, 426 / 416 (240 C2R 271 / 275, the one of
// these that is not faster).
#pragma once
#include "fft_launch.cuh"

namespace nlp {
template <typename T> struct OtherLens {
    template <class Fn> static bool with(int N, Fn &&fn) {
        switch (N) {
            case 48: fn(Radices<4, 12>{}); return true;
            case 60: fn(Pick<T, Radices<5, 4, 3>, Radices<6, 10>>{}); return true;
            case 72: fn(Pick<T, Radices<6, 4, 3>, Radices<6, 12>>{}); return true;
            case 80: fn(Pick<T, Radices<4, 5, 4>, Radices<8, 10>>{}); return true;
            case 100: fn(Pick<T, Radices<5, 4, 5>, Radices<10, 10>>{}); return true;
            case 108: fn(Radices<6, 3, 6>{}); return true;
            case 120: fn(Pick<T, Radices<12, 10>, Radices<10, 12>>{}); return true;
            case 144: fn(Radices<12, 12>{}); return true;
            case 180: fn(Pick<T, Radices<12, 5, 3>, Radices<5, 6, 6>>{}); return true;
            case 200: fn(Pick<T, Radices<10, 4, 5>, Radices<10, 20>>{}); return true;
            case 216: fn(Radices<6, 6, 6>{}); return true;
            case 240: fn(Pick<T, Radices<12, 4, 5>, Radices<12, 20>>{}); return true;
            case 288: fn(Radices<6, 8, 6>{}); return true;
            case 300: fn(Radices<5, 6, 10>{}); return true;
            case 324: fn(Radices<6, 3, 3, 6>{}); return true;
            case 360: fn(Pick<T, Radices<6, 10, 6>, Radices<12, 6, 5>>{}); return true;
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
