// Register DFTs of the lengths 6, 9, 10, 15, 18, 25, 27, 30 and 32, beside those of
// pp_fft4.cuh: with them every even length up to 1024 with prime factors 2, 3 and
// 5 splits into two register factors (but 972 and 1000).
#pragma once
#include "pp_fft4.cuh"

namespace pp {

// cos and sin of 2 pi m / N at compile time: reduced to an eighth turn, Taylor
// series in double.
struct CosSin {
    double c, s;
};
constexpr CosSin eighth_turn(double x) {   // |x| <= pi / 4
    double c = 0.0, s = 0.0, t = 1.0;
    for (int k = 0; k < 24; ++k) {
        switch (k & 3) {
            case 0: c += t; break;
            case 1: s += t; break;
            case 2: c -= t; break;
            default: s -= t; break;
        }
        t *= x / (k + 1);
    }
    return {c, s};
}
constexpr CosSin root_of_unity(int m, int N) {
    // angle = 2 pi m / N = (pi / 2) q + r, |r| <= pi / 4
    const int q = (4 * m + N / 2) / N;
    const CosSin e = eighth_turn(1.57079632679489661923 * (double)(4 * m - q * N) / N);
    switch (q & 3) {
        case 0: return {e.c, e.s};
        case 1: return {-e.s, e.c};
        case 2: return {-e.c, -e.s};
        default: return {e.s, -e.c};
    }
}
template <int N> struct RootTable {
    float x[N], y[N];
    constexpr RootTable() : x(), y() {
        for (int m = 0; m < N; ++m) {
            const CosSin e = root_of_unity(m, N);
            x[m] = (float)e.c;
            y[m] = (float)-e.s;
        }
    }
};
#define PP_ROOTS(N)                                                                      \
    static __constant__ RootTable<N> c_r##N = RootTable<N>();                            \
    template <> __device__ __forceinline__ float2 cw<N>(int m) {                         \
        return make_float2(c_r##N.x[m], c_r##N.y[m]);                                    \
    }
PP_ROOTS(6) PP_ROOTS(9) PP_ROOTS(10) PP_ROOTS(15) PP_ROOTS(18) PP_ROOTS(25) PP_ROOTS(27) PP_ROOTS(30)
PP_ROOTS(32)
#undef PP_ROOTS

#define PP_REGFFT(N, A, B)                                                                         \
    template <bool INV> struct RegFft<N, INV> {                                                    \
        static __device__ __forceinline__ void run(float2* v, const float2* tw, int s) {           \
            reg_fft_ab<A, B, INV>(v, tw, s);                                                       \
        }                                                                                          \
    };
PP_REGFFT(6, 3, 2) PP_REGFFT(9, 3, 3) PP_REGFFT(10, 5, 2) PP_REGFFT(15, 5, 3) PP_REGFFT(18, 9, 2)
PP_REGFFT(25, 5, 5) PP_REGFFT(27, 9, 3) PP_REGFFT(30, 10, 3) PP_REGFFT(32, 8, 4)
#undef PP_REGFFT

}  // namespace pp
