// Two-factor FFT for every supported length (prime factors 2, 3, 5): n = N1 N2
// with both factors among the register DFT lengths below, chosen at run time.
// The decomposition is pp_fft4.cuh's: input m = N2 m1 + m2, output
// k = k1 + N1 k2; phase 1 is a length-N1 DFT over m1 with the twiddle
// W_n^(m2 k1), phase 2 a length-N2 DFT over m2.  A phase switches on its DFT
// length (the same for the whole launch) and is unrolled inside each case, so
// one kernel serves all lengths with two passes over shared memory instead of
// one per radix stage of the Stockham form (3 to 5 for these lengths).
#pragma once
#include <type_traits>

#include "pp_fft4.cuh"
#include "pp_internal.h"

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

// Length-n DFT for the register lengths up to NMAX (16, 24 or 32: the cases above
// it are left out, which bounds the kernel's registers).  ld fills and st
// consumes the whole array, so that a phase's global loads are all issued before
// anything waits for one of them.
#define PP_GEN_CASES(X) X(3) X(4) X(5) X(6) X(8) X(9) X(10) X(12) X(15) X(16) X(18) X(20) X(24) X(25) X(27) X(30) X(32)

template <class A> __host__ __device__ constexpr int len_of() {
    return (int)(sizeof(A) / sizeof(float2));
}
#define PP_LEN(v) (::pp::len_of<std::remove_reference_t<decltype(v)>>())

template <int NMAX, bool INV, class Ld, class St>
__device__ __forceinline__ void dft_any(int n, Ld ld, St st) {
    switch (n) {
#define PP_CASE(N)                                  \
        case N:                                     \
            if constexpr (N <= NMAX) {              \
                float2 v[N];                        \
                ld(v);                              \
                RegFft<N, INV>::run(v, nullptr, 1); \
                st(v);                              \
            }                                       \
            break;
        PP_GEN_CASES(PP_CASE)
#undef PP_CASE
        default: break;
    }
}

// Length-n DFT, `mid` on its outputs, inverse length-n DFT.
template <int NMAX, class Ld, class Mid, class St>
__device__ __forceinline__ void dft_round_trip_any(int n, Ld ld, Mid mid, St st) {
    switch (n) {
#define PP_CASE(N)                                    \
        case N:                                       \
            if constexpr (N <= NMAX) {                \
                float2 v[N];                          \
                ld(v);                                \
                RegFft<N, false>::run(v, nullptr, 1); \
                mid(v);                               \
                RegFft<N, true>::run(v, nullptr, 1);  \
                st(v);                                \
            }                                         \
            break;
        PP_GEN_CASES(PP_CASE)
#undef PP_CASE
        default: break;
    }
}

// n = n1 * n2 with both factors register DFT lengths, the larger as small as
// possible (n2 >= n1); false when there is no such pair (n above 32 * 32, or
// tiny).
inline bool gen_split(int n, int* n1, int* n2) {
    static const int len[] = {3, 4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32};
    int best = 0;
    for (int a : len)
        for (int b : len)
            if (a <= b && a * b == n && (!best || b < best)) {
                best = b;
                *n1 = a;
                *n2 = b;
            }
    return best != 0;
}

// ---- shared by the stage kernels ----
constexpr int TXG = 8;    // columns per CTA
constexpr int RBG = 8;    // lines (rows, or rows x coils) per CTA in the row stages

__device__ __forceinline__ float2 twiddle(const float2* tws, int t, bool inv) {
    float2 w = tws[t];
    if (inv) w.y = -w.y;
    return w;
}
// A copy the compiler cannot see through: inside a coil loop it keeps the index
// arithmetic of every DFT-length case from being hoisted out of the loop, which
// took 255 registers.
__device__ __forceinline__ int opaque(int v) {
    asm volatile("" : "+r"(v));
    return v;
}
__device__ __forceinline__ void load_tw(float2* dst, const float2* __restrict__ src, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

inline int y_elems(const GenSplit& g) { return g.n1 * (g.n2 | 1); }

inline pp_status check_gen(const char* what) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_status(e, what);
    ++g_launches;
    if (g_profiler) g_profiler->mark(what);
    return PP_OK;
}

// Register class of the split: the larger factor decides.
#define PP_GEN_CLASS(n2, CALL)      \
    do {                            \
        if ((n2) <= 16) { CALL(16); } \
        else if ((n2) <= 24) { CALL(24); } \
        else { CALL(32); }          \
    } while (0)

}  // namespace pp
