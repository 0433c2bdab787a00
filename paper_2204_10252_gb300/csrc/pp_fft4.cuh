// Register-resident FFTs for the transform lengths of the workloads
// (n = N1 * N2 with N1 = 16 and N2 in {8, 12, 16, 20, 24}: 128 ... 384).
//
// Four-step decomposition, input index m = N2*m1 + m2, output k = k1 + N1*k2:
//   X[k] = sum_m2 W_N2^(m2 k2) [ W_n^(m2 k1) sum_m1 x[N2 m1 + m2] W_N1^(m1 k1) ]
// Phase 1: one thread per (transform, m2) loads N1 inputs into registers,
//          runs the length-N1 DFT, applies W_n^(m2 k1), writes Y[k1][m2] to
//          shared memory.
// Phase 2: one thread per (transform, k1) reads Y[k1][0..N2), runs the
//          length-N2 DFT and holds X[k1 + N1 k2] in registers.
// Each register DFT of composite length A*B is itself a four-step over the
// radix-2/3/4/5/8 kernels of pp_fft.cuh, fully unrolled.  Twiddles come from
// the shared table w[t] = exp(-2 pi i t / n): W_L^m = w[m * n / L].
#pragma once
#include "pp_fft.cuh"

namespace pp {

// W_N^m = exp(-2 pi i m / N) for the register DFT lengths (mathematical
// constants, rounded to float); indexed with compile-time m after unrolling,
// so they become constant-bank operands.
static __constant__ float2 c_w12[12] = {{1.000000000e+00f, -0.000000000e+00f}, {8.660254038e-01f, -5.000000000e-01f}, {5.000000000e-01f, -8.660254038e-01f}, {6.123233996e-17f, -1.000000000e+00f}, {-5.000000000e-01f, -8.660254038e-01f}, {-8.660254038e-01f, -5.000000000e-01f}, {-1.000000000e+00f, -1.224646799e-16f}, {-8.660254038e-01f, 5.000000000e-01f}, {-5.000000000e-01f, 8.660254038e-01f}, {-1.836970199e-16f, 1.000000000e+00f}, {5.000000000e-01f, 8.660254038e-01f}, {8.660254038e-01f, 5.000000000e-01f}};
static __constant__ float2 c_w16[16] = {{1.000000000e+00f, -0.000000000e+00f}, {9.238795325e-01f, -3.826834324e-01f}, {7.071067812e-01f, -7.071067812e-01f}, {3.826834324e-01f, -9.238795325e-01f}, {6.123233996e-17f, -1.000000000e+00f}, {-3.826834324e-01f, -9.238795325e-01f}, {-7.071067812e-01f, -7.071067812e-01f}, {-9.238795325e-01f, -3.826834324e-01f}, {-1.000000000e+00f, -1.224646799e-16f}, {-9.238795325e-01f, 3.826834324e-01f}, {-7.071067812e-01f, 7.071067812e-01f}, {-3.826834324e-01f, 9.238795325e-01f}, {-1.836970199e-16f, 1.000000000e+00f}, {3.826834324e-01f, 9.238795325e-01f}, {7.071067812e-01f, 7.071067812e-01f}, {9.238795325e-01f, 3.826834324e-01f}};
static __constant__ float2 c_w20[20] = {{1.000000000e+00f, -0.000000000e+00f}, {9.510565163e-01f, -3.090169944e-01f}, {8.090169944e-01f, -5.877852523e-01f}, {5.877852523e-01f, -8.090169944e-01f}, {3.090169944e-01f, -9.510565163e-01f}, {6.123233996e-17f, -1.000000000e+00f}, {-3.090169944e-01f, -9.510565163e-01f}, {-5.877852523e-01f, -8.090169944e-01f}, {-8.090169944e-01f, -5.877852523e-01f}, {-9.510565163e-01f, -3.090169944e-01f}, {-1.000000000e+00f, -1.224646799e-16f}, {-9.510565163e-01f, 3.090169944e-01f}, {-8.090169944e-01f, 5.877852523e-01f}, {-5.877852523e-01f, 8.090169944e-01f}, {-3.090169944e-01f, 9.510565163e-01f}, {-1.836970199e-16f, 1.000000000e+00f}, {3.090169944e-01f, 9.510565163e-01f}, {5.877852523e-01f, 8.090169944e-01f}, {8.090169944e-01f, 5.877852523e-01f}, {9.510565163e-01f, 3.090169944e-01f}};
static __constant__ float2 c_w24[24] = {{1.000000000e+00f, -0.000000000e+00f}, {9.659258263e-01f, -2.588190451e-01f}, {8.660254038e-01f, -5.000000000e-01f}, {7.071067812e-01f, -7.071067812e-01f}, {5.000000000e-01f, -8.660254038e-01f}, {2.588190451e-01f, -9.659258263e-01f}, {6.123233996e-17f, -1.000000000e+00f}, {-2.588190451e-01f, -9.659258263e-01f}, {-5.000000000e-01f, -8.660254038e-01f}, {-7.071067812e-01f, -7.071067812e-01f}, {-8.660254038e-01f, -5.000000000e-01f}, {-9.659258263e-01f, -2.588190451e-01f}, {-1.000000000e+00f, -1.224646799e-16f}, {-9.659258263e-01f, 2.588190451e-01f}, {-8.660254038e-01f, 5.000000000e-01f}, {-7.071067812e-01f, 7.071067812e-01f}, {-5.000000000e-01f, 8.660254038e-01f}, {-2.588190451e-01f, 9.659258263e-01f}, {-1.836970199e-16f, 1.000000000e+00f}, {2.588190451e-01f, 9.659258263e-01f}, {5.000000000e-01f, 8.660254038e-01f}, {7.071067812e-01f, 7.071067812e-01f}, {8.660254038e-01f, 5.000000000e-01f}, {9.659258263e-01f, 2.588190451e-01f}};

template <int L> __device__ __forceinline__ float2 cw(int m);
template <> __device__ __forceinline__ float2 cw<12>(int m) { return c_w12[m]; }
template <> __device__ __forceinline__ float2 cw<16>(int m) { return c_w16[m]; }
template <> __device__ __forceinline__ float2 cw<20>(int m) { return c_w20[m]; }
template <> __device__ __forceinline__ float2 cw<24>(int m) { return c_w24[m]; }

template <int N, bool INV> struct RegFft;

template <bool INV> struct RegFft<2, INV> {
    static __device__ __forceinline__ void run(float2* v, const float2*, int) { Dft<2, INV>::run(v); }
};
template <bool INV> struct RegFft<3, INV> {
    static __device__ __forceinline__ void run(float2* v, const float2*, int) { Dft<3, INV>::run(v); }
};
template <bool INV> struct RegFft<4, INV> {
    static __device__ __forceinline__ void run(float2* v, const float2*, int) { Dft<4, INV>::run(v); }
};
template <bool INV> struct RegFft<5, INV> {
    static __device__ __forceinline__ void run(float2* v, const float2*, int) { Dft<5, INV>::run(v); }
};
template <bool INV> struct RegFft<8, INV> {
    static __device__ __forceinline__ void run(float2* v, const float2*, int) { Dft<8, INV>::run(v); }
};

// Length A*B in registers; `step` = n / (A*B) indexes the shared twiddle table.
template <int A, int B, bool INV>
__device__ __forceinline__ void reg_fft_ab(float2* v, const float2* __restrict__ tw, int step) {
    float2 t[A * B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
        float2 u[A];
#pragma unroll
        for (int a = 0; a < A; ++a) u[a] = v[B * a + b];
        RegFft<A, INV>::run(u, tw, step * B);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) t[b * A + k1] = u[k1];
    }
#pragma unroll
    for (int b = 1; b < B; ++b)
#pragma unroll
        for (int k1 = 1; k1 < A; ++k1) {
            float2 w = cw<A * B>(b * k1);
            if (INV) w.y = -w.y;
            t[b * A + k1] = cmul(t[b * A + k1], w);
        }
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
        float2 u[B];
#pragma unroll
        for (int b = 0; b < B; ++b) u[b] = t[b * A + k1];
        RegFft<B, INV>::run(u, tw, step * A);
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = u[k2];
    }
}

template <bool INV> struct RegFft<12, INV> {
    static __device__ __forceinline__ void run(float2* v, const float2* tw, int s) { reg_fft_ab<4, 3, INV>(v, tw, s); }
};
template <bool INV> struct RegFft<16, INV> {
    static __device__ __forceinline__ void run(float2* v, const float2* tw, int s) { reg_fft_ab<4, 4, INV>(v, tw, s); }
};
template <bool INV> struct RegFft<20, INV> {
    static __device__ __forceinline__ void run(float2* v, const float2* tw, int s) { reg_fft_ab<4, 5, INV>(v, tw, s); }
};
template <bool INV> struct RegFft<24, INV> {
    static __device__ __forceinline__ void run(float2* v, const float2* tw, int s) { reg_fft_ab<8, 3, INV>(v, tw, s); }
};

// Fast lengths: returns N2 for n = 16 * N2 with a register kernel, else 0.
__host__ __device__ __forceinline__ int fft4_n2(int n) {
    if (n % 16) return 0;
    const int n2 = n / 16;
    return (n2 == 8 || n2 == 12 || n2 == 16 || n2 == 20 || n2 == 24) ? n2 : 0;
}

// Phase 1 for one (transform, m2): v holds x[N2*m1 + m2], m1 < N1, on entry;
// on exit v[k1] = W_n^(m2 k1) * sum_m1 x[N2 m1 + m2] W_N1^(m1 k1).
template <int N1, int N2, bool INV>
__device__ __forceinline__ void fft4_phase1(float2* v, int m2, const float2* __restrict__ tw) {
    RegFft<N1, INV>::run(v, tw, N2);
    // W_n^(m2 k1): four table loads (k1 = 1..4), the rest by w_k = w_(k-4) w_4
    float2 w[N1];
    w[0] = make_float2(1.f, 0.f);
#pragma unroll
    for (int k1 = 1; k1 <= 4 && k1 < N1; ++k1) w[k1] = tw[m2 * k1];
#pragma unroll
    for (int k1 = 5; k1 < N1; ++k1) w[k1] = cmul(w[k1 - 4], w[4]);
#pragma unroll
    for (int k1 = 1; k1 < N1; ++k1) {
        float2 ww = w[k1];
        if (INV) ww.y = -ww.y;
        v[k1] = cmul(v[k1], ww);
    }
}

// The same with every twiddle from the table: the products of the form above
// leave up to three more roundings in them.  One more shared-memory read per
// element, so not where shared memory bounds the kernel.
template <int N1, int N2, bool INV>
__device__ __forceinline__ void fft4_phase1_exact(float2* v, int m2, const float2* __restrict__ tw) {
    RegFft<N1, INV>::run(v, tw, N2);
#pragma unroll
    for (int k1 = 1; k1 < N1; ++k1) {
        float2 ww = tw[m2 * k1];
        if (INV) ww.y = -ww.y;
        v[k1] = cmul(v[k1], ww);
    }
}

// Phase 2 for one (transform, k1): u holds Y[k1][m2], m2 < N2; on exit
// u[k2] = X[k1 + N1 k2].
template <int N1, int N2, bool INV>
__device__ __forceinline__ void fft4_phase2(float2* u, const float2* __restrict__ tw) {
    RegFft<N2, INV>::run(u, tw, N1);
}

}  // namespace pp

namespace pp {

// Split thread-block-cluster barrier.  arrive_release publishes this CTA's
// earlier shared-memory writes to the cluster, wait_acquire makes the other
// CTAs' visible; arrive_relaxed orders nothing (for a barrier that only
// says "done reading").  All threads of the CTA execute each of them.
__device__ __forceinline__ void cluster_arrive_release() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive_relaxed() {
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_wait_acquire() {
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

}  // namespace pp
