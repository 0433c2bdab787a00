// Row and column FFT stages, compiled for every even length up to 1024 with prime
// factors 2, 3 and 5 (972 and 1000 have no pair of register factors), on the
// two-factor decomposition of pp_fft4.cuh: n = N1 N2, N1 <= N2 <= 32, input
// m = N2 m1 + m2, output k = k1 + N1 k2; one shared-memory transpose a transform,
// all global loads of a thread issued together, every twiddle from the table.
// Same index maps as the Stockham kernels of pp_kernels.cu (RowArgs, ColArgs).  In
// the row stages the second half's (line, k1) pairs are packed into the first
// RBG N1 threads, so that it runs in N1 / N2 of the warps.
//
// What bounds them: one read and one write per element, N1 loads in flight a
// thread.  A kernel that switches on the two factors at run time moves the same
// bytes at half the rate (two to three times the instructions, 70 to 150
// registers), and takes longer to compile than the 60 lengths do one by one.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "pp_fftgen.cuh"
#include "pp_lines.h"

namespace pp {

template <int N1, int N2> struct Line {
    static constexpr int n = N1 * N2, P = N2 | 1;
    static constexpr int cols_threads = TXG * N2, rows_threads = RBG * N2;
    static constexpr size_t cols_smem = sizeof(float2) * (n + N1 * P * TXG);
    static constexpr size_t yinv_smem = cols_smem + sizeof(float2) * n * TXG;
    static constexpr size_t rows_smem = sizeof(float2) * (n + N1 * P * RBG);
    static size_t rows_adj_smem(int nimg) { return rows_smem + sizeof(float2) * (size_t)RBG * nimg; }
};
// At most 128 registers a thread, and 8 CTAs an SM of the small blocks.
__host__ __device__ constexpr int line_min_ctas(int threads) { return threads < 512 ? 512 / threads : 1; }

// The round trip holds one transform at a time: 80 registers are enough up to
// N2 = 16 and 102 up to 20 (32 bytes spilled at 16 x 16, 40 at 20 x 20), and half as
// many threads more an SM: 148 -> 134 us at 12 x 80 x 180 x 200, whole normal operator
// of 100 x 256 x 108 x 7 256 -> 240 us.  The inverse y stage, which holds the map's N2
// values across the barrier as well, spills at 128 registers already (stores of 30 to
// 260 bytes for most lengths from 80 points on, 300 to 460 for N2 = 25 and 27 and at
// 10 x 20, 720 at 16 x 32) and took 156 -> 181 us under this cap.
__host__ __device__ constexpr int roundtrip_min_ctas(int threads) {
    const int t = threads <= 128 ? 768 : (threads <= 160 ? 640 : 512);
    return threads < t ? t / threads : 1;
}

__device__ __forceinline__ float2 tw_of(const float2* tws, int t, bool inv) {
    float2 w = tws[t];
    if (inv) w.y = -w.y;
    return w;
}
__device__ __forceinline__ void load_tw(float2* dst, const float2* __restrict__ src, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

// Column stage: TXG adjacent columns of one batch, thread (r, lane), lane the
// column; phase 1 thread r is m2, phase 2 thread r is k1; Y[k1][m2][lane] with an
// odd m2 pitch, so that the two k1 rows of a half-warp lie on different banks.
// Lanes past the last column load it again and store nothing.  Offsets within a
// batch fit 32 bits (the launcher checks).  src == dst is allowed.
template <int N1, int N2, bool INV, bool XIMG>
__global__ void __launch_bounds__(TXG * N2, line_min_ctas(TXG * N2)) line_cols_kernel(const LineCols L) {
    constexpr int n = N1 * N2, P = N2 | 1;
    extern __shared__ float2 sm[];
    float2* tws = sm;
    float2* Y = sm + n;
    const ColArgs& a = L.a;
    int ncols = a.ncols;
    float scale = a.scale;
    int64_t so = (int64_t)blockIdx.y * a.in_batch_stride, dof = (int64_t)blockIdx.y * a.out_batch_stride;
    const float *mi = a.mul_in, *mo = a.mul_out;
    if (L.items) {
        const ColItem it = L.items[blockIdx.y];
        ncols = it.ncols;
        if ((int)blockIdx.x * TXG >= ncols) return;
        so = it.src;
        dof = it.dst;
        scale *= it.scale;
        (INV ? mi : mo) = it.mask;
    }
    load_tw(tws, L.tw, n);
    const int lane = threadIdx.x & (TXG - 1), r = threadIdx.x / TXG;
    const int col = blockIdx.x * TXG + lane;
    const bool colok = col < ncols;
    const int lcol = colok ? col : ncols - 1;
    const float2* sb = L.src + so + lcol;
    const float2* xb = XIMG ? L.ximg + (int64_t)(blockIdx.y % L.nimgs) * a.Hin * ncols + lcol : nullptr;
    float2* db = L.dst + dof + col;
    if (mi) mi += (lcol / a.mi_cdiv) * a.mi_c;
    if (mo) mo += (lcol / a.mo_cdiv) * a.mo_c;
    int r0 = r + a.off_in;
    if (r0 >= n) r0 -= n;
    {
        float2 v[N1];
#pragma unroll
        for (int m1 = 0; m1 < N1; ++m1) {
            int row = N2 * m1 + r0;
            if (row >= n) row -= n;
            v[m1] = row < a.Hin ? sb[row * ncols] : make_float2(0.f, 0.f);
        }
        if (XIMG) {   // Hin = n
            float2 x[N1];
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) {
                int row = N2 * m1 + r0;
                if (row >= n) row -= n;
                x[m1] = xb[row * ncols];
            }
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) v[m1] = cmul(v[m1], x[m1]);
        }
        if (mi) {
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) {
                int row = N2 * m1 + r0;
                if (row >= n) row -= n;
                v[m1] = cscale(v[m1], row < a.Hin ? mi[row * a.mi_q] : 0.f);
            }
        }
        __syncthreads();   // the twiddle table
        fft4_phase1_exact<N1, N2, INV>(v, r, tws);
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) Y[(k1 * P + r) * TXG + lane] = v[k1];
    }
    __syncthreads();
    if (r < N1) {
        float2 u[N2];
#pragma unroll
        for (int m2 = 0; m2 < N2; ++m2) u[m2] = Y[(r * P + m2) * TXG + lane];
        RegFft<N2, INV>::run(u, tws, N1);
        if (mo) {
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) {
                int q = r + N1 * k2 + a.off_out;
                if (q >= n) q -= n;
                u[k2] = cscale(u[k2], q < a.Hout ? mo[q * a.mo_q] : 0.f);
            }
        }
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) {
            int q = r + N1 * k2 + a.off_out;
            if (q >= n) q -= n;
            if (q < a.Hout && colok) db[q * ncols] = cscale(u[k2], scale);
        }
    }
}

// Inverse y FFT of W[c][z][y][x] for every coil of a chunk, times conj(S_c),
// summed over the chunk: out = sum (+ out when !first); the last chunk applies
// out = scale * sum + alpha * operand.  grid (column groups, nz).
template <int N1, int N2>
__global__ void __launch_bounds__(TXG * N2, line_min_ctas(TXG * N2)) line_yinv_kernel(const LineYinv L) {
    constexpr int n = N1 * N2, P = N2 | 1;
    extern __shared__ float2 sm[];
    float2* tws = sm;
    float2* Y = sm + n;
    float2* acc = Y + N1 * P * TXG;
    load_tw(tws, L.tw, n);
    const int lane = threadIdx.x & (TXG - 1), r = threadIdx.x / TXG;
    const int nx = L.nx, col = blockIdx.x * TXG + lane;
    const bool colok = col < nx;
    const int64_t base = (int64_t)blockIdx.y * n * nx + (colok ? col : nx - 1);
    __syncthreads();
    for (int c = 0; c < L.ncoils; ++c) {
        const float2* Wc = L.W + c * L.nimg + base;
        const float2* Sc = L.S + c * L.nimg + base;
        {
            float2 v[N1];
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) v[m1] = Wc[(N2 * m1 + r) * nx];
            fft4_phase1_exact<N1, N2, true>(v, r, tws);
#pragma unroll
            for (int k1 = 0; k1 < N1; ++k1) Y[(k1 * P + r) * TXG + lane] = v[k1];
        }
        float2 s[N2];   // the map, read across the barrier
        if (r < N1) {
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) s[k2] = Sc[(r + N1 * k2) * nx];
        }
        __syncthreads();
        if (r < N1) {
            float2 u[N2];
#pragma unroll
            for (int m2 = 0; m2 < N2; ++m2) u[m2] = Y[(r * P + m2) * TXG + lane];
            RegFft<N2, true>::run(u, tws, N1);
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) u[k2] = cmulc(s[k2], u[k2]);
            if (c > 0) {
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) u[k2] = cadd(u[k2], acc[(r + N1 * k2) * TXG + lane]);
            }
            if (c + 1 < L.ncoils) {   // each element stays with this thread
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) acc[(r + N1 * k2) * TXG + lane] = u[k2];
            } else {
                float2* o = L.out + base;
                if (!L.first) {
#pragma unroll
                    for (int k2 = 0; k2 < N2; ++k2) u[k2] = cadd(u[k2], o[(r + N1 * k2) * nx]);
                }
                if (L.last) {
#pragma unroll
                    for (int k2 = 0; k2 < N2; ++k2) u[k2] = cscale(u[k2], L.scale);
                    if (L.operand) {
#pragma unroll
                        for (int k2 = 0; k2 < N2; ++k2)
                            u[k2] = cadd(u[k2], cscale(L.operand[base + (r + N1 * k2) * nx], L.alpha));
                    }
                }
                if (colok) {
#pragma unroll
                    for (int k2 = 0; k2 < N2; ++k2) o[(r + N1 * k2) * nx] = u[k2];
                }
            }
        }
        __syncthreads();
    }
}

// Column round trip: IFFT(mask . FFT(col)), mask in a.mul_out (mo_*).  The forward
// transform's output X[k1 + N1 k2] stays with its (k1) threads, whose inverse
// length-N2 DFT over k2 and twiddle W^-(m2 k1) feed the (m2) threads' inverse
// length-N1 DFT.  src == dst is allowed.
template <int N1, int N2>
__global__ void __launch_bounds__(TXG * N2, roundtrip_min_ctas(TXG * N2)) line_roundtrip_kernel(const LineCols L) {
    constexpr int n = N1 * N2, P = N2 | 1;
    extern __shared__ float2 sm[];
    float2* tws = sm;
    float2* Y = sm + n;
    const ColArgs& a = L.a;
    load_tw(tws, L.tw, n);
    const int lane = threadIdx.x & (TXG - 1), r = threadIdx.x / TXG;
    const int col = blockIdx.x * TXG + lane;
    const bool colok = col < a.ncols;
    const int lcol = colok ? col : a.ncols - 1;
    const float2* sb = L.src + (int64_t)blockIdx.y * a.in_batch_stride + lcol;
    float2* db = L.dst + (int64_t)blockIdx.y * a.out_batch_stride + lcol;
    const float* mk = a.mul_out + (lcol / a.mo_cdiv) * a.mo_c;
    {
        float2 v[N1];
#pragma unroll
        for (int m1 = 0; m1 < N1; ++m1) v[m1] = sb[(N2 * m1 + r) * a.ncols];
        __syncthreads();   // the twiddle table
        fft4_phase1_exact<N1, N2, false>(v, r, tws);
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) Y[(k1 * P + r) * TXG + lane] = v[k1];
    }
    __syncthreads();
    if (r < N1) {
        float2 u[N2];
#pragma unroll
        for (int m2 = 0; m2 < N2; ++m2) u[m2] = Y[(r * P + m2) * TXG + lane];
        RegFft<N2, false>::run(u, tws, N1);
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) u[k2] = cscale(u[k2], mk[(r + N1 * k2) * a.mo_q]);
        RegFft<N2, true>::run(u, tws, N1);
#pragma unroll
        for (int m2 = 0; m2 < N2; ++m2)
            Y[(r * P + m2) * TXG + lane] = m2 ? cmul(u[m2], tw_of(tws, m2 * r, true)) : u[m2];
    }
    __syncthreads();
    {
        float2 v[N1];
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) v[k1] = Y[(k1 * P + r) * TXG + lane];
        RegFft<N1, true>::run(v, tws, N2);
        if (colok) {
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) db[(N2 * m1 + r) * a.ncols] = v[m1];
        }
    }
}

// Row stage image -> k rows (coil expansion, weights, circular placement): RBG
// rows of one coil per CTA, thread (row, r).
template <int N1, int N2>
__global__ void __launch_bounds__(RBG * N2, line_min_ctas(RBG * N2)) line_rows_fwd_kernel(const LineRows L) {
    constexpr int n = N1 * N2, P = N2 | 1;
    extern __shared__ float2 sm[];
    float2* tws = sm;
    const RowArgs& a = L.a;
    int nrows = a.nrows;
    const float2* xs = L.src + (int64_t)blockIdx.y * L.src_batch_stride;
    const float2* ss = L.sens ? L.sens + (int64_t)blockIdx.y * a.coil_img_stride : nullptr;
    float2* od = L.dst + (int64_t)blockIdx.y * a.nrows * n;
    if (L.items) {
        const RowItem it = L.items[blockIdx.y];
        nrows = it.nrows;
        if ((int)blockIdx.x * RBG >= nrows) return;
        xs = L.src + it.src;
        ss = it.sens;
        od = L.dst + it.dst;
    }
    load_tw(tws, L.tw, n);
    const int b = threadIdx.x / N2, r = threadIdx.x - b * N2;
    float2* Y = sm + n + b * N1 * P;
    const int row = blockIdx.x * RBG + b;
    const int lrow = row < nrows ? row : nrows - 1;
    const float2* xr = xs + (int64_t)lrow * a.n;
    const float2* sr = ss ? ss + (int64_t)lrow * a.n : nullptr;
    const float wr = a.scale * (L.wrow ? L.wrow[lrow] : 1.f);
    int r0 = r + a.off_in;
    if (r0 >= n) r0 -= n;
    {
        float2 v[N1];
#pragma unroll
        for (int m1 = 0; m1 < N1; ++m1) {
            int i = N2 * m1 + r0;
            if (i >= n) i -= n;
            v[m1] = i < a.n ? xr[i] : make_float2(0.f, 0.f);
        }
        if (sr) {
            float2 s[N1];
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) {
                int i = N2 * m1 + r0;
                if (i >= n) i -= n;
                s[m1] = i < a.n ? sr[i] : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) v[m1] = cmul(v[m1], s[m1]);
        }
        if (L.wcol) {
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) {
                int i = N2 * m1 + r0;
                if (i >= n) i -= n;
                v[m1] = cscale(v[m1], i < a.n ? wr * L.wcol[i] : 0.f);
            }
        } else {
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) v[m1] = cscale(v[m1], wr);
        }
        __syncthreads();   // the twiddle table
        fft4_phase1_exact<N1, N2, false>(v, r, tws);
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) Y[k1 * P + r] = v[k1];
    }
    __syncthreads();
    if (threadIdx.x < RBG * N1) {
        const int b2 = N1 == N2 ? b : threadIdx.x / N1, k1 = N1 == N2 ? r : threadIdx.x - b2 * N1;
        const int row2 = blockIdx.x * RBG + b2;
        const float2* Y2 = sm + n + (b2 * N1 + k1) * P;
        float2 u[N2];
#pragma unroll
        for (int m2 = 0; m2 < N2; ++m2) u[m2] = Y2[m2];
        RegFft<N2, false>::run(u, tws, N1);
        if (row2 < nrows) {
            float2* o = od + (int64_t)row2 * n;
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) {
                int q = k1 + N1 * k2 + a.off_out;
                if (q >= n) q -= n;
                o[q] = u[k2];
            }
        }
    }
}

// Row stage k rows -> image with the conjugate-coil reduction and axpy epilogue of
// rows_adj_kernel.  A CTA's RBG lines are `rb` rows x RBG / rb coils; every line
// accumulates its coils (c = slot, slot + RBG / rb, ...) in shared memory, each
// element by one thread, and the slots of a row are summed at the end.
template <int N1, int N2>
__global__ void __launch_bounds__(RBG * N2, line_min_ctas(RBG * N2)) line_rows_adj_kernel(const LineRows L) {
    constexpr int n = N1 * N2, P = N2 | 1;
    extern __shared__ float2 sm[];
    float2* tws = sm;
    const RowArgs& a = L.a;
    int nrows = a.nrows, ncoils = L.ncoils;
    float scale = a.scale;
    const float2 *src = L.src, *sens = L.sens;
    float2* out = L.dst;
    int64_t cstride = a.coil_img_stride;
    const int rb = L.rb, cb = RBG / rb;
    if (L.items) {
        const RowItem it = L.items[blockIdx.y];
        nrows = it.nrows;
        if ((int)blockIdx.x * rb >= nrows) return;
        ncoils = it.ncoils;
        src += it.src;
        out += it.dst;
        sens = it.sens;
        scale *= it.scale;
        cstride = (int64_t)nrows * a.n;
    }
    load_tw(tws, L.tw, n);
    // (line, m2) in the first half, (line, k1) on the first RBG N1 threads after it
    const int b = threadIdx.x / N2, r = threadIdx.x - b * N2;
    const int b2 = N1 == N2 ? b : threadIdx.x / N1, k1 = N1 == N2 ? r : threadIdx.x - b2 * N1;
    // r < N1 holds where N1 = N2; written out it keeps the map's loads behind the
    // first half (in front of it, 18 x 18 and 20 x 20 spill 140 to 220 bytes)
    const bool second = N1 == N2 ? r < N1 : threadIdx.x < RBG * N1;
    float2* Y = sm + n + b * N1 * P;
    const float2* Y2 = sm + n + (b2 * N1 + k1) * P;
    float2* accs = sm + n + RBG * N1 * P;
    float2* acc = accs + b2 * a.n;
    for (int e = threadIdx.x; e < RBG * a.n; e += blockDim.x) accs[e] = make_float2(0.f, 0.f);
    const int slot = b / rb, row = blockIdx.x * rb + b - slot * rb;
    const int slot2 = N1 == N2 ? slot : b2 / rb, row2 = N1 == N2 ? row : blockIdx.x * rb + b2 - slot2 * rb;
    const float wr = (L.wrow && second && row2 < nrows) ? L.wrow[row2] : 1.f;
    int r0 = r + a.off_in;
    if (r0 >= n) r0 -= n;
    __syncthreads();
    for (int c0 = 0; c0 < ncoils; c0 += cb) {
        const int c = c0 + slot, c2 = c0 + slot2;
        const bool live2 = second && row2 < nrows && c2 < ncoils;
        const float2* sc = sens ? sens + c2 * cstride + (int64_t)row2 * a.n : nullptr;
        float2 s[N2];   // the map, read across the barrier
        auto read_map = [&] {
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) {
                int i = k1 + N1 * k2 + a.off_out;
                if (i >= n) i -= n;
                s[k2] = i < a.n ? sc[i] : make_float2(0.f, 0.f);
            }
        };
        if (row < nrows && c < ncoils) {
            const float2* sr = src + ((int64_t)c * nrows + row) * n;
            float2 v[N1];
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) {
                int s = N2 * m1 + r0;
                if (s >= n) s -= n;
                v[m1] = sr[s];
            }
            fft4_phase1_exact<N1, N2, true>(v, r, tws);
#pragma unroll
            for (int k1 = 0; k1 < N1; ++k1) Y[k1 * P + r] = v[k1];
            if (N1 == N2 && sc && second) read_map();
        }
        if (N1 != N2 && sc && live2) read_map();
        __syncthreads();
        if (live2) {
            float2 u[N2];
#pragma unroll
            for (int m2 = 0; m2 < N2; ++m2) u[m2] = Y2[m2];
            RegFft<N2, true>::run(u, tws, N1);
            if (sc) {
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) u[k2] = cmulc(s[k2], u[k2]);
            }
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) {
                int i = k1 + N1 * k2 + a.off_out;
                if (i >= n) i -= n;
                if (i < a.n) acc[i] = cadd(acc[i], cscale(u[k2], L.wcol ? wr * L.wcol[i] : wr));
            }
        }
        __syncthreads();
    }
    // the CTA's rows are contiguous in the image; eight loads of the operand in
    // flight (one at a time they took 26 us of a 68 us launch)
    const int64_t o0 = (int64_t)blockIdx.x * rb * a.n;
    const int ne = min(rb, nrows - (int)blockIdx.x * rb) * a.n, sn = rb * a.n;
    for (int e0 = threadIdx.x; e0 < ne; e0 += 8 * blockDim.x) {
        float2 op[8];
        if (L.operand) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int e = e0 + u * blockDim.x;
                if (e < ne) op[u] = L.operand[o0 + e];
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int e = e0 + u * blockDim.x;
            if (e >= ne) break;
            float2 v = accs[e];
            for (int s = 1; s < cb; ++s) v = cadd(v, accs[s * sn + e]);
            v = cscale(v, scale);
            if (L.operand) v = cadd(v, cscale(op[u], L.alpha));
            out[o0 + e] = v;
        }
    }
}

constexpr int kLineSmem = 200 * 1024;

template <auto Kernel, class Args>
cudaError_t line_go(dim3 grid, int threads, size_t smem, cudaStream_t st, const Args& args) {
    if (smem > 48 * 1024) {
        if (smem > (size_t)kLineSmem) return cudaErrorInvalidValue;
        const cudaError_t e = allow_smem<Kernel, kLineSmem>();
        if (e != cudaSuccess) return e;
    }
    return launch_ex(Kernel, grid, dim3(threads), smem, st, false, 0, args);
}

template <int N1, int N2> cudaError_t line_launch(LineOp op, const LineUnion& u, dim3 grid, cudaStream_t st) {
    using K = Line<N1, N2>;
    switch (op) {
        case LineOp::ColsFwd:
            return line_go<line_cols_kernel<N1, N2, false, false>>(grid, K::cols_threads, K::cols_smem, st, *u.cols);
        case LineOp::ColsInv:
            return line_go<line_cols_kernel<N1, N2, true, false>>(grid, K::cols_threads, K::cols_smem, st, *u.cols);
        case LineOp::RowsFwd:
            return line_go<line_rows_fwd_kernel<N1, N2>>(grid, K::rows_threads, K::rows_smem, st, *u.rows);
        case LineOp::RowsAdj:
            return line_go<line_rows_adj_kernel<N1, N2>>(grid, K::rows_threads, K::rows_adj_smem(u.rows->a.n), st,
                                                         *u.rows);
        default: break;
    }
    // the 3-D normal operator's: image axes end at 512, only grids are longer
    if constexpr (K::n <= 512) switch (op) {
        case LineOp::ColsFwdImg:
            return line_go<line_cols_kernel<N1, N2, false, true>>(grid, K::cols_threads, K::cols_smem, st, *u.cols);
        case LineOp::RoundTrip:
            return line_go<line_roundtrip_kernel<N1, N2>>(grid, K::cols_threads, K::cols_smem, st, *u.cols);
        case LineOp::Yinv:
            return line_go<line_yinv_kernel<N1, N2>>(grid, K::cols_threads, K::yinv_smem, st, *u.yinv);
        default: break;
    }
    return cudaErrorInvalidValue;
}

}  // namespace pp
