// Row and column stages on the two-factor FFT of
// pp_fftgen.cuh, for the lengths without a compiled four-step kernel
// (pp_kernels4.cu).  Same contracts as the Stockham kernels of pp_kernels.cu,
// which remain for lengths without two register factors.
//
// What bounds them: one read and one write per element, with as many loads in
// flight per thread as the first factor.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "pp_fftgen.cuh"
#include "pp_internal.h"

namespace pp {
namespace {

// Phase 1's output with its twiddle into Y[k1][m2], phase 2's input from it; `es`
// and `base` place element (k1, m2) at Y[(k1 * P + m2) * es + base].
template <bool INV, class A>
__device__ __forceinline__ void put_twiddled(A& v, float2* Y, const float2* tws, int P, int r, int es,
                                             int base) {
#pragma unroll
    for (int k1 = 0; k1 < PP_LEN(v); ++k1) Y[(k1 * P + r) * es + base] = cmul(v[k1], twiddle(tws, r * k1, INV));
}
template <class A>
__device__ __forceinline__ void get_row(A& v, const float2* Y, int P, int r, int es, int base) {
#pragma unroll
    for (int m2 = 0; m2 < PP_LEN(v); ++m2) v[m2] = Y[(r * P + m2) * es + base];
}

// ---------------------------------------------------------------------------
// Column stages: TXG adjacent columns of one batch, thread (r, lane), lane the
// column.  Phase 1 thread r is m2, phase 2 thread r is k1; Y[k1][m2][lane] with
// an odd m2 pitch, so that the two k1 rows of a half-warp lie on different banks.
// Lanes past the last column load it again and store nothing.  XIMG: the input
// is multiplied by an image, batch b by image b % nimgs.  Offsets within one
// batch fit 32 bits (the launcher checks).
// ---------------------------------------------------------------------------
template <int NMAX, bool INV, bool XIMG>
__global__ void __launch_bounds__(TXG * NMAX)
gen_cols_kernel(GenSplit g, const float2* __restrict__ tw, ColArgs a, const float2* src, float2* dst,
                const float2* __restrict__ ximg, int nimgs) {
    extern __shared__ float2 sm[];
    const int n = g.n1 * g.n2, P = g.n2 | 1;
    float2* tws = sm;
    float2* Y = sm + n;
    load_tw(tws, tw, n);
    const int lane = threadIdx.x & (TXG - 1), r = threadIdx.x / TXG;
    const int col = blockIdx.x * TXG + lane;
    const bool colok = col < a.ncols;
    const int lcol = colok ? col : a.ncols - 1;
    const float2* sb = src + (int64_t)blockIdx.y * a.in_batch_stride + lcol;
    const float2* xb = XIMG ? ximg + (int64_t)(blockIdx.y % nimgs) * a.Hin * a.ncols + lcol : nullptr;
    float2* db = dst + (int64_t)blockIdx.y * a.out_batch_stride + col;
    const float* mi = a.mul_in ? a.mul_in + (lcol / a.mi_cdiv) * a.mi_c : nullptr;
    const float* mo = a.mul_out ? a.mul_out + (lcol / a.mo_cdiv) * a.mo_c : nullptr;
    int r0 = r + a.off_in;
    if (r0 >= n) r0 -= n;
    __syncthreads();
    dft_any<NMAX, INV>(
        g.n1,
        [&](auto& v) {
#pragma unroll
            for (int m1 = 0; m1 < PP_LEN(v); ++m1) {
                int row = g.n2 * m1 + r0;
                if (row >= n) row -= n;
                v[m1] = row < a.Hin ? sb[row * a.ncols] : make_float2(0.f, 0.f);
                if (XIMG) v[m1] = cmul(v[m1], xb[row * a.ncols]);   // Hin = n
            }
            if (mi) {
#pragma unroll
                for (int m1 = 0; m1 < PP_LEN(v); ++m1) {
                    int row = g.n2 * m1 + r0;
                    if (row >= n) row -= n;
                    v[m1] = cscale(v[m1], row < a.Hin ? mi[row * a.mi_q] : 0.f);
                }
            }
        },
        [&](auto& v) { put_twiddled<INV>(v, Y, tws, P, r, TXG, lane); });
    __syncthreads();
    if (r < g.n1) {
        dft_any<NMAX, INV>(
            g.n2, [&](auto& v) { get_row(v, Y, P, r, TXG, lane); },
            [&](auto& v) {
                if (mo) {
#pragma unroll
                    for (int k2 = 0; k2 < PP_LEN(v); ++k2) {
                        int q = r + g.n1 * k2 + a.off_out;
                        if (q >= n) q -= n;
                        v[k2] = cscale(v[k2], q < a.Hout ? mo[q * a.mo_q] : 0.f);
                    }
                }
#pragma unroll
                for (int k2 = 0; k2 < PP_LEN(v); ++k2) {
                    int q = r + g.n1 * k2 + a.off_out;
                    if (q >= n) q -= n;
                    if (q < a.Hout && colok) db[q * a.ncols] = cscale(v[k2], a.scale);
                }
            });
    }
}

// Inverse y FFT of W[c][z][y][x] for every coil of a chunk, times conj(S_c),
// summed over the chunk: out = sum (+ out when !first); the last chunk applies
// out = scale * sum + alpha * operand.  grid (column groups, nz).
template <int NMAX>
__global__ void __launch_bounds__(TXG * NMAX)
gen_yinv_accum_kernel(GenSplit g, const float2* __restrict__ tw, int nx, int64_t nimg, int ncoils,
                      const float2* __restrict__ W, const float2* __restrict__ S, float2* out,
                      int first, int last, float scale, const float2* operand, float alpha) {
    extern __shared__ float2 sm[];
    const int n = g.n1 * g.n2, P = g.n2 | 1;
    float2* tws = sm;
    float2* Y = sm + n;
    float2* acc = Y + g.n1 * P * TXG;
    load_tw(tws, tw, n);
    const int lane = threadIdx.x & (TXG - 1);
    const int col = blockIdx.x * TXG + lane;
    const bool colok = col < nx;
    const int64_t base = (int64_t)blockIdx.y * n * nx + (colok ? col : nx - 1);
    __syncthreads();
    for (int c = 0; c < ncoils; ++c) {
        const int r = opaque(threadIdx.x / TXG);
        const float2* Wc = W + c * nimg + base;
        const float2* Sc = S + c * nimg + base;
        dft_any<NMAX, true>(
            g.n1,
            [&](auto& v) {
#pragma unroll
                for (int m1 = 0; m1 < PP_LEN(v); ++m1) v[m1] = Wc[(g.n2 * m1 + r) * nx];
            },
            [&](auto& v) { put_twiddled<true>(v, Y, tws, P, r, TXG, lane); });
        __syncthreads();
        if (r < g.n1)
            dft_any<NMAX, true>(
                g.n2, [&](auto& v) { get_row(v, Y, P, r, TXG, lane); },
                [&](auto& v) {
#pragma unroll
                    for (int k2 = 0; k2 < PP_LEN(v); ++k2)
                        v[k2] = cmulc(Sc[(r + g.n1 * k2) * nx], v[k2]);
                    if (c > 0) {
#pragma unroll
                        for (int k2 = 0; k2 < PP_LEN(v); ++k2)
                            v[k2] = cadd(v[k2], acc[(r + g.n1 * k2) * TXG + lane]);
                    }
                    if (c + 1 < ncoils) {   // each element stays with this thread
#pragma unroll
                        for (int k2 = 0; k2 < PP_LEN(v); ++k2) acc[(r + g.n1 * k2) * TXG + lane] = v[k2];
                        return;
                    }
                    float2* o = out + base;
                    if (!first) {
#pragma unroll
                        for (int k2 = 0; k2 < PP_LEN(v); ++k2) v[k2] = cadd(v[k2], o[(r + g.n1 * k2) * nx]);
                    }
                    if (last) {
#pragma unroll
                        for (int k2 = 0; k2 < PP_LEN(v); ++k2) v[k2] = cscale(v[k2], scale);
                        if (operand) {
#pragma unroll
                            for (int k2 = 0; k2 < PP_LEN(v); ++k2)
                                v[k2] = cadd(v[k2], cscale(operand[base + (r + g.n1 * k2) * nx], alpha));
                        }
                    }
                    if (!colok) return;
#pragma unroll
                    for (int k2 = 0; k2 < PP_LEN(v); ++k2) o[(r + g.n1 * k2) * nx] = v[k2];
                });
        __syncthreads();
    }
}

// Column round trip in place: IFFT(mask . FFT(col)); the forward transform's
// output X[k1 + n1 k2] stays with its (k1) threads, whose inverse length-n2 DFT
// over k2 and twiddle W^-(m2 k1) feed the (m2) threads' inverse length-n1 DFT.
template <int NMAX>
__global__ void __launch_bounds__(TXG * NMAX)
gen_cols_roundtrip_kernel(GenSplit g, const float2* __restrict__ tw, ColArgs a,
                          const float* __restrict__ mask_fo, const float2* src, float2* dst) {
    extern __shared__ float2 sm[];
    const int n = g.n1 * g.n2, P = g.n2 | 1;
    float2* tws = sm;
    float2* Y = sm + n;
    load_tw(tws, tw, n);
    const int lane = threadIdx.x & (TXG - 1), r = threadIdx.x / TXG;
    const int col = blockIdx.x * TXG + lane;
    const bool colok = col < a.ncols;
    const int lcol = colok ? col : a.ncols - 1;
    const float2* sb = src + (int64_t)blockIdx.y * a.in_batch_stride + lcol;
    float2* db = dst + (int64_t)blockIdx.y * a.out_batch_stride + lcol;
    const float* mk = mask_fo + (lcol / a.mo_cdiv) * a.mo_c;
    __syncthreads();
    dft_any<NMAX, false>(
        g.n1,
        [&](auto& v) {
#pragma unroll
            for (int m1 = 0; m1 < PP_LEN(v); ++m1) v[m1] = sb[(g.n2 * m1 + r) * a.ncols];
        },
        [&](auto& v) { put_twiddled<false>(v, Y, tws, P, r, TXG, lane); });
    __syncthreads();
    if (r < g.n1)
        dft_round_trip_any<NMAX>(
            g.n2, [&](auto& v) { get_row(v, Y, P, r, TXG, lane); },
            [&](auto& v) {
#pragma unroll
                for (int k2 = 0; k2 < PP_LEN(v); ++k2)
                    v[k2] = cscale(v[k2], mk[(r + g.n1 * k2) * a.mo_q]);
            },
            [&](auto& v) {
#pragma unroll
                for (int m2 = 0; m2 < PP_LEN(v); ++m2)
                    Y[(r * P + m2) * TXG + lane] = cmul(v[m2], twiddle(tws, r * m2, true));
            });
    __syncthreads();
    dft_any<NMAX, true>(
        g.n1,
        [&](auto& v) {
#pragma unroll
            for (int k1 = 0; k1 < PP_LEN(v); ++k1) v[k1] = Y[(k1 * P + r) * TXG + lane];
        },
        [&](auto& v) {
            if (!colok) return;
#pragma unroll
            for (int m1 = 0; m1 < PP_LEN(v); ++m1) db[(g.n2 * m1 + r) * a.ncols] = v[m1];
        });
}

// ---------------------------------------------------------------------------
// Row stages: RBG lines per CTA, thread (line, r).
// ---------------------------------------------------------------------------
template <int NMAX>
__global__ void __launch_bounds__(RBG * NMAX)
gen_rows_fwd_kernel(GenSplit g, const float2* __restrict__ tw, RowArgs a, const float2* __restrict__ x,
                    int64_t x_batch_stride, const float2* __restrict__ sens,
                    const float* __restrict__ wrow, const float* __restrict__ wcol,
                    float2* __restrict__ out) {
    extern __shared__ float2 sm[];
    const int n = g.n1 * g.n2, P = g.n2 | 1;
    float2* tws = sm;
    load_tw(tws, tw, n);
    const int b = threadIdx.x / g.n2, r = threadIdx.x - b * g.n2;
    float2* Y = sm + n + b * g.n1 * P;
    const int c = blockIdx.y;
    const int row = blockIdx.x * RBG + b;
    const bool live = row < a.nrows;
    const int lrow = live ? row : a.nrows - 1;
    const float2* xr = x + (int64_t)c * x_batch_stride + (int64_t)lrow * a.n;
    const float2* sr = sens ? sens + (int64_t)c * a.coil_img_stride + (int64_t)lrow * a.n : nullptr;
    const float wr = a.scale * (wrow ? wrow[lrow] : 1.f);
    int r0 = r + a.off_in;
    if (r0 >= n) r0 -= n;
    __syncthreads();
    dft_any<NMAX, false>(
        g.n1,
        [&](auto& v) {
            constexpr int N = PP_LEN(v);
#pragma unroll
            for (int m1 = 0; m1 < N; ++m1) {
                int i = g.n2 * m1 + r0;
                if (i >= n) i -= n;
                v[m1] = i < a.n ? xr[i] : make_float2(0.f, 0.f);
            }
            if (sr) {
                float2 s[N];
#pragma unroll
                for (int m1 = 0; m1 < N; ++m1) {
                    int i = g.n2 * m1 + r0;
                    if (i >= n) i -= n;
                    s[m1] = i < a.n ? sr[i] : make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int m1 = 0; m1 < N; ++m1) v[m1] = cmul(v[m1], s[m1]);
            }
            if (wcol) {
#pragma unroll
                for (int m1 = 0; m1 < N; ++m1) {
                    int i = g.n2 * m1 + r0;
                    if (i >= n) i -= n;
                    v[m1] = cscale(v[m1], i < a.n ? wr * wcol[i] : 0.f);
                }
            } else {
#pragma unroll
                for (int m1 = 0; m1 < N; ++m1) v[m1] = cscale(v[m1], wr);
            }
        },
        [&](auto& v) { put_twiddled<false>(v, Y, tws, P, r, 1, 0); });
    __syncthreads();
    if (r < g.n1) {
        float2* o = out + ((int64_t)c * a.nrows + lrow) * n;
        dft_any<NMAX, false>(
            g.n2, [&](auto& v) { get_row(v, Y, P, r, 1, 0); },
            [&](auto& v) {
                if (!live) return;
#pragma unroll
                for (int k2 = 0; k2 < PP_LEN(v); ++k2) {
                    int q = r + g.n1 * k2 + a.off_out;
                    if (q >= n) q -= n;
                    o[q] = v[k2];
                }
            });
    }
}

// k rows -> image with the conjugate-coil reduction and axpy epilogue of
// rows_adj_kernel.  A CTA's RBG lines are `rb` rows x RBG / rb coils; every line
// accumulates its coils (c = slot, slot + RBG / rb, ...) in shared memory, each
// element by one thread, and the slots of a row are summed at the end.
template <int NMAX>
__global__ void __launch_bounds__(RBG * NMAX)
gen_rows_adj_kernel(GenSplit g, const float2* __restrict__ tw, RowArgs a, int rb,
                    const float2* __restrict__ src, const float2* __restrict__ sens,
                    const float* __restrict__ wrow, const float* __restrict__ wcol, float2* out,
                    const float2* operand, float alpha, int ncoils) {
    extern __shared__ float2 sm[];
    const int n = g.n1 * g.n2, P = g.n2 | 1;
    float2* tws = sm;
    load_tw(tws, tw, n);
    const int b = threadIdx.x / g.n2;
    const int cb = RBG / rb;
    const int slot = b / rb, lrow = b - slot * rb;
    float2* Y = sm + n + b * g.n1 * P;
    float2* accs = sm + n + RBG * g.n1 * P;
    float2* acc = accs + b * a.n;
    for (int e = threadIdx.x; e < RBG * a.n; e += blockDim.x) accs[e] = make_float2(0.f, 0.f);
    const int row = blockIdx.x * rb + lrow;
    const float wr = (wrow && row < a.nrows) ? wrow[row] : 1.f;
    __syncthreads();
    for (int c0 = 0; c0 < ncoils; c0 += cb) {
        const int c = c0 + slot, r = opaque(threadIdx.x - b * g.n2);
        const bool live = row < a.nrows && c < ncoils;
        if (live) {
            const float2* sr = src + ((int64_t)c * a.nrows + row) * n;
            int r0 = r + a.off_in;
            if (r0 >= n) r0 -= n;
            dft_any<NMAX, true>(
                g.n1,
                [&](auto& v) {
#pragma unroll
                    for (int m1 = 0; m1 < PP_LEN(v); ++m1) {
                        int s = g.n2 * m1 + r0;
                        if (s >= n) s -= n;
                        v[m1] = sr[s];
                    }
                },
                [&](auto& v) { put_twiddled<true>(v, Y, tws, P, r, 1, 0); });
        }
        __syncthreads();
        if (live && r < g.n1) {
            const float2* sc = sens ? sens + (int64_t)c * a.coil_img_stride + (int64_t)row * a.n : nullptr;
            dft_any<NMAX, true>(
                g.n2, [&](auto& v) { get_row(v, Y, P, r, 1, 0); },
                [&](auto& v) {
                    constexpr int N = PP_LEN(v);
                    if (sc) {
                        float2 s[N];
#pragma unroll
                        for (int k2 = 0; k2 < N; ++k2) {
                            int i = r + g.n1 * k2 + a.off_out;
                            if (i >= n) i -= n;
                            s[k2] = i < a.n ? sc[i] : make_float2(0.f, 0.f);
                        }
#pragma unroll
                        for (int k2 = 0; k2 < N; ++k2) v[k2] = cmulc(s[k2], v[k2]);
                    }
#pragma unroll
                    for (int k2 = 0; k2 < N; ++k2) {
                        int i = r + g.n1 * k2 + a.off_out;
                        if (i >= n) i -= n;
                        if (i < a.n) acc[i] = cadd(acc[i], cscale(v[k2], wcol ? wr * wcol[i] : wr));
                    }
                });
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < rb * a.n; e += blockDim.x) {
        const int lr = e / a.n, i = e - lr * a.n;
        const int orow = blockIdx.x * rb + lr;
        if (orow >= a.nrows) continue;
        float2 v = accs[lr * a.n + i];
        for (int s = 1; s < cb; ++s) v = cadd(v, accs[(s * rb + lr) * a.n + i]);
        const int64_t o = (int64_t)orow * a.n + i;
        v = cscale(v, a.scale);
        if (operand) v = cadd(v, cscale(operand[o], alpha));
        out[o] = v;
    }
}

size_t cols_smem(const GenSplit& g) { return sizeof(float2) * ((size_t)g.n1 * g.n2 + (size_t)y_elems(g) * TXG); }

}  // namespace

GenSplit gen_split_of(int n) {
    GenSplit g;
    if (!gen_split(n, &g.n1, &g.n2)) g.n1 = g.n2 = 0;
    return g;
}

pp_status configure_gen_kernels() {
    const int big = 200 * 1024;
#define PP_ATTR(K) PP_TRY_CUDA(cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, big));
#define PP_ATTRS(NM)                                                                             \
    PP_ATTR((gen_cols_kernel<NM, false, false>)) PP_ATTR((gen_cols_kernel<NM, true, false>))     \
    PP_ATTR((gen_cols_kernel<NM, false, true>))                                                  \
    PP_ATTR(gen_yinv_accum_kernel<NM>) PP_ATTR(gen_cols_roundtrip_kernel<NM>)                    \
    PP_ATTR(gen_rows_fwd_kernel<NM>) PP_ATTR(gen_rows_adj_kernel<NM>)
    PP_ATTRS(16) PP_ATTRS(24) PP_ATTRS(32)
#undef PP_ATTRS
#undef PP_ATTR
    return PP_OK;
}

// ximg: images multiplied into a forward transform's input (batch b takes image
// b % nimgs), or NULL
pp_status launch_gen_cols(const DevFft& f, const ColArgs& a, const float2* src, float2* dst, bool inv,
                          const float2* ximg, int nimgs, cudaStream_t st, bool* done) {
    *done = false;
    const GenSplit g = gen_split_of(a.G);
    if (!g.n1 || (int64_t)a.G * a.ncols >= (1ll << 31)) return PP_OK;   // 32-bit offsets in a batch
    const dim3 grid((a.ncols + TXG - 1) / TXG, a.nbatch);
#define PP_CALL(NM)                                                                               \
    if (ximg)                                                                                     \
        gen_cols_kernel<NM, false, true><<<grid, TXG * g.n2, cols_smem(g), st>>>(g, f.tw, a, src, dst, ximg, nimgs); \
    else if (inv)                                                                                 \
        gen_cols_kernel<NM, true, false><<<grid, TXG * g.n2, cols_smem(g), st>>>(g, f.tw, a, src, dst, nullptr, 1); \
    else                                                                                          \
        gen_cols_kernel<NM, false, false><<<grid, TXG * g.n2, cols_smem(g), st>>>(g, f.tw, a, src, dst, nullptr, 1)
    PP_GEN_CLASS(g.n2, PP_CALL);
#undef PP_CALL
    *done = true;
    return check_gen("gen_cols_kernel");
}

pp_status launch_gen_roundtrip(const DevFft& f, const ColArgs& a, const float* mask_fo,
                               const float2* src, float2* dst, cudaStream_t st, bool* done) {
    *done = false;
    const GenSplit g = gen_split_of(a.G);
    if (!g.n1 || (int64_t)a.G * a.ncols >= (1ll << 31)) return PP_OK;   // 32-bit offsets in a batch
    const dim3 grid((a.ncols + TXG - 1) / TXG, a.nbatch);
#define PP_CALL(NM) \
    gen_cols_roundtrip_kernel<NM><<<grid, TXG * g.n2, cols_smem(g), st>>>(g, f.tw, a, mask_fo, src, dst)
    PP_GEN_CLASS(g.n2, PP_CALL);
#undef PP_CALL
    *done = true;
    return check_gen("gen_cols_roundtrip_kernel");
}

pp_status launch_gen_rows_fwd(const DevFft& f, const RowArgs& a, const float2* x, const float2* sens,
                              const float* wrow, const float* wcol, float2* out, int ncoils,
                              int64_t img_batch_stride, cudaStream_t st, bool* done) {
    *done = false;
    const GenSplit g = gen_split_of(a.G);
    if (!g.n1) return PP_OK;
    const dim3 grid((a.nrows + RBG - 1) / RBG, ncoils);
    const size_t smem = sizeof(float2) * ((size_t)a.G + (size_t)RBG * y_elems(g));
#define PP_CALL(NM)                                                                                \
    gen_rows_fwd_kernel<NM><<<grid, RBG * g.n2, smem, st>>>(g, f.tw, a, x, img_batch_stride, sens, \
                                                            wrow, wcol, out)
    PP_GEN_CLASS(g.n2, PP_CALL);
#undef PP_CALL
    *done = true;
    return check_gen("gen_rows_fwd_kernel");
}

pp_status launch_gen_rows_adj(const DevFft& f, const RowArgs& a, const float2* src, const float2* sens,
                              const float* wrow, const float* wcol, float2* out, const float2* operand,
                              float alpha, int ncoils, cudaStream_t st, bool* done) {
    *done = false;
    const GenSplit g = gen_split_of(a.G);
    if (!g.n1) return PP_OK;
    const size_t smem = sizeof(float2) * ((size_t)a.G + (size_t)RBG * y_elems(g) + (size_t)RBG * a.n);
    if (smem > 200 * 1024) return PP_OK;
    // whole rows per CTA when they fill the GPU, else one row with its coils
    // side by side (152 SMs, several CTAs each)
    int rb = RBG;
    while (rb > 1 && (a.nrows + rb - 1) / rb < 4 * 152 && RBG / rb * 2 <= std::max(1, ncoils)) rb >>= 1;
    const int grid = (a.nrows + rb - 1) / rb;
#define PP_CALL(NM)                                                                              \
    gen_rows_adj_kernel<NM><<<grid, RBG * g.n2, smem, st>>>(g, f.tw, a, rb, src, sens, wrow, wcol, \
                                                            out, operand, alpha, ncoils)
    PP_GEN_CLASS(g.n2, PP_CALL);
#undef PP_CALL
    *done = true;
    return check_gen("gen_rows_adj_kernel");
}

// 3-D normal operator, `chunk` coils at a time: y FFT of S_c x into W, z round
// trip in place, inverse y FFT with the coil sum.  W: chunk * nimg elements.
pp_status gen_cart3d_normal(const Plan& p, const float2* x, float2* out, float scale,
                            const float2* operand, float alpha, float2* W, int chunk, cudaStream_t st,
                            bool* done) {
    *done = false;
    const GenSplit gy = gen_split_of(p.ny), gz = gen_split_of(p.nz);
    if (!gy.n1 || !gz.n1 || p.nimg >= (1ll << 31)) return PP_OK;
    const size_t ysm = cols_smem(gy) + sizeof(float2) * (size_t)p.ny * TXG;
    if (ysm > 200 * 1024 || cols_smem(gz) > 200 * 1024) return PP_OK;
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int64_t n = p.nimg;
    for (int c0 = 0; c0 < p.C; c0 += chunk) {
        const int nc = std::min(chunk, p.C - c0);
        const float2* S = p.sens + (int64_t)c0 * n;
        ColArgs ay{};
        ay.Hin = ay.Hout = ay.G = ny; ay.ncols = nx; ay.nbatch = nc * nz; ay.scale = 1.f;
        ay.in_batch_stride = ay.out_batch_stride = (int64_t)ny * nx;
        ay.mi_cdiv = ay.mo_cdiv = 1;
        bool ok = false;
        PP_TRY(launch_gen_cols(p.fy, ay, S, W, false, x, nz, st, &ok));
        ColArgs az{};
        az.Hin = az.Hout = az.G = nz; az.ncols = ny * nx; az.nbatch = nc; az.scale = 1.f;
        az.in_batch_stride = az.out_batch_stride = n;
        az.mi_cdiv = 1;
        az.mo_q = ny; az.mo_c = 1; az.mo_cdiv = nx;
        PP_TRY(launch_gen_roundtrip(p.fz, az, p.mask_fo, W, W, st, &ok));
        const dim3 grid((nx + TXG - 1) / TXG, nz);
#define PP_CALL(NM)                                                                                \
        gen_yinv_accum_kernel<NM><<<grid, TXG * gy.n2, ysm, st>>>(gy, p.fy.tw, nx, n, nc, W, S, out, \
                                                                  c0 == 0, c0 + nc == p.C, scale,  \
                                                                  operand, alpha)
        PP_GEN_CLASS(gy.n2, PP_CALL);
#undef PP_CALL
        PP_TRY(check_gen("gen_yinv_accum_kernel"));
    }
    *done = true;
    return PP_OK;
}

}  // namespace pp
