// Batched kernels for many independent 2-D Cartesian problems of uneven size
// (one persistent launch per stage over a work list).  Each slice s is its
// own SENSE problem (Sec. 5.1 operator) with its own L_s; the batch shares
// the iteration index k of Algorithm "pfista" (Sec. 3.1).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "pp_batch.h"
#include "pp_fft4.cuh"

namespace pp {

namespace {

__device__ __forceinline__ void load_table_b(float2* dst, const float2* __restrict__ src, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

// Work item (s, col0): columns col0 .. col0 + 2^LGT - 1 of slice s, all coils.
//   out_s = coef * invL_s * sum_c conj(S_c) F_y^H M_fo F_y (S_c x_s) + alpha * operand_s
template <int KM, int LGT>
__global__ void __launch_bounds__(kThreads)
cart2d_batch_normal_kernel(const SliceDesc* __restrict__ descs, const int2* __restrict__ items,
                           int nitems, int ny_max, const float2* __restrict__ x,
                           float2* __restrict__ out, float coef, const float2* __restrict__ operand,
                           float alpha) {
    constexpr int T = 1 << LGT;
    extern __shared__ float2 sm[];
    float2* tws = sm;
    float2* b0 = sm + ny_max;
    float2* b1 = b0 + ny_max * T;
    float* pm = reinterpret_cast<float*>(b1 + ny_max * T);
    int cur = -1;
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const int2 item = items[it];
        const int s = item.x, col0 = item.y;
        const SliceDesc D = descs[s];
        const int ny = D.ny, nx = D.nx;
        if (s != cur) {
            load_table_b(tws, D.tw, ny);
            for (int i = threadIdx.x; i < ny; i += blockDim.x) pm[i] = D.mask_fo[i];
            cur = s;
        }
        const float2* xs = x + D.img_off;
        const int nel = ny * T;
        float2 xr[KM], sr[KM], acc[KM];
#pragma unroll
        for (int k = 0; k < KM; ++k) {
            const int e = threadIdx.x + k * kThreads;
            const int yy = e >> LGT;
            const int col = col0 + (e & (T - 1));
            xr[k] = (e < nel && col < nx) ? xs[(int64_t)yy * nx + col] : make_float2(0.f, 0.f);
            acc[k] = make_float2(0.f, 0.f);
        }
        const int64_t cs = (int64_t)ny * nx;
        for (int c = 0; c < D.C; ++c) {
#pragma unroll
            for (int k = 0; k < KM; ++k) {
                const int e = threadIdx.x + k * kThreads;
                if (e < nel) {
                    const int yy = e >> LGT;
                    const int col = col0 + (e & (T - 1));
                    sr[k] = (col < nx) ? D.sens[c * cs + (int64_t)yy * nx + col] : make_float2(0.f, 0.f);
                    b0[e] = cmul(sr[k], xr[k]);
                }
            }
            __syncthreads();
            float2* r1 = fft_batch<false>(b0, b1, D.fd, T, 1, LGT, tws, nullptr);
            float2* other = (r1 == b0) ? b1 : b0;
            float2* r2 = fft_batch<true>(r1, other, D.fd, T, 1, LGT, tws, pm);
#pragma unroll
            for (int k = 0; k < KM; ++k) {
                const int e = threadIdx.x + k * kThreads;
                if (e < nel) acc[k] = cadd(acc[k], cmulc(sr[k], r2[e]));
            }
            __syncthreads();
        }
        const float sc = coef * D.invL;
        float2* os = out + D.img_off;
        const float2* ops = operand ? operand + D.img_off : nullptr;
#pragma unroll
        for (int k = 0; k < KM; ++k) {
            const int e = threadIdx.x + k * kThreads;
            const int yy = e >> LGT;
            const int col = col0 + (e & (T - 1));
            if (e < nel && col < nx) {
                const int64_t o = (int64_t)yy * nx + col;
                float2 v = cscale(acc[k], sc);
                if (ops) v = cadd(v, cscale(ops[o], alpha));
                os[o] = v;
            }
        }
    }
}

// Segmented FP64 reduction: block b works on segment seg = blk_seg[b], as
// block j = b - seg_first_blk[seg] of that segment's nb blocks.
// partials[b] = (Re<a,b>, Im<a,b>, |b|^2) over the block's share.
__global__ void __launch_bounds__(kThreads)
seg_dot_partial_kernel(const float2* __restrict__ a, const float2* __restrict__ bv,
                       const int64_t* __restrict__ seg_off, const int* __restrict__ blk_seg,
                       const int* __restrict__ seg_first_blk, double* __restrict__ partials) {
    const int seg = blk_seg[blockIdx.x];
    const int j = blockIdx.x - seg_first_blk[seg];
    const int nb = seg_first_blk[seg + 1] - seg_first_blk[seg];
    const int64_t lo = seg_off[seg], hi = seg_off[seg + 1];
    double re = 0.0, im = 0.0, nn = 0.0;
    for (int64_t i = lo + (int64_t)j * blockDim.x + threadIdx.x; i < hi; i += (int64_t)nb * blockDim.x) {
        const float2 y = bv[i];
        if (a) {
            const float2 x = a[i];
            re += (double)x.x * y.x + (double)x.y * y.y;
            im += (double)x.x * y.y - (double)x.y * y.x;
        }
        nn += (double)y.x * y.x + (double)y.y * y.y;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        re += __shfl_down_sync(0xffffffffu, re, off);
        im += __shfl_down_sync(0xffffffffu, im, off);
        nn += __shfl_down_sync(0xffffffffu, nn, off);
    }
    __shared__ double s[3][kThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        s[0][wid] = re;
        s[1][wid] = im;
        s[2][wid] = nn;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double r0 = 0, r1 = 0, r2 = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
            r0 += s[0][i];
            r1 += s[1][i];
            r2 += s[2][i];
        }
        partials[3 * blockIdx.x] = r0;
        partials[3 * blockIdx.x + 1] = r1;
        partials[3 * blockIdx.x + 2] = r2;
    }
}

// One block per segment: out_re[seg*stride], out_nb[seg*stride].
__global__ void seg_dot_final_kernel(const double* __restrict__ partials,
                                     const int* __restrict__ seg_first_blk, double* out_re,
                                     double* out_nb, int stride) {
    __shared__ double s[2][kThreads];
    const int seg = blockIdx.x;
    const int b0 = seg_first_blk[seg], b1 = seg_first_blk[seg + 1];
    double re = 0.0, nn = 0.0;
    for (int i = b0 + threadIdx.x; i < b1; i += blockDim.x) {
        re += partials[3 * i];
        nn += partials[3 * i + 2];
    }
    s[0][threadIdx.x] = re;
    s[1][threadIdx.x] = nn;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            s[0][threadIdx.x] += s[0][threadIdx.x + h];
            s[1][threadIdx.x] += s[1][threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        if (out_re) out_re[seg * stride] = s[0][0];
        if (out_nb) out_nb[seg * stride] = s[1][0];
    }
}

// out = in * factor_seg / sqrt(norm2[seg*stride]) (invert) or * sqrt(...) (not)
__global__ void seg_scale_kernel(const float2* __restrict__ in, float2* __restrict__ out,
                                 const int64_t* __restrict__ seg_off, const int* __restrict__ blk_seg,
                                 const int* __restrict__ seg_first_blk,
                                 const double* __restrict__ norm2, int stride,
                                 const double* __restrict__ factor, int invert) {
    const int seg = blk_seg[blockIdx.x];
    const int j = blockIdx.x - seg_first_blk[seg];
    const int nb = seg_first_blk[seg + 1] - seg_first_blk[seg];
    const int64_t lo = seg_off[seg], hi = seg_off[seg + 1];
    const double nv = norm2 ? sqrt(norm2[seg * stride]) : 1.0;
    const double fs = factor ? factor[seg] : 1.0;
    const double fi = isfinite(nv) ? (nv > 0.0 ? fs / nv : 0.0) : __longlong_as_double(0x7ff8000000000000ll);
    const float f = (float)(invert ? fi : fs * nv);
    for (int64_t i = lo + (int64_t)j * blockDim.x + threadIdx.x; i < hi; i += (int64_t)nb * blockDim.x)
        out[i] = cscale(in[i], f);
}

__device__ __forceinline__ void haar2x2_b(float2& a, float2& b, float2& c, float2& d) {
    const float2 s0 = cadd(a, b), d0 = csub(a, b), s1 = cadd(c, d), d1 = csub(c, d);
    a = cscale(cadd(s0, s1), 0.5f);
    b = cscale(cadd(d0, d1), 0.5f);
    c = cscale(csub(s0, s1), 0.5f);
    d = cscale(csub(d0, d1), 0.5f);
}

__device__ __forceinline__ float2 soft_b(float2 v, float lam) {
    const float m2 = v.x * v.x + v.y * v.y;
    // |v| <= lambda -> 0 (also v = 0, so no 0 * inf); a NaN fails the test and
    // stays NaN instead of being thresholded to 0
    if (m2 <= lam * lam) return make_float2(0.f, 0.f);
    return cscale(v, 1.f - lam * rsqrtf(m2));
}

// Four adjacent lanes hold one 4 x 4 tile, lane 2 qy + qx its 2 x 2 block (qx, qy):
// level 1 of the Haar transform in registers, level 2 on the four approximation
// coefficients by shuffles, in the operation order of haar2x2_b.  Its own inverse.
__device__ __forceinline__ float2 shfl2_b(float2 v, int m) {
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}
__device__ __forceinline__ float2 haar_level2(float2 a, int qx, int qy) {
    const float2 p = shfl2_b(a, 1);
    const float2 t = qx ? csub(p, a) : cadd(a, p);
    const float2 r = shfl2_b(t, 2);
    return cscale(qy ? csub(r, t) : cadd(t, r), 0.5f);
}
__device__ __forceinline__ void haar_quad(float2* v, int qx, int qy) {
    haar2x2_b(v[0], v[1], v[2], v[3]);
    v[0] = haar_level2(v[0], qx, qy);
}
__device__ __forceinline__ void haar_quad_inv(float2* v, int qx, int qy) {
    v[0] = haar_level2(v[0], qx, qy);
    haar2x2_b(v[0], v[1], v[2], v[3]);
}
// The 2 x 2 block as two 16-byte accesses (its columns start at even elements of
// 16-byte aligned arrays of even pitch).
__device__ __forceinline__ void load_quad(float2* v, const float2* p, int64_t pitch) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + pitch);
    v[0] = make_float2(a.x, a.y);
    v[1] = make_float2(a.z, a.w);
    v[2] = make_float2(b.x, b.y);
    v[3] = make_float2(b.z, b.w);
}
__device__ __forceinline__ void store_quad(const float2* v, float2* p, int64_t pitch) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    *reinterpret_cast<float4*>(p + pitch) = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
}

// Batched fused prox + momentum over 4x4 tiles, four lanes a tile (one thread a
// tile left 128 CTAs of one long load chain for eight 256 x 256 slices: 12.6 us);
// block -> slice map as above (segments count tiles).  Statistics are summed over
// the whole batch.
__global__ void __launch_bounds__(kThreads)
batch_prox_fista_kernel(const SliceDesc* __restrict__ descs, const int64_t* __restrict__ tile_off,
                        const int* __restrict__ blk_seg, const int* __restrict__ seg_first_blk,
                        float lam, float gamma, float beta, float2* __restrict__ z,
                        const float2* __restrict__ u, float2* __restrict__ y,
                        float2* __restrict__ w_out, const float2* __restrict__ ref,
                        double* __restrict__ hist) {
    const int s = blk_seg[blockIdx.x];
    const int j = blockIdx.x - seg_first_blk[s];
    const SliceDesc D = descs[s];
    const int64_t t = (int64_t)j * (blockDim.x / 4) + (threadIdx.x >> 2);
    const int64_t ntl = tile_off[s + 1] - tile_off[s];
    const int qx = threadIdx.x & 1, qy = (threadIdx.x >> 1) & 1;
    const bool live = t < ntl;
    double dd = 0.0, yy = 0.0, rr = 0.0;
    const int ntx = D.nx / 4;
    const int64_t ty = live ? t / ntx : 0, tx = live ? t - ty * ntx : 0;
    const int64_t o = D.img_off + (ty * 4 + 2 * qy) * D.nx + tx * 4 + 2 * qx;
    float2 v[4], uv[4], yo[4];
    load_quad(v, z + o, D.nx);
    load_quad(uv, u + o, D.nx);
    load_quad(yo, y + o, D.nx);
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = make_float2(v[i].x - gamma * uv[i].x, v[i].y - gamma * uv[i].y);
    if (w_out && live) store_quad(v, w_out + o, D.nx);
    haar_quad(v, qx, qy);
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = soft_b(v[i], lam);
    haar_quad_inv(v, qx, qy);
    if (live) {
        float2 zn[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 df = csub(v[i], yo[i]);
            zn[i] = make_float2(v[i].x + beta * df.x, v[i].y + beta * df.y);
            if (hist) {   // FP64 arithmetic is slow on this part: only when asked for
                dd += (double)df.x * df.x + (double)df.y * df.y;
                yy += (double)v[i].x * v[i].x + (double)v[i].y * v[i].y;
            }
            if (ref) {
                const float2 rv = ref[o + (int64_t)(i >> 1) * D.nx + (i & 1)];
                const double ex = (double)v[i].x - rv.x, ey = (double)v[i].y - rv.y;
                rr += ex * ex + ey * ey;
            }
        }
        store_quad(v, y + o, D.nx);
        store_quad(zn, z + o, D.nx);
    }
    if (hist) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            dd += __shfl_down_sync(0xffffffffu, dd, off);
            yy += __shfl_down_sync(0xffffffffu, yy, off);
            rr += __shfl_down_sync(0xffffffffu, rr, off);
        }
        __shared__ double sd[kThreads / 32], sy[kThreads / 32], sr[kThreads / 32];
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        if (lane == 0) {
            sd[wid] = dd;
            sy[wid] = yy;
            sr[wid] = rr;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double a = 0.0, b = 0.0, c = 0.0;
            for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
                a += sd[i];
                b += sy[i];
                c += sr[i];
            }
            atomicAdd(&hist[0], a);
            atomicAdd(&hist[1], b);
            atomicAdd(&hist[2], c);
        }
    }
}

// Reverse pass of one unrolled iteration at the prox (per 4x4 tile):
//   ybar_{k+1} = Ybar + (1 + beta) Zbar          (adjoint of y_{k+1})
//   Ybar      <- -beta Zbar                      (partial adjoint of y_k)
//   wbar       = W^T J_s^T W ybar_{k+1},  J_s the soft threshold's Jacobian
//                at the coefficients W w_k
//   lam_bar   += sum Re(conj(W ybar_{k+1}) . (-v/|v|)) over |v| > lambda
__global__ void __launch_bounds__(kThreads)
batch_prox_vjp_kernel(const SliceDesc* __restrict__ descs, const int64_t* __restrict__ tile_off,
                      const int* __restrict__ blk_seg, const int* __restrict__ seg_first_blk,
                      float lam, float beta, const float2* __restrict__ w, float2* __restrict__ Ybar,
                      const float2* __restrict__ Zbar, float2* __restrict__ wbar,
                      double* __restrict__ lam_bar) {
    const int s = blk_seg[blockIdx.x];
    const int j = blockIdx.x - seg_first_blk[s];
    const SliceDesc D = descs[s];
    const int64_t t = (int64_t)j * (blockDim.x / 4) + (threadIdx.x >> 2);
    const int64_t ntl = tile_off[s + 1] - tile_off[s];
    const int qx = threadIdx.x & 1, qy = (threadIdx.x >> 1) & 1;
    const bool live = t < ntl;
    double lb = 0.0;
    const int ntx = D.nx / 4;
    const int64_t ty = live ? t / ntx : 0, tx = live ? t - ty * ntx : 0;
    const int64_t o = D.img_off + (ty * 4 + 2 * qy) * D.nx + tx * 4 + 2 * qx;
    float2 cw[4], cy[4], zb[4];
    load_quad(zb, Zbar + o, D.nx);
    load_quad(cy, Ybar + o, D.nx);
    load_quad(cw, w + o, D.nx);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        cy[i] = make_float2(cy[i].x + (1.f + beta) * zb[i].x, cy[i].y + (1.f + beta) * zb[i].y);
        zb[i] = make_float2(-beta * zb[i].x, -beta * zb[i].y);
    }
    if (live) store_quad(zb, Ybar + o, D.nx);
    haar_quad(cw, qx, qy);
    haar_quad(cy, qx, qy);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 v = cw[i], g = cy[i];
        const float m2 = v.x * v.x + v.y * v.y;
        if (m2 > lam * lam) {
            const float rm = rsqrtf(m2);
            const float hx = v.x * rm, hy = v.y * rm;          // v / |v|
            const float q = lam * rm;                            // lambda / |v|
            const float proj = hx * g.x + hy * g.y;              // Re(conj(vhat) g)
            cy[i] = make_float2((1.f - q) * g.x + q * hx * proj, (1.f - q) * g.y + q * hy * proj);
            if (live) lb -= (double)proj;
        } else {
            cy[i] = make_float2(0.f, 0.f);
        }
    }
    haar_quad_inv(cy, qx, qy);
    if (live) store_quad(cy, wbar + o, D.nx);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) lb += __shfl_down_sync(0xffffffffu, lb, off);
    __shared__ double sl[kThreads / 32];
    if ((threadIdx.x & 31) == 0) sl[threadIdx.x >> 5] = lb;
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) a += sl[i];
        atomicAdd(lam_bar, a);
    }
}

// One pass over the d + 2 vectors, the gradient and the two accumulators where
// d + 1 dot products and two linear combinations read them three times over:
//   partials[block][i] = Re<v_i, g> over the block's share,
//   Zbar = wbar - sum_i c_i v_{i+1},  ahb_bar += sum_i c_i v_i.
template <int D>
__global__ void __launch_bounds__(kThreads) rev_combine_kernel(const RevCombine r) {
    double dot[D + 1];
#pragma unroll
    for (int i = 0; i <= D; ++i) dot[i] = 0.0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < r.n; e += (int64_t)gridDim.x * blockDim.x) {
        float2 v[D + 2];
        v[0] = r.wbar[e];
#pragma unroll
        for (int i = 1; i <= D + 1; ++i) v[i] = r.v[(i - 1) * r.n + e];
        const float2 g = r.g[e];
        float2 z = v[0], a = r.ahb_bar[e];
#pragma unroll
        for (int i = 0; i <= D; ++i) {
            dot[i] += (double)v[i].x * g.x + (double)v[i].y * g.y;
            z.x -= r.c[i] * v[i + 1].x;
            z.y -= r.c[i] * v[i + 1].y;
            a.x += r.c[i] * v[i].x;
            a.y += r.c[i] * v[i].y;
        }
        r.Zbar[e] = z;
        r.ahb_bar[e] = a;
    }
    __shared__ double s[D + 1][kThreads / 32];
#pragma unroll
    for (int i = 0; i <= D; ++i) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) dot[i] += __shfl_down_sync(0xffffffffu, dot[i], off);
        if ((threadIdx.x & 31) == 0) s[i][threadIdx.x >> 5] = dot[i];
    }
    __syncthreads();
    if (threadIdx.x <= D) {
        double a = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) a += s[threadIdx.x][w];
        r.partials[blockIdx.x * (D + 1) + threadIdx.x] = a;
    }
}

// dots[i] = sum of the blocks' partials, one warp each, in a fixed order
__global__ void rev_dots_kernel(const double* __restrict__ partials, int nblocks, int nd,
                                double* __restrict__ dots) {
    const int i = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double a = 0.0;
    for (int b = lane; b < nblocks; b += 32) a += partials[b * nd + i];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) a += __shfl_down_sync(0xffffffffu, a, off);
    if (lane == 0) dots[i] = a;
}

}  // namespace

extern thread_local int64_t g_launches;
extern thread_local Profiler* g_profiler;

static pp_status check_launch_b(const char* what) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_status(e, what);
    ++g_launches;
    if (g_profiler) g_profiler->mark(what);
    return PP_OK;
}

size_t batch_normal_smem(int ny_max, int lgt) {
    return sizeof(float2) * (size_t)(ny_max + 2 * ny_max * (1 << lgt)) + sizeof(float) * ny_max;
}

template <int KM, int LGT>
static void* batch_kernel_ptr() {
    return reinterpret_cast<void*>(cart2d_batch_normal_kernel<KM, LGT>);
}

// kernel pointer for (km, lgt); nullptr when not instantiated
void* batch_normal_fn(int km, int lgt) {
#define PP_B(KM_, L_) if (km == KM_ && lgt == L_) return batch_kernel_ptr<KM_, L_>();
    PP_B(4, 2) PP_B(8, 2)
    PP_B(4, 3) PP_B(8, 3) PP_B(12, 3)
    PP_B(4, 4) PP_B(8, 4) PP_B(12, 4) PP_B(16, 4)
#undef PP_B
    return nullptr;
}

pp_status configure_batch_kernels() {
    const int big = 200 * 1024;
    const int kms[] = {4, 8, 12, 16};
    for (int lgt = 2; lgt <= 4; ++lgt)
        for (int km : kms) {
            void* f = batch_normal_fn(km, lgt);
            if (f) PP_TRY_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, big));
        }
    return PP_OK;
}

pp_status launch_batch_chain(const BatchDev& b, const float2* x, const CartChain& ch, cudaStream_t st) {
    // one launch per length; each after the first may start while its
    // predecessor's last CTAs run (same input, other slices)
    bool first = true;
    const std::vector<CartGroup>& groups = ch.J > 1 ? b.groups : b.one;
    int all = 0;
    for (const CartGroup& g : groups) all += g.nitems;
    for (const CartGroup& g : groups) {
        CartLaunch L;
        L.descs = b.descs;
        L.items = g.items;
        L.nitems = g.nitems;
        L.W = g.W;
        L.max_coils = g.max_coils;
        L.lean = g.lean;
        L.beside = all - g.nitems;
        L.pdl = L.follows = !first;
        PP_TRY(launch_cart_cols(g.n, L, x, ch, st));
        first = false;
    }
    return PP_OK;
}

pp_status launch_batch_normal(const BatchDev& b, const float2* x, float2* out, float coef,
                              const float2* operand, float alpha, cudaStream_t st) {
    if (b.cols > 0) {
        CartChain ch;
        ch.sc[0] = coef;
        ch.al[0] = alpha;
        ch.ext = operand;
        ch.out = out;
        return launch_batch_chain(b, x, ch, st);
    }
    void* fn = batch_normal_fn(b.km, b.lgt);
    if (!fn) {
        set_error("no batched kernel for km=%d lgt=%d", b.km, b.lgt);
        return PP_ERR_UNSUPPORTED;
    }
    void* args[] = {(void*)&b.descs, (void*)&b.items, (void*)&b.nitems, (void*)&b.ny_max,
                    (void*)&x, (void*)&out, (void*)&coef, (void*)&operand, (void*)&alpha};
    PP_TRY_CUDA(cudaLaunchKernel(fn, dim3(b.grid), dim3(kThreads), args,
                                 batch_normal_smem(b.ny_max, b.lgt), st));
    return check_launch_b("cart2d_batch_normal_kernel");
}

pp_status launch_seg_dot(const float2* a, const float2* bv, const Segments& sg, double* partials,
                         double* out_re, double* out_nb, int stride, cudaStream_t st) {
    seg_dot_partial_kernel<<<sg.nblocks, kThreads, 0, st>>>(a, bv, sg.off, sg.blk_seg,
                                                             sg.seg_first_blk, partials);
    PP_TRY(check_launch_b("seg_dot_partial_kernel"));
    seg_dot_final_kernel<<<sg.nseg, kThreads, 0, st>>>(partials, sg.seg_first_blk, out_re, out_nb,
                                                        stride);
    return check_launch_b("seg_dot_final_kernel");
}

pp_status launch_seg_scale(const float2* in, float2* out, const Segments& sg, const double* norm2,
                           int stride, const double* factor, int invert, cudaStream_t st) {
    seg_scale_kernel<<<sg.nblocks, kThreads, 0, st>>>(in, out, sg.off, sg.blk_seg, sg.seg_first_blk,
                                                       norm2, stride, factor, invert);
    return check_launch_b("seg_scale_kernel");
}

pp_status launch_batch_prox_fista(const BatchDev& b, float lam, float gamma, float beta,
                                  float2* z, const float2* u, float2* y, float2* w_out, const float2* ref,
                                  double* hist, cudaStream_t st) {
    batch_prox_fista_kernel<<<b.tiles.nblocks, kTileThreads, 0, st>>>(
        b.descs, b.tiles.off, b.tiles.blk_seg, b.tiles.seg_first_blk, lam, gamma, beta, z, u, y, w_out,
        ref, hist);
    return check_launch_b("batch_prox_fista_kernel");
}

pp_status launch_batch_prox_vjp(const BatchDev& b, float lam, float beta, const float2* w,
                                float2* Ybar, const float2* Zbar, float2* wbar, double* lam_bar,
                                cudaStream_t st) {
    batch_prox_vjp_kernel<<<b.tiles.nblocks, kTileThreads, 0, st>>>(
        b.descs, b.tiles.off, b.tiles.blk_seg, b.tiles.seg_first_blk, lam, beta, w, Ybar, Zbar, wbar,
        lam_bar);
    return check_launch_b("batch_prox_vjp_kernel");
}

pp_status launch_rev_combine(const RevCombine& r, double* dots, cudaStream_t st) {
    const int nblk = (int)std::max<int64_t>(1, std::min<int64_t>(kRevBlocks, (r.n + kThreads - 1) / kThreads));
    switch (r.d) {
#define PP_REV(D) case D: rev_combine_kernel<D><<<nblk, kThreads, 0, st>>>(r); break;
        PP_REV(0) PP_REV(1) PP_REV(2) PP_REV(3) PP_REV(4) PP_REV(5) PP_REV(6) PP_REV(7) PP_REV(8) PP_REV(9)
        PP_REV(10)
#undef PP_REV
        default:
            set_error("unrolled solve: degree %d", r.d);
            return PP_ERR_UNSUPPORTED;
    }
    PP_TRY(check_launch_b("rev_combine_kernel"));
    rev_dots_kernel<<<1, 32 * (r.d + 1), 0, st>>>(r.partials, nblk, r.d + 1, dots);
    return check_launch_b("rev_dots_kernel");
}

}  // namespace pp
