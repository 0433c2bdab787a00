// Daubechies-4 l1 prox (Eq. "proxdef" with W the Daubechies-4 wavelet, the
// transform of the paper's experiments, Sec. 5.1 and Sec. 5.2), 2-D.
//
// W: the four-coefficient orthonormal Daubechies filter
//   h = ((1 + s3), (3 + s3), (3 - s3), (1 - s3)) / (4 sqrt 2),  s3 = sqrt 3,
//   g[k] = (-1)^k h[3 - k],
// periodic boundary, separable, Mallat layout: at level l the band of
// ny >> (l-1) rows and nx >> (l-1) columns is transformed along x (rows),
// then along y (columns), approximation first:
//   a[i] = sum_k h[k] v[(2i + k) mod n],  d[i] = sum_k g[k] v[(2i + k) mod n].
// The inverse is the transpose: v[2m] = h0 a[m] + h2 a[m-1] + g0 d[m] + g2 d[m-1],
// v[2m+1] = h1 a[m] + h3 a[m-1] + g1 d[m] + g3 d[m-1] (indices mod n/2).
//
// Unlike the 2-level Haar (tile-local), every level couples neighbouring
// tiles.  Images that fit the shared memory of one thread-block cluster run in
// one launch (db4_cluster_kernel); larger ones as one pass per level and
// direction: a CTA owns whole rows (or 8 whole columns) of the band, stages
// them in shared memory and writes its outputs back in place.  The soft threshold is applied when
// a coefficient becomes final (column passes); the FISTA step w = z - gamma u
// is fused into the first pass, the momentum update and the FP64 statistics
// into the last.
#include <cuda_runtime.h>
#include <cooperative_groups.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "pp_fft4.cuh"
#include "pp_internal.h"

namespace cg = cooperative_groups;

namespace pp {
namespace {

constexpr int MAXN = 512;   // longest row / column
constexpr int CW = 8;       // columns per CTA in the column passes
constexpr int kDb4Threads = 512;   // threads of a CTA of the cluster form

struct Db4 {
    float h[4], g[4];
};

Db4 db4_filter() {
    const double s3 = sqrt(3.0), r = 1.0 / (4.0 * sqrt(2.0));
    const double h[4] = {(1 + s3) * r, (3 + s3) * r, (3 - s3) * r, (1 - s3) * r};
    Db4 f;
    for (int k = 0; k < 4; ++k) {
        f.h[k] = (float)h[k];
        f.g[k] = (float)((k & 1) ? -h[3 - k] : h[3 - k]);
    }
    return f;
}

__device__ __forceinline__ float2 soft4(float2 v, float lam) {
    const float m2 = v.x * v.x + v.y * v.y;
    // |v| <= lambda -> 0 (also v = 0, so no 0 * inf); a NaN fails the test and
    // stays NaN instead of being thresholded to 0
    if (m2 <= lam * lam) return make_float2(0.f, 0.f);
    return cscale(v, 1.f - lam * rsqrtf(m2));
}

__device__ __forceinline__ float2 fma2(float c, float2 v, float2 acc) {
    return make_float2(fmaf(c, v.x, acc.x), fmaf(c, v.y, acc.y));
}

// FISTA epilogue arguments of the last inverse pass (z, y updated in place).
struct Epi {
    float2* z;
    float2* y;
    const float2* ref;
    double* hist;
    float beta;
};

// Block-level FP64 sums of (dd, yy, rr) added to hist[0..2].
__device__ __forceinline__ void hist_add(double dd, double yy, double rr, double* hist) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        dd += __shfl_down_sync(0xffffffffu, dd, off);
        yy += __shfl_down_sync(0xffffffffu, yy, off);
        rr += __shfl_down_sync(0xffffffffu, rr, off);
    }
    __shared__ double s[3][kDb4Threads / 32];   // the widest block that calls this
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        s[0][wid] = dd;
        s[1][wid] = yy;
        s[2][wid] = rr;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0, c = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
            a += s[0][i];
            b += s[1][i];
            c += s[2][i];
        }
        atomicAdd(&hist[0], a);
        atomicAdd(&hist[1], b);
        atomicAdd(&hist[2], c);
    }
}

// Row pass over the band [0, h) x [0, w) of an image with row pitch nx.
// Forward: reads src (or z - gamma u when u != NULL), writes [a | d] to dst.
// Inverse: reads [a | d] from src, writes v to dst, or, with EPI, runs the
// FISTA epilogue on v.  grid (h), block kThreads; src may equal dst.
template <bool INV, bool EPI>
__global__ void __launch_bounds__(kThreads)
db4_rows_kernel(Db4 f, int w, int nx, const float2* src, const float2* __restrict__ u, float gamma,
                float2* dst, Epi e) {
    __shared__ float2 s[MAXN];
    pdl_trigger();
    pdl_wait();
    const int64_t row = (int64_t)blockIdx.x * nx;
    for (int i = threadIdx.x; i < w; i += blockDim.x) {
        float2 v = src[row + i];
        if (u) {
            const float2 q = u[row + i];
            v = make_float2(v.x - gamma * q.x, v.y - gamma * q.y);
        }
        s[i] = v;
    }
    __syncthreads();
    const int hw = w >> 1;
    if (!INV) {
        for (int i = threadIdx.x; i < hw; i += blockDim.x) {
            float2 a = make_float2(0.f, 0.f), d = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                int j = 2 * i + k;
                if (j >= w) j -= w;
                a = fma2(f.h[k], s[j], a);
                d = fma2(f.g[k], s[j], d);
            }
            dst[row + i] = a;
            dst[row + hw + i] = d;
        }
        return;
    }
    double dd = 0.0, yy = 0.0, rr = 0.0;
    for (int j = threadIdx.x; j < w; j += blockDim.x) {
        const int m = j >> 1, par = j & 1, m1 = m == 0 ? hw - 1 : m - 1;
        float2 v = make_float2(0.f, 0.f);
        v = fma2(f.h[par], s[m], v);
        v = fma2(f.h[par + 2], s[m1], v);
        v = fma2(f.g[par], s[hw + m], v);
        v = fma2(f.g[par + 2], s[hw + m1], v);
        if (!EPI) {
            dst[row + j] = v;
        } else {
            const float2 yo = e.y[row + j];
            const float2 df = csub(v, yo);
            e.z[row + j] = make_float2(v.x + e.beta * df.x, v.y + e.beta * df.y);
            e.y[row + j] = v;
            if (e.hist) {
                dd += (double)df.x * df.x + (double)df.y * df.y;
                yy += (double)v.x * v.x + (double)v.y * v.y;
                if (e.ref) {
                    const float2 r = e.ref[row + j];
                    const double ex = (double)v.x - r.x, ey = (double)v.y - r.y;
                    rr += ex * ex + ey * ey;
                }
            }
        }
    }
    if (EPI && e.hist) hist_add(dd, yy, rr, e.hist);
}

// Column pass over the band [0, h) x [0, w): CTA b owns columns
// 8b .. 8b+7 (those below w).  Forward writes [a ; d] down each column and
// soft-thresholds the coefficients that are final: every d, and a when the
// level is the last or the column holds row details (col >= w/2).
// grid (ceil(w / 8)), block kThreads; in place.
template <bool INV>
__global__ void __launch_bounds__(kThreads)
db4_cols_kernel(Db4 f, int h, int w, int nx, float lam, int last, float2* v) {
    __shared__ float2 s[MAXN * CW];
    pdl_trigger();
    pdl_wait();
    const int col0 = blockIdx.x * CW;
    for (int e = threadIdx.x; e < h * CW; e += blockDim.x) {
        const int r = e / CW, c = e % CW;
        if (col0 + c < w) s[e] = v[(int64_t)r * nx + col0 + c];
    }
    __syncthreads();
    const int hh = h >> 1;
    if (!INV) {
        for (int e = threadIdx.x; e < hh * CW; e += blockDim.x) {
            const int i = e / CW, c = e % CW, col = col0 + c;
            if (col >= w) continue;
            float2 a = make_float2(0.f, 0.f), d = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                int j = 2 * i + k;
                if (j >= h) j -= h;
                a = fma2(f.h[k], s[j * CW + c], a);
                d = fma2(f.g[k], s[j * CW + c], d);
            }
            if (last || col >= (w >> 1)) a = soft4(a, lam);
            v[(int64_t)i * nx + col] = a;
            v[(int64_t)(hh + i) * nx + col] = soft4(d, lam);
        }
        return;
    }
    for (int e = threadIdx.x; e < h * CW; e += blockDim.x) {
        const int j = e / CW, c = e % CW, col = col0 + c;
        if (col >= w) continue;
        const int m = j >> 1, par = j & 1, m1 = m == 0 ? hh - 1 : m - 1;
        float2 x = make_float2(0.f, 0.f);
        x = fma2(f.h[par], s[m * CW + c], x);
        x = fma2(f.h[par + 2], s[m1 * CW + c], x);
        x = fma2(f.g[par], s[(hh + m) * CW + c], x);
        x = fma2(f.g[par + 2], s[(hh + m1) * CW + c], x);
        v[(int64_t)j * nx + col] = x;
    }
}

// The whole prox in one launch of one cluster.  CTA q owns a slab of rows, a
// multiple of 2^levels, in two shared buffers; the x passes are local, and a y
// pass needs two rows of the next slab (forward) or the last approximation and
// detail row of the previous one (inverse), which their owner pushes into this
// CTA's halo rows through distributed shared memory before one cluster barrier a
// level and direction.  Halo rows are used once, so nothing waits for readers.
// B0 holds the band in Mallat order (a rows above d rows, [a | d] along x), B1 the
// band between the two passes of a level.  Same arithmetic, in the same order, as
// the passes above.  Bound by latency: 2 levels + 1 cluster barriers and
// 2 * levels passes over a slab in place of 4 * levels kernels of 2 to 3 us each
// (40 iterations at 128 x 128 and 8 coils, d = 3, 2 levels: 1000 -> 701 us).

struct Db4Cluster {
    Db4 f;
    int nx, ny, levels, R;
    float lam, gamma;
    const float2* in;
    const float2* u;     // NULL: the input is `in` alone
    float2* out;         // NULL: the FISTA epilogue
    Epi e;
};

__global__ void __launch_bounds__(kDb4Threads) db4_cluster_kernel(const Db4Cluster p) {
    extern __shared__ float2 sm[];
    cg::cluster_group cluster = cg::this_cluster();
    const int nx = p.nx, L = p.levels, R = p.R, q = (int)cluster.block_rank();
    const int units = p.ny >> L;
    const int r0 = (int)((int64_t)units * q / R) << L, rows = ((int)((int64_t)units * (q + 1) / R) << L) - r0;
    const int slab = ((units + R - 1) / R) << L;   // rows that every CTA's buffers hold
    float2* B0 = sm;
    float2* B1 = B0 + slab * nx;
    float2* HF = B1 + slab * nx;          // [level][2][nx]: the next slab's first rows
    float2* HI = HF + 2 * L * nx;         // [level][2][nx]: the previous slab's last a and d row
    pdl_trigger();
    cluster_arrive_relaxed();             // every CTA of the cluster runs before the first push
    pdl_wait();
    const int64_t g0 = (int64_t)r0 * nx;
    for (int e = threadIdx.x; e < rows * nx; e += blockDim.x) {
        float2 v = p.in[g0 + e];
        if (p.u) {
            const float2 s = p.u[g0 + e];
            v = make_float2(v.x - p.gamma * s.x, v.y - p.gamma * s.y);
        }
        B0[e] = v;
    }
    cluster_wait_acquire();
    float2* const next = cluster.map_shared_rank(sm, (q + 1) % R);
    float2* const prev = cluster.map_shared_rank(sm, (q + R - 1) % R);
    const int oHF = (int)(HF - sm), oHI = (int)(HI - sm);
    __syncthreads();
    for (int l = 0; l < L; ++l) {
        const int h = rows >> l, w = nx >> l, hw = w >> 1, hh = h >> 1;
        for (int e = threadIdx.x; e < h * hw; e += blockDim.x) {
            const int r = e / hw, i = e - r * hw;
            const float2* s = B0 + r * nx;
            float2 a = make_float2(0.f, 0.f), d = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                int j = 2 * i + k;
                if (j >= w) j -= w;
                a = fma2(p.f.h[k], s[j], a);
                d = fma2(p.f.g[k], s[j], d);
            }
            B1[r * nx + i] = a;
            B1[r * nx + hw + i] = d;
            if (r < 2) {
                prev[oHF + (2 * l + r) * nx + i] = a;
                prev[oHF + (2 * l + r) * nx + hw + i] = d;
            }
        }
        cluster_arrive_release();
        cluster_wait_acquire();
        const bool last = l == L - 1;
        for (int e = threadIdx.x; e < hh * w; e += blockDim.x) {
            const int i = e / w, c = e - i * w;
            float2 a = make_float2(0.f, 0.f), d = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = 2 * i + k;
                const float2 s = j < h ? B1[j * nx + c] : HF[(2 * l + j - h) * nx + c];
                a = fma2(p.f.h[k], s, a);
                d = fma2(p.f.g[k], s, d);
            }
            if (last || c >= hw) a = soft4(a, p.lam);
            B0[i * nx + c] = a;
            B0[(hh + i) * nx + c] = soft4(d, p.lam);
        }
        __syncthreads();
    }
    double dd = 0.0, yy = 0.0, rr = 0.0;
    for (int l = L - 1; l >= 0; --l) {
        const int h = rows >> l, w = nx >> l, hw = w >> 1, hh = h >> 1;
        for (int c = threadIdx.x; c < w; c += blockDim.x) {
            next[oHI + (2 * l) * nx + c] = B0[(hh - 1) * nx + c];
            next[oHI + (2 * l + 1) * nx + c] = B0[(h - 1) * nx + c];
        }
        cluster_arrive_release();
        cluster_wait_acquire();
        for (int e = threadIdx.x; e < h * w; e += blockDim.x) {
            const int j = e / w, c = e - j * w, m = j >> 1, par = j & 1;
            const float2 a1 = m ? B0[(m - 1) * nx + c] : HI[(2 * l) * nx + c];
            const float2 d1 = m ? B0[(hh + m - 1) * nx + c] : HI[(2 * l + 1) * nx + c];
            float2 x = make_float2(0.f, 0.f);
            x = fma2(par ? p.f.h[1] : p.f.h[0], B0[m * nx + c], x);
            x = fma2(par ? p.f.h[3] : p.f.h[2], a1, x);
            x = fma2(par ? p.f.g[1] : p.f.g[0], B0[(hh + m) * nx + c], x);
            x = fma2(par ? p.f.g[3] : p.f.g[2], d1, x);
            B1[j * nx + c] = x;
        }
        __syncthreads();
        for (int e = threadIdx.x; e < h * w; e += blockDim.x) {
            const int r = e / w, j = e - r * w;
            const float2* s = B1 + r * nx;
            const int m = j >> 1, par = j & 1, m1 = m == 0 ? hw - 1 : m - 1;
            const int64_t o = g0 + (int64_t)r * nx + j;
            float2 yo = make_float2(0.f, 0.f);
            if (l == 0 && !p.out) yo = p.e.y[o];
            float2 v = make_float2(0.f, 0.f);
            v = fma2(par ? p.f.h[1] : p.f.h[0], s[m], v);
            v = fma2(par ? p.f.h[3] : p.f.h[2], s[m1], v);
            v = fma2(par ? p.f.g[1] : p.f.g[0], s[hw + m], v);
            v = fma2(par ? p.f.g[3] : p.f.g[2], s[hw + m1], v);
            if (l > 0) {
                B0[r * nx + j] = v;
            } else if (p.out) {
                p.out[o] = v;
            } else {
                const float2 df = csub(v, yo);
                p.e.z[o] = make_float2(v.x + p.e.beta * df.x, v.y + p.e.beta * df.y);
                p.e.y[o] = v;
                if (p.e.hist) {
                    dd += (double)df.x * df.x + (double)df.y * df.y;
                    yy += (double)v.x * v.x + (double)v.y * v.y;
                    if (p.e.ref) {
                        const float2 t = p.e.ref[o];
                        const double ex = (double)v.x - t.x, ey = (double)v.y - t.y;
                        rr += ex * ex + ey * ey;
                    }
                }
            }
        }
        __syncthreads();
    }
    if (!p.out && p.e.hist) hist_add(dd, yy, rr, p.e.hist);
}

// Cluster size for an image, 0 when it does not fit: 8 CTAs, or 16 (beyond the
// portable size) for images of more than 128 x 128 where the device takes them.
size_t db4_cluster_smem(int nx, int ny, int levels, int R) {
    const int units = ny >> levels, slab = ((units + R - 1) / R) << levels;
    return sizeof(float2) * ((size_t)2 * slab * nx + (size_t)4 * levels * nx);
}
constexpr int kDb4Smem = 220 * 1024;
// Largest cluster that the current device takes: 16, 8 (the portable size), or 0
// when the kernel's attributes are refused.
int db4_largest_cluster() {
    static PerDevice largest;
    return largest.get(current_device(), [] {
        cudaError_t e = cudaFuncSetAttribute(db4_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDb4Smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(db4_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cudaGetLastError();
        if (e != cudaSuccess) return 0;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 16;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(16);
        cfg.blockDim = dim3(kDb4Threads);
        cfg.dynamicSmemBytes = kDb4Smem;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        e = cudaOccupancyMaxActiveClusters(&n, db4_cluster_kernel, &cfg);
        cudaGetLastError();
        return e == cudaSuccess && n > 0 ? 16 : 8;
    });
}
int db4_cluster_size(int nx, int ny, int levels) {
    const int largest = db4_largest_cluster();
    if (!largest) return 0;
    const int units = ny >> levels;
    int R = (int64_t)nx * ny > 128 * 128 ? largest : 8;
    while (R > units) R >>= 1;
    return db4_cluster_smem(nx, ny, levels, R) <= (size_t)kDb4Smem ? R : 0;
}

pp_status check_db4(const char* what) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_status(e, what);
    ++g_launches;
    if (g_profiler) g_profiler->mark(what);
    return PP_OK;
}

// The whole prox: forward levels 1..L, thresholds, inverse levels L..1.
// First pass reads `in` (minus gamma u when u != NULL) and writes `coef`;
// the rest runs in place on `coef`; the last pass writes `out` or, with
// `epi`, the FISTA epilogue.
pp_status db4_prox(int nx, int ny, int levels, float lambda, const float2* in, const float2* u,
                   float gamma, float2* coef, float2* out, const Epi* epi, bool pdl,
                   cudaStream_t st) {
    const Db4 f = db4_filter();
    const Epi none{nullptr, nullptr, nullptr, nullptr, 0.f};
    if (const int R = db4_cluster_size(nx, ny, levels)) {
        const Db4Cluster p{f, nx, ny, levels, R, lambda, gamma, in, u, epi ? nullptr : out, epi ? *epi : none};
        PP_TRY_CUDA(launch_ex(db4_cluster_kernel, dim3(R), dim3(kDb4Threads), db4_cluster_smem(nx, ny, levels, R),
                              st, pdl, R, p));
        return check_db4("db4_cluster_kernel");
    }
    for (int l = 0; l < levels; ++l) {
        const int h = ny >> l, w = nx >> l;
        PP_TRY_CUDA(launch_ex(db4_rows_kernel<false, false>, dim3(h), dim3(kThreads), 0, st, pdl, 0, f,
                              w, nx, l == 0 ? in : (const float2*)coef, l == 0 ? u : nullptr, gamma,
                              coef, none));
        PP_TRY(check_db4("db4_rows_kernel"));
        PP_TRY_CUDA(launch_ex(db4_cols_kernel<false>, dim3((w + CW - 1) / CW), dim3(kThreads), 0, st,
                              pdl, 0, f, h, w, nx, lambda, (int)(l == levels - 1), coef));
        PP_TRY(check_db4("db4_cols_kernel"));
    }
    for (int l = levels - 1; l >= 0; --l) {
        const int h = ny >> l, w = nx >> l;
        PP_TRY_CUDA(launch_ex(db4_cols_kernel<true>, dim3((w + CW - 1) / CW), dim3(kThreads), 0, st,
                              pdl, 0, f, h, w, nx, lambda, 0, coef));
        PP_TRY(check_db4("db4_cols_kernel"));
        if (l == 0 && epi) {
            PP_TRY_CUDA(launch_ex(db4_rows_kernel<true, true>, dim3(h), dim3(kThreads), 0, st, pdl, 0,
                                  f, w, nx, (const float2*)coef, (const float2*)nullptr, 0.f,
                                  (float2*)nullptr, *epi));
        } else {
            PP_TRY_CUDA(launch_ex(db4_rows_kernel<true, false>, dim3(h), dim3(kThreads), 0, st, pdl, 0,
                                  f, w, nx, (const float2*)coef, (const float2*)nullptr, 0.f,
                                  l == 0 ? out : coef, none));
        }
        PP_TRY(check_db4("db4_rows_kernel"));
    }
    return PP_OK;
}

}  // namespace

void db4_prepare() { (void)db4_largest_cluster(); }

bool db4_supported(int ndim, int nx, int ny, int levels) {
    return ndim == 2 && levels >= 1 && levels <= 4 && nx <= MAXN && ny <= MAXN && nx > 0 && ny > 0 &&
           nx % (1 << levels) == 0 && ny % (1 << levels) == 0;
}

pp_status launch_prox_db4(int nx, int ny, int levels, float lambda, const float2* in, float2* out,
                          cudaStream_t st) {
    return db4_prox(nx, ny, levels, lambda, in, nullptr, 0.f, out, out, nullptr, false, st);
}

pp_status launch_prox_fista_db4(const Plan& p, int levels, float lambda, float gamma, float beta,
                                const float2* u, float2* scratch, const float2* ref, double* hist_slot,
                                cudaStream_t st) {
    const Epi e{p.z, p.y, ref, hist_slot, beta};
    return db4_prox(p.nx, p.ny, levels, lambda, p.z, u, gamma, scratch, nullptr, &e, p.pdl != 0, st);
}

}  // namespace pp
