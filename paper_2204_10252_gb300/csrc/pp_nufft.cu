// Kaiser-Bessel gridding between samples and the oversampled grid (Sec. 5.2):
// G^T (spread, of the adjoint) and G (interpolation, of the forward model).
//
// Spread by gathering.  The samples are sorted by the grid cell of their first
// tap (plan time), so the samples that reach grid point (gy, gx), those whose
// first tap lies in rows gy-3 .. gy and columns gx-3 .. gx (periodic), are at
// most two contiguous runs a row: eight runs a point.  A group of LC lanes owns
// a point, one coil a lane; it fetches LC entries' (sample, weight) at a time,
// a lane each, and broadcasts them while every lane reads its own coil's
// value.  With the k-space transposed to [sample][coil] each read is one
// contiguous run, and a point's sum needs neither atomics nor a fixed tile.
//
// What bounds it: L2 reads of 16 values per sample and coil (268 MB at 65 536
// samples, 32 coils).  The scatter form it replaces (a CTA per 32 x 32 tile,
// shared-memory atomics) took 459 us there: a spiral puts a tenth of its samples
// into the four centre tiles, whose CTAs ran long after the others had ended.
#include <cuda_runtime.h>
#include <stdint.h>

#include "pp_internal.h"

namespace pp {
namespace {

constexpr int PT = 32;   // grid points or samples per CTA

// ksp [C][K] -> out [K][Cp], coils c0 .. c0 + LC of chunk blockIdx.y; coils at or
// past C are not written.
template <int LC>
__global__ void __launch_bounds__(256)
ksp_transpose_kernel(const float2* __restrict__ ksp, int K, int C, int Cp, float2* __restrict__ out) {
    __shared__ float2 t[LC][PT + 1];
    const int k0 = blockIdx.x * PT, c0 = blockIdx.y * LC;
    const int tx = threadIdx.x & 31;
#pragma unroll
    for (int c = threadIdx.x >> 5; c < LC; c += 8)
        if (c0 + c < C && k0 + tx < K) t[c][tx] = ksp[(int64_t)(c0 + c) * K + k0 + tx];
    __syncthreads();
    for (int e = threadIdx.x; e < PT * LC; e += 256) {
        const int kk = e / LC, c = e - kk * LC;
        if (c0 + c < C && k0 + kk < K) out[(int64_t)(k0 + kk) * Cp + c0 + c] = t[c][kk];
    }
}

// The eight runs of sorted samples that reach grid point `lin`, one a lane (lanes
// l < 8 of a group of LC): its start `s` and the inclusive prefix `pre` of the
// lengths; returns their total.  All 32 lanes of the warp call it.
template <int LC>
__device__ __forceinline__ int spread_runs(const int* __restrict__ cell_start, int Gx, int Gy, int lin,
                                           bool live, int l, int* s, int* pre) {
    const int gy = lin / Gx, gx = lin - gy * Gx;
    int st = 0, len = 0;
    if (live && l < 8) {
        int row = gy - (l >> 1);
        if (row < 0) row += Gy;
        int lo = 1, hi = 0;
        if ((l & 1) == 0) {
            lo = gx > 3 ? gx - 3 : 0;
            hi = gx;
        } else if (gx < 3) {
            lo = Gx + gx - 3;
            hi = Gx - 1;
        }
        if (lo <= hi) {
            const int* cp = cell_start + (int64_t)row * Gx;
            st = cp[lo];
            len = cp[hi + 1] - st;
        }
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, len, o, LC);
        if (l >= o) len += v;
    }
    *s = st;
    *pre = len;
    return __shfl_sync(0xffffffffu, len, 7, LC);
}

// Sum of weight * sample over entries base0 .. base0 + LC, base0 + step .. of the
// point's n entries, for this lane's coil (kc, NULL: none).  A lane fetches one
// entry, then all lanes read their coil's value of each; eight reads in flight.
// nmax: the largest n of the warp's groups.
template <int LC>
__device__ __forceinline__ float2 spread_sum(const float* __restrict__ wxf, const float* __restrict__ wyf,
                                             const int2* __restrict__ kx, int Gx, int gx, int l, int s,
                                             int pre, int n, int nmax, int base0, int step,
                                             const float2* kc, int64_t ks) {
    float2 acc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u] = make_float2(0.f, 0.f);
    for (int base = base0; base < nmax; base += step) {
        const int t = base + l;
        int idx = 0, before = 0;
#pragma unroll
        for (int r = 0; r < 7; ++r) {
            const int pr = __shfl_sync(0xffffffffu, pre, r, LC);
            if (t >= pr) {
                idx = r + 1;
                before = pr;
            }
        }
        const int sr = __shfl_sync(0xffffffffu, s, idx, LC);
        int k = 0;
        float w = 0.f;
        if (t < n) {
            const int j = sr + t - before;
            const int2 e = kx[j];
            int a = gx - e.y;
            if (a < 0) a += Gx;
            k = e.x;
            w = wxf[4 * (int64_t)j + a] * wyf[4 * (int64_t)j + (idx >> 1)];
        }
        const int m = n - base;
        const int mw = nmax - base < LC ? nmax - base : LC;
        for (int u0 = 0; u0 < mw; u0 += 8) {
            float2 v[8];
            float ww[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int kk = __shfl_sync(0xffffffffu, k, (u0 + u) & (LC - 1), LC);
                ww[u] = __shfl_sync(0xffffffffu, w, (u0 + u) & (LC - 1), LC);
                const bool on = u0 + u < m && kc;
                if (!on) ww[u] = 0.f;
                v[u] = on ? kc[kk * ks] : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                acc[u & 3].x = fmaf(ww[u], v[u].x, acc[u & 3].x);
                acc[u & 3].y = fmaf(ww[u], v[u].y, acc[u & 3].y);
            }
        }
    }
    return cadd(cadd(acc[0], acc[1]), cadd(acc[2], acc[3]));
}

// Every point is written once.  Sample k of coil c is ksp[c * cs + k * ks].  CI:
// grid_out[point][32] (zero at or past C), else grid_out[c][point].  A point with
// more than kHeavy entries (the centre of a spiral holds a thousand: one group
// would need 40 us for it) is summed by all groups of its CTA together: forward +
// adjoint of a 256 x 256 spiral, 32 coils, 208 -> 198 us, and no longer 290 where
// the heavy points meet in one SM.
constexpr int kHeavy = 128;

template <int LC, bool CI>
__global__ void __launch_bounds__(256)
nufft_spread_kernel(const int* __restrict__ cell_start, const float4* __restrict__ wx,
                    const float4* __restrict__ wy, const int2* __restrict__ kx, int Gx, int Gy, int C,
                    const float2* __restrict__ ksp, int64_t cs, int64_t ks,
                    float2* __restrict__ grid_out) {
    constexpr int NG = 256 / LC;   // groups (points in flight) per CTA
    static_assert(LC >= 8, "a group finds its eight runs one a lane");
    __shared__ float2 tile[CI ? 1 : LC][PT + 1];
    __shared__ float2 part[NG][LC];
    __shared__ int heavy[PT], nheavy;
    const int l = threadIdx.x & (LC - 1), g = threadIdx.x / LC;
    const int c = blockIdx.y * LC + l;
    const int np = Gx * Gy;
    const float* wxf = reinterpret_cast<const float*>(wx);
    const float* wyf = reinterpret_cast<const float*>(wy);
    const float2* kc = c < C ? ksp + c * cs : nullptr;
    if (threadIdx.x == 0) nheavy = 0;
    __syncthreads();
#pragma unroll 1
    for (int q = 0; q < PT / NG; ++q) {
        const int pt = q * NG + g, lin = blockIdx.x * PT + pt;
        const bool live = lin < np;
        int s, pre;
        int n = spread_runs<LC>(cell_start, Gx, Gy, lin, live, l, &s, &pre);
        const bool big = n > kHeavy;
        if (big && l == 0) heavy[atomicAdd(&nheavy, 1)] = pt;
        if (big) n = 0;
        const int nmax = LC < 32 ? __reduce_max_sync(0xffffffffu, n) : n;
        const float2 sum = spread_sum<LC>(wxf, wyf, kx, Gx, lin % Gx, l, s, pre, n, nmax, 0, LC, kc, ks);
        if (big || !live) continue;
        if (CI) grid_out[(int64_t)lin * 32 + l] = sum;
        else tile[l][pt] = sum;
    }
    __syncthreads();
    const int nh = nheavy;
    for (int h = 0; h < nh; ++h) {
        const int pt = heavy[h], lin = blockIdx.x * PT + pt;
        int s, pre;
        const int n = spread_runs<LC>(cell_start, Gx, Gy, lin, true, l, &s, &pre);
        // every group of a warp takes the same number of turns
        const int turns = (n + NG * LC - 1) / (NG * LC);
        part[g][l] = spread_sum<LC>(wxf, wyf, kx, Gx, lin % Gx, l, s, pre, n,
                                    g * LC + (turns - 1) * NG * LC + LC, g * LC, NG * LC, kc, ks);
        __syncthreads();
        if (g == 0) {
            float2 sum = part[0][l];
            for (int p = 1; p < NG; ++p) sum = cadd(sum, part[p][l]);
            if (CI) grid_out[(int64_t)lin * 32 + l] = sum;
            else tile[l][pt] = sum;
        }
        __syncthreads();
    }
    if (!CI) {
        const int tx = threadIdx.x & 31, lin = blockIdx.x * PT + tx;
        for (int cc = threadIdx.x >> 5; cc < LC; cc += 8) {
            const int cg = blockIdx.y * LC + cc;
            if (cg < C && lin < np) grid_out[(int64_t)cg * np + lin] = tile[cc][tx];
        }
    }
}

__device__ __forceinline__ int wrapG(int a, int G) {
    a %= G;
    return a < 0 ? a + G : a;
}

// Interpolation in trajectory order, coil-major grid:
// ksp[c][k] = sum_ab wy_b wx_a grid_c[iy0 + b][ix0 + a].
__global__ void __launch_bounds__(256)
nufft_degrid_kernel(const SampleTaps* __restrict__ st, int K, int Gx, int Gy,
                    const float2* __restrict__ grid, float2* __restrict__ ksp) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = blockIdx.y;
    if (k >= K) return;
    const SampleTaps s = st[k];
    const float wx[4] = {s.wx.x, s.wx.y, s.wx.z, s.wx.w};
    const float wy[4] = {s.wy.x, s.wy.y, s.wy.z, s.wy.w};
    const float2* gc = grid + (int64_t)c * Gx * Gy;
    float2 v = make_float2(0.f, 0.f);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const int gy = wrapG(s.iy0 + b, Gy);
        float2 rs = make_float2(0.f, 0.f);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int gx = wrapG(s.ix0 + a, Gx);
            const float2 g = gc[(int64_t)gy * Gx + gx];
            rs.x += wx[a] * g.x;
            rs.y += wx[a] * g.y;
        }
        v.x += wy[b] * rs.x;
        v.y += wy[b] * rs.y;
    }
    ksp[(int64_t)c * K + k] = v;
}

// The same from the coil-innermost grid [Gy][Gx][32]: a warp takes 4 samples in
// turn, one coil a lane (256-byte rows, which neighbouring samples of a readout
// find in L1); 32 samples x 32 coils are transposed through shared memory.
__global__ void __launch_bounds__(256)
ci_degrid_kernel(const SampleTaps* __restrict__ st, int K, int Gx, int Gy, int C,
                 const float2* __restrict__ grid, float2* __restrict__ ksp) {
    __shared__ float2 tile[32][PT + 1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
        const int kk = 4 * w + q, k = blockIdx.x * PT + kk;
        if (k >= K) break;
        const SampleTaps s = st[k];
        const float wx[4] = {s.wx.x, s.wx.y, s.wx.z, s.wx.w};
        const float wy[4] = {s.wy.x, s.wy.y, s.wy.z, s.wy.w};
        const int y0 = wrapG(s.iy0, Gy), x0 = wrapG(s.ix0, Gx);
        float2 v = make_float2(0.f, 0.f);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int gy = y0 + b >= Gy ? y0 + b - Gy : y0 + b;
            float2 rs = make_float2(0.f, 0.f);
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const int gx = x0 + a >= Gx ? x0 + a - Gx : x0 + a;
                const float2 g = grid[((int64_t)gy * Gx + gx) * 32 + lane];
                rs.x += wx[a] * g.x;
                rs.y += wx[a] * g.y;
            }
            v.x += wy[b] * rs.x;
            v.y += wy[b] * rs.y;
        }
        tile[lane][kk] = v;
    }
    __syncthreads();
    const int k = blockIdx.x * PT + lane;
    for (int c = w; c < C; c += 8)
        if (k < K) ksp[(int64_t)c * K + k] = tile[c][lane];
}

pp_status check_nufft(const char* what) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_status(e, what);
    ++g_launches;
    if (g_profiler) g_profiler->mark(what);
    return PP_OK;
}

// Lanes a point: the coil count rounded up to 8, 16 or 32.
int lanes_for(int C) { return C <= 8 ? 8 : (C <= 16 ? 16 : 32); }

// [C][K] -> [K][Cp], Cp the coil count rounded up to whole chunks of lc lanes
pp_status transpose_ksp(const Plan& p, int lc, const float2* ksp, int Cp, float2* kt, cudaStream_t st) {
    const dim3 g((p.K + PT - 1) / PT, Cp / lc);
    if (lc == 8) ksp_transpose_kernel<8><<<g, 256, 0, st>>>(ksp, p.K, p.C, Cp, kt);
    else if (lc == 16) ksp_transpose_kernel<16><<<g, 256, 0, st>>>(ksp, p.K, p.C, Cp, kt);
    else ksp_transpose_kernel<32><<<g, 256, 0, st>>>(ksp, p.K, p.C, Cp, kt);
    return check_nufft("ksp_transpose_kernel");
}

template <int LC, bool CI>
pp_status spread(const Plan& p, const float2* ksp, int64_t cs, int64_t ks, float2* grid_out,
                 cudaStream_t st) {
    const dim3 g((p.G_x * p.G_y + PT - 1) / PT, (p.C + LC - 1) / LC);
    nufft_spread_kernel<LC, CI><<<g, 256, 0, st>>>(p.cell_start, p.sort_wx, p.sort_wy, p.sort_kx, p.G_x,
                                                   p.G_y, p.C, ksp, cs, ks, grid_out);
    return check_nufft("nufft_spread_kernel");
}

}  // namespace

size_t nufft_transposed_elems(const Plan& p) {
    const int lc = lanes_for(p.C);
    return (size_t)p.K * ((p.C + lc - 1) / lc) * lc;
}

// grid_out = G^T ksp.  kt: nufft_transposed_elems(p) elements of scratch, or
// NULL to read the [C][K] array in place (for callers without that much
// scratch: a lane's reads then lie K apart).  ci: grid_out is [Gy][Gx][32].
pp_status launch_nufft_spread(const Plan& p, const float2* ksp, float2* kt, float2* grid_out, bool ci,
                              cudaStream_t st) {
    const int lc = lanes_for(p.C), Cp = (p.C + lc - 1) / lc * lc;
    int64_t cs = p.K, ks = 1;
    if (kt) {
        PP_TRY(transpose_ksp(p, lc, ksp, Cp, kt, st));
        ksp = kt;
        cs = 1;
        ks = Cp;
    }
    // all 32 lanes write on the coil-innermost grid (zeros at or past C), so
    // that the padding coils of its later stages hold finite values
    if (ci) return spread<32, true>(p, ksp, cs, ks, grid_out, st);
    if (lc == 8) return spread<8, false>(p, ksp, cs, ks, grid_out, st);
    if (lc == 16) return spread<16, false>(p, ksp, cs, ks, grid_out, st);
    return spread<32, false>(p, ksp, cs, ks, grid_out, st);
}

pp_status launch_nufft_degrid(const Plan& p, const float2* grid_in, float2* ksp, bool ci,
                              cudaStream_t st) {
    if (ci) {
        ci_degrid_kernel<<<(p.K + PT - 1) / PT, 256, 0, st>>>(p.samp, p.K, p.G_x, p.G_y, p.C, grid_in, ksp);
        return check_nufft("ci_degrid_kernel");
    }
    nufft_degrid_kernel<<<dim3((p.K + 255) / 256, p.C), 256, 0, st>>>(p.samp, p.K, p.G_x, p.G_y, grid_in,
                                                                      ksp);
    return check_nufft("nufft_degrid_kernel");
}

}  // namespace pp
