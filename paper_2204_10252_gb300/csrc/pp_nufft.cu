// Kaiser-Bessel gridding between samples and the oversampled grid (Sec. 5.2):
// G^T (spread, of the adjoint) and G (interpolation, of the forward model).
//
// Spread by gathering.  The samples are sorted by the grid cell of their first
// tap (plan time), so the samples that reach a 4 x 4 tile of grid points are those
// of 7 x 7 cells (periodic): seven contiguous runs, and seven more where the tile
// touches column 0.  A group of LC lanes owns a tile, one coil a lane and the 16
// points' sums in registers; it prepares LC entries' weights at a time, a lane
// each, and then reads the coils' values of one sample after another.  With the
// k-space transposed to [sample][coil] each read is one contiguous run, and the
// sums need no atomics and have a fixed order.
//
// What bounds it: latency of the reads (cell starts, entries, weights, samples in
// turn), 16 warps an SM.  At 65 536 samples on a 320 x 320 grid, 32 coils, a
// sample's values are read three times on average (51 MB); a group that owned one
// point read them 16 times (268 MB), 119 us against 33 us here.  The scatter form
// before that (a CTA per 32 x 32 tile, shared-memory atomics) took 459 us.  85
// registers a thread for three CTAs an SM: 38 us.
//
// Tiles go by the samples that reach them, most first: 50 us in grid order, where
// the centre of a spiral starts late and its neighbours share a CTA.
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

// Rows of 7 cells whose samples reach a 4 x 4 tile of grid points at (ty, tx), one
// a lane (lanes l < 7 of a group of LC): the run's start `s` in the sorted samples
// and the inclusive prefix `pre` of the lengths; returns their total.  wrap: the
// cells left of column 0 (tx < 3) in place of the others; cells right of the tile's
// last column, or below its last row, reach none of its points.  All 32 lanes of
// the warp call it.
template <int LC>
__device__ __forceinline__ int spread_runs(const int* __restrict__ cell_start, int Gx, int Gy, int ty,
                                           int tx, bool live, bool wrap, int l, int* s, int* pre) {
    int st = 0, len = 0;
    int row = ty + l - 3;
    if (live && l < 7 && row < Gy) {
        if (row < 0) row += Gy;
        const int lo = wrap ? Gx + tx - 3 : max(tx - 3, 0);
        const int hi = wrap ? Gx - 1 : min(tx + 3, Gx - 1);
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

struct SpreadTables {
    const int* cell_start;
    const float *wx, *wy;   // [K][4], sorted
    const int2* kx;         // (sample, first-tap column), sorted
    const int* order;       // tiles, those with most entries first
    int Gx, Gy;
};

// One entry of a group's work list: the weights of tile columns 0 .. 3 and rows
// 0 .. 3, each twice (for packed multiplies), zero where the sample does not reach.
struct SpreadEntry {
    float4 x01, x23, y01, y23;
};

// acc[4 b + a] += wy_b wx_a * sample over entries base0 .. base0 + LC,
// base0 + step .. of the n entries of the tile's runs, for this lane's coil (kc,
// NULL: none).  A lane prepares one entry, then all lanes read their coil's value
// of each; eight reads in flight.  nmax: the largest n of the warp's groups.
template <int LC>
__device__ __forceinline__ void spread_sum(float2 (&acc)[16], const SpreadTables& T, int tx, bool wrap,
                                           int l, int s, int pre, int n, int nmax, int base0, int step,
                                           const float2* kc, int64_t ks, SpreadEntry* ent, int* ek) {
    for (int base = base0; base < nmax; base += step) {
        const int t = base + l;
        int idx = 0, before = 0;
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            const int pr = __shfl_sync(0xffffffffu, pre, r, LC);
            if (t >= pr) {
                idx = r + 1;
                before = pr;
            }
        }
        const int sr = __shfl_sync(0xffffffffu, s, idx, LC);
        int k = 0;
        float x[4] = {0.f, 0.f, 0.f, 0.f}, y[4] = {0.f, 0.f, 0.f, 0.f};
        if (t < n) {
            const int j = sr + t - before;
            const int2 e = T.kx[j];
            const int dx = tx - e.y + (wrap ? T.Gx : 0), dy = 3 - idx;
            const float *wx = T.wx + 4 * (int64_t)j, *wy = T.wy + 4 * (int64_t)j;
            k = e.x;
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                if ((unsigned)(a + dx) < 4u) x[a] = wx[a + dx];
                if ((unsigned)(a + dy) < 4u) y[a] = wy[a + dy];
            }
        }
        __syncwarp();
        ent[l].x01 = make_float4(x[0], x[0], x[1], x[1]);
        ent[l].x23 = make_float4(x[2], x[2], x[3], x[3]);
        ent[l].y01 = make_float4(y[0], y[0], y[1], y[1]);
        ent[l].y23 = make_float4(y[2], y[2], y[3], y[3]);
        ek[l] = k;
        __syncwarp();
        const int m = n - base;
        const int mw = nmax - base < LC ? nmax - base : LC;
        for (int u0 = 0; u0 < mw; u0 += 8) {
            float2 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                v[u] = u0 + u < m && kc ? kc[ek[u0 + u] * ks] : make_float2(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const SpreadEntry& e = ent[u0 + u];
                const float4 x01 = e.x01, x23 = e.x23, y01 = e.y01, y23 = e.y23;
                const float2 z = make_float2(0.f, 0.f);
                const float2 w[4] = {__ffma2_rn(make_float2(x01.x, x01.y), v[u], z),
                                     __ffma2_rn(make_float2(x01.z, x01.w), v[u], z),
                                     __ffma2_rn(make_float2(x23.x, x23.y), v[u], z),
                                     __ffma2_rn(make_float2(x23.z, x23.w), v[u], z)};
                const float2 yy[4] = {make_float2(y01.x, y01.y), make_float2(y01.z, y01.w),
                                      make_float2(y23.x, y23.y), make_float2(y23.z, y23.w)};
#pragma unroll
                for (int p = 0; p < 16; ++p) acc[p] = __ffma2_rn(yy[p >> 2], w[p & 3], acc[p]);
            }
        }
    }
}

// Entries above which all groups of a CTA share a tile: 35 us at 64, 34 at 96, 33 at
// 128, 34 at 192 (the 320 x 320 grid above; its centre tile has 1400).
constexpr int kHeavy = 128;

// Every point is written once.  Sample k of coil c is ksp[c * cs + k * ks].  CI:
// grid_out[point][32] (zero at or past C), else grid_out[c][point].  A CTA's groups
// take a tile each, gridDim.x apart in the order, so that the dense ones fall to
// different CTAs; a tile with more than kHeavy
// entries is summed by all groups of its CTA together, one chunk of LC entries at
// a time in turn.
template <int LC, bool CI>
__global__ void __launch_bounds__(256, 2)
nufft_spread_kernel(const SpreadTables T, int C, const float2* __restrict__ ksp, int64_t cs, int64_t ks,
                    float2* __restrict__ grid_out) {
    constexpr int NG = 256 / LC;   // groups (tiles in flight) per CTA
    static_assert(LC >= 8, "a group finds its seven runs one a lane");
    union Shared {
        struct {
            SpreadEntry ent[256];
            int ek[256];
        } w;
        float2 part[16][256];
    };
    __shared__ Shared sh;
    __shared__ int heavy[NG], nheavy;
    const int l = threadIdx.x & (LC - 1), g = threadIdx.x / LC;
    const int c = blockIdx.y * LC + l;
    const int Gx = T.Gx, Gy = T.Gy;
    const int ntx = (Gx + 3) >> 2, ntiles = ntx * ((Gy + 3) >> 2);
    const int64_t np = (int64_t)Gx * Gy;
    const float2* kc = c < C ? ksp + c * cs : nullptr;
    SpreadEntry* ent = sh.w.ent + g * LC;
    int* ek = sh.w.ek + g * LC;
    if (threadIdx.x == 0) nheavy = 0;
    __syncthreads();
    {
        const int place = g * gridDim.x + blockIdx.x;
        const bool live = place < ntiles;
        const int tile = live ? T.order[place] : 0;
        const int ty = 4 * (tile / ntx), tx = 4 * (tile % ntx);
        int s, pre, s2 = 0, pre2 = 0, n2 = 0;
        int n = spread_runs<LC>(T.cell_start, Gx, Gy, ty, tx, live, false, l, &s, &pre);
        const bool edge = __any_sync(0xffffffffu, live && tx < 3);
        if (edge) n2 = spread_runs<LC>(T.cell_start, Gx, Gy, ty, tx, live && tx < 3, true, l, &s2, &pre2);
        const bool big = n + n2 > kHeavy;
        if (big && l == 0) heavy[atomicAdd(&nheavy, 1)] = tile;
        if (big) n = n2 = 0;
        float2 acc[16];
#pragma unroll
        for (int p = 0; p < 16; ++p) acc[p] = make_float2(0.f, 0.f);
        const int nmax = LC < 32 ? __reduce_max_sync(0xffffffffu, n) : n;
        spread_sum<LC>(acc, T, tx, false, l, s, pre, n, nmax, 0, LC, kc, ks, ent, ek);
        if (edge) {
            const int nmax2 = LC < 32 ? __reduce_max_sync(0xffffffffu, n2) : n2;
            spread_sum<LC>(acc, T, tx, true, l, s2, pre2, n2, nmax2, 0, LC, kc, ks, ent, ek);
        }
        if (live && !big) {
            if (CI) {
                float2* o = grid_out + ((int64_t)ty * Gx + tx) * 32 + l;
#pragma unroll
                for (int p = 0; p < 16; ++p)
                    if (ty + (p >> 2) < Gy && tx + (p & 3) < Gx) o[((p >> 2) * Gx + (p & 3)) * 32] = acc[p];
            } else if (c < C) {
                float2* o = grid_out + c * np + (int64_t)ty * Gx + tx;
#pragma unroll
                for (int p = 0; p < 16; p += 2)   // plans have even grids, 16-byte aligned
                    if (ty + (p >> 2) < Gy && tx + (p & 3) < Gx)
                        *reinterpret_cast<float4*>(o + (p >> 2) * Gx + (p & 3)) =
                            make_float4(acc[p].x, acc[p].y, acc[p + 1].x, acc[p + 1].y);
            }
        }
    }
    __syncthreads();
    const int nh = nheavy;
    for (int h = 0; h < nh; ++h) {
        const int tile = heavy[h];
        const int ty = 4 * (tile / ntx), tx = 4 * (tile % ntx);
        float2 acc[16];
#pragma unroll
        for (int p = 0; p < 16; ++p) acc[p] = make_float2(0.f, 0.f);
        for (int wrap = 0; wrap < (tx < 3 ? 2 : 1); ++wrap) {
            int s, pre;
            const int n = spread_runs<LC>(T.cell_start, Gx, Gy, ty, tx, true, wrap != 0, l, &s, &pre);
            // every group of a warp takes the same number of turns
            const int turns = (n + NG * LC - 1) / (NG * LC);
            spread_sum<LC>(acc, T, tx, wrap != 0, l, s, pre, n, g * LC + turns * NG * LC, g * LC, NG * LC,
                           kc, ks, ent, ek);
        }
        __syncthreads();   // the entries and the parts share their memory
#pragma unroll
        for (int p = 0; p < 16; ++p) sh.part[p][threadIdx.x] = acc[p];
        __syncthreads();
        for (int e = threadIdx.x; e < 16 * LC; e += 256) {
            const int p = e / LC, ll = e - p * LC, cc = blockIdx.y * LC + ll;
            const int gy = ty + (p >> 2), gx = tx + (p & 3);
            float2 sum = sh.part[p][ll];
            for (int q = 1; q < NG; ++q) sum = cadd(sum, sh.part[p][q * LC + ll]);
            if (gy >= Gy || gx >= Gx) continue;
            const int64_t lin = (int64_t)gy * Gx + gx;
            if (CI) grid_out[lin * 32 + ll] = sum;
            else if (cc < C) grid_out[cc * np + lin] = sum;
        }
        __syncthreads();
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
// find in L1); 32 samples x 32 coils are transposed through shared memory.  26.6 us
// at 65 536 samples with a sample's taps and values in turn, 25.5 us with the taps of
// all four first and two samples' values in flight.
__global__ void __launch_bounds__(256)
ci_degrid_kernel(const SampleTaps* __restrict__ st, int K, int Gx, int Gy, int C,
                 const float2* __restrict__ grid, float2* __restrict__ ksp) {
    __shared__ float2 tile[32][PT + 1];
    __shared__ SampleTaps taps[PT];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // a warp's four samples' taps at once (past the last sample: the last again,
    // not stored), then 32 grid values in flight
    if (lane < 4) taps[4 * w + lane] = st[min((int)blockIdx.x * PT + 4 * w + lane, K - 1)];
    __syncwarp();
#pragma unroll 2
    for (int q = 0; q < 4; ++q) {
        const int kk = 4 * w + q;
        const SampleTaps s = taps[kk];
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
    const int ntiles = ((p.G_x + 3) / 4) * ((p.G_y + 3) / 4), ng = 256 / LC;
    const dim3 g((ntiles + ng - 1) / ng, (p.C + LC - 1) / LC);
    const SpreadTables T{p.cell_start, reinterpret_cast<const float*>(p.sort_wx),
                         reinterpret_cast<const float*>(p.sort_wy), p.sort_kx, p.tile_order,
                         p.G_x, p.G_y};
    nufft_spread_kernel<LC, CI><<<g, 256, 0, st>>>(T, p.C, ksp, cs, ks, grid_out);
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
