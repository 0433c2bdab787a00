// C ABI of libpp: plan set-up on the host, operator orchestration, the
// Horner recursion of Listing "pcode" and Algorithm "pfista" (Sec. 3.1, 3.6).
#include <cuda_runtime.h>
#include <math.h>

#include <cmath>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <thread>
#include <functional>
#include <map>
#include <mutex>
#include <tuple>
#include <string>
#include <vector>

#include "pp_batch.h"
#include "pp_fft4.cuh"
#include "pp_internal.h"
#include "pp_twiddles.h"

namespace pp {

// ---------------------------------------------------------------------------
// errors
// ---------------------------------------------------------------------------
static thread_local std::string g_last_error;

void set_error(const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_last_error = buf;
}

pp_status cuda_status(cudaError_t e, const char* what) {
    set_error("%s: %s", what, cudaGetErrorString(e));
    cudaGetLastError();   // a refused launch is not to be found by the next one's check
    return e == cudaErrorMemoryAllocation ? PP_ERR_OOM : PP_ERR_CUDA;
}

// ---------------------------------------------------------------------------
// host helpers
// ---------------------------------------------------------------------------
// Stage radices for length n: as many 8s as the power of two allows (a
// remainder of 2^1 becomes 4*4 in place of one 8, or a single 2), then 5s and
// 3s.  Returns false when n has a prime factor above 5.
static bool factorize(int n, FftDesc& d) {
    if (n < 2) return false;
    int e2 = 0, m = n;
    while (m % 2 == 0) { m /= 2; ++e2; }
    int n5 = 0, n3 = 0;
    while (m % 5 == 0) { m /= 5; ++n5; }
    while (m % 3 == 0) { m /= 3; ++n3; }
    if (m != 1) return false;
    std::vector<int> r;
    int q = e2 / 3, rem = e2 % 3;
    if (rem == 1 && q >= 1) { for (int i = 0; i < q - 1; ++i) r.push_back(8); r.push_back(4); r.push_back(4); }
    else { for (int i = 0; i < q; ++i) r.push_back(8); if (rem == 2) r.push_back(4); if (rem == 1) r.push_back(2); }
    for (int i = 0; i < n5; ++i) r.push_back(5);
    for (int i = 0; i < n3; ++i) r.push_back(3);
    if ((int)r.size() > 8) return false;
    d.n = n;
    d.nst = (int)r.size();
    for (int i = 0; i < 8; ++i) d.rad[i] = i < d.nst ? r[i] : 0;
    return true;
}

static pp_status dev_alloc(Plan& p, void** ptr, size_t bytes) {
    *ptr = nullptr;
    if (bytes == 0) return PP_OK;
    cudaError_t e = cudaMalloc(ptr, bytes);
    if (e != cudaSuccess) {
        *ptr = nullptr;
        cudaGetLastError();
        return cuda_status(e, "cudaMalloc");
    }
    p.allocs.push_back(*ptr);
    return PP_OK;
}

template <class T>
static pp_status alloc_n(Plan& p, T** ptr, size_t n) {
    return dev_alloc(p, reinterpret_cast<void**>(ptr), n * sizeof(T));
}

// A workspace that only makes things faster: NULL, and no error, where it would take
// more than half of the free memory.
static void* spare_alloc(size_t bytes) {
    size_t room = 0, total = 0;
    void* ptr = nullptr;
    if (cudaMemGetInfo(&room, &total) == cudaSuccess && bytes <= room / 2 && cudaMalloc(&ptr, bytes) == cudaSuccess)
        return ptr;
    cudaGetLastError();
    return nullptr;
}

// The balanced table of a length, kept for the life of the process (60 lengths at
// most): a batch makes two a slice.
static const std::vector<Twiddle>& twiddles_of(int n, const GenSplit& g) {
    static std::mutex mu;
    static std::map<int, std::vector<Twiddle>> kept;
    std::lock_guard<std::mutex> lock(mu);
    std::vector<Twiddle>& tw = kept[n];
    if (tw.empty()) tw = balanced_twiddles(g.n1, g.n2);
    return tw;
}

static pp_status make_fft(Plan& p, int n, DevFft& f) {
    if (!factorize(n, f.d)) {
        set_error("FFT length %d has a prime factor above 5", n);
        return PP_ERR_UNSUPPORTED;
    }
    std::vector<float2> tw(n);
    for (int t = 0; t < n; ++t) {
        const double a = -2.0 * M_PI * (double)t / (double)n;
        tw[t] = make_float2((float)cos(a), (float)sin(a));
    }
    const GenSplit g = gen_split_of(n);
    if (g.n1)   // both tables in one array
        for (const Twiddle& w : twiddles_of(n, g)) tw.push_back(make_float2(w.x, w.y));
    PP_TRY(alloc_n(p, &f.tw, tw.size()));
    PP_TRY_CUDA(cudaMemcpy(f.tw, tw.data(), tw.size() * sizeof(float2), cudaMemcpyHostToDevice));
    f.twb = g.n1 ? f.tw + n : f.tw;
    return PP_OK;
}

template <class T>
static pp_status upload(Plan& p, T** dst, const std::vector<T>& src) {
    PP_TRY(alloc_n(p, dst, src.size()));
    PP_TRY_CUDA(cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice));
    return PP_OK;
}

// Kaiser-Bessel pieces (width W, shape beta):
//   kernel  phi(u) = I0(beta sqrt(1 - (2u/W)^2)), |u| <= W/2
//   its Fourier transform psi(nu) = W sinh(sqrt(a))/sqrt(a), a = beta^2 - (pi W nu)^2
// Kaiser-Bessel kernel phi(u) = I0(beta sqrt(1 - (2u/W)^2)) for |u| <= W/2,
// 0 outside, by the power series I0(x) = sum_k q^k / (k!)^2, q = x^2 / 4.
// Every argument of a plan is at most beta, so one term count serves all:
// the first k at which q_max^k / (k!)^2 < 1e-17 (the sum is >= 1, and past
// the largest term each term shrinks by q / (k + 1)^2 < 1).
static int kb_series_terms(double beta) {
    const double q = 0.25 * beta * beta;
    double t = 1.0;
    int k = 1;
    for (; k < 200; ++k) {
        t *= q / ((double)k * k);
        if (t < 1e-17) break;
    }
    return k;
}
// phi at the 8 offsets u[0..7] (a sample's 4 x-taps and 4 y-taps), the 8
// series summed side by side; inv_k2[k - 1] = 1 / k^2
static void kb_phi8(const double* u, double W, double beta, int nterms, const double* inv_k2,
                    float* out) {
    double q[8], term[8], sum[8];
    for (int i = 0; i < 8; ++i) {
        const double r = 2.0 * u[i] / W, t = 1.0 - r * r;
        q[i] = t < 0.0 ? 0.0 : 0.25 * beta * beta * t;
        term[i] = 1.0;
        sum[i] = 1.0;
    }
    for (int k = 0; k < nterms; ++k)
        for (int i = 0; i < 8; ++i) {
            term[i] *= q[i] * inv_k2[k];
            sum[i] += term[i];
        }
    for (int i = 0; i < 8; ++i) {
        const double r = 2.0 * u[i] / W;
        out[i] = 1.0 - r * r < 0.0 ? 0.f : (float)sum[i];
    }
}
static double kb_psi(double nu, double W, double beta) {
    const double a = beta * beta - (M_PI * W * nu) * (M_PI * W * nu);
    if (a > 0) return W * sinh(sqrt(a)) / sqrt(a);
    if (a < 0) return W * sin(sqrt(-a)) / sqrt(-a);
    return W;
}

static inline int wrap_host(int a, int G) {
    a %= G;
    return a < 0 ? a + G : a;
}

// ---------------------------------------------------------------------------
// operator orchestration
// ---------------------------------------------------------------------------
static ColArgs col_args(int Hin, int Hout, int G, int off_in, int off_out, int ncols,
                        int64_t ibs, int64_t obs, int nbatch, float scale) {
    ColArgs a;
    a.Hin = Hin; a.Hout = Hout; a.G = G; a.off_in = off_in; a.off_out = off_out;
    a.ncols = ncols; a.in_batch_stride = ibs; a.out_batch_stride = obs; a.nbatch = nbatch;
    a.scale = scale; a.mul_in = nullptr; a.mul_out = nullptr; a.mo_q = 0; a.mo_c = 0; a.mo_cdiv = 1;
    a.mi_q = 1; a.mi_c = 0; a.mi_cdiv = 1;
    return a;
}

static RowArgs row_args(int n, int G, int off_in, int off_out, int nrows, int64_t cis, float scale) {
    RowArgs a;
    a.n = n; a.G = G; a.off_in = off_in; a.off_out = off_out; a.nrows = nrows;
    a.coil_img_stride = cis; a.scale = scale;
    return a;
}

// Whether a non-Cartesian plan runs on the coil-innermost arrays: as the tuner
// found faster for its normal operator (the forward and adjoint applies share
// its FFT stages).
static bool use_ci(const Plan& p) { return !p.toep && p.tune_stencil_kind >= 7 && p.ci_sens && p.ci_a; }

// A chain of normal-operator applications in one launch (2-D Cartesian plans
// whose ny has a column-resident kernel).
static pp_status cart_chain(const Plan& p, const float2* x, const CartChain& ch, cudaStream_t st) {
    CartLaunch L;
    L.one.twb = p.fy.twb; L.one.sens = p.sens; L.one.mask_fo = p.mask_fo;
    L.one.ny = p.ny; L.one.nx = p.nx; L.one.C = p.C; L.one.img_off = 0; L.one.invL = 1.f;
    L.max_coils = p.C;
    L.W = ch.J > 1 ? p.tune_c2 : p.tune_c2_one;
    while (L.W > 1 && !cart_cols_width_ok(p.ny, L.W)) L.W >>= 1;
    L.pdl = p.pdl != 0;
    return launch_cart_cols(p.ny, L, x, ch, st);
}

// Appends the Horner recursion (Listing "pcode") u = c_d v, u = c_i v + N u to a
// chain, d >= 1; coefficients in units of the operator times `invL`.
static void chain_horner(CartChain& ch, const double* c, int d, double invL) {
    for (int i = d - 1; i >= 0; --i) {
        ch.sc[ch.J] = (float)(i == d - 1 ? c[d] * invL : invL);
        ch.al[ch.J] = (float)c[i];
        ++ch.J;
    }
}

// out = scale * (A^H A x) + alpha * operand   (operand may be NULL)
static pp_status normal_into(const Plan& p, const float2* x, float2* out, float scale,
                             const float2* operand, float alpha, cudaStream_t st) {
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int64_t n = p.nimg;
    if (p.kind == PP_CARTESIAN && p.ndim == 2) {
        if (!p.cols) return launch_cart2d_normal(p, x, out, scale, operand, alpha, st);
        CartChain ch;
        ch.sc[0] = scale;
        ch.al[0] = alpha;
        ch.ext = operand;
        ch.out = out;
        return cart_chain(p, x, ch, st);
    }
    if (p.kind == PP_CARTESIAN) {
        if (p.tune_c3 == 1 && p.c3cl_clusters > 0)
            return c3cl_normal(p, 4, x, out, scale, operand, alpha, st);
        if (p.tune_c3 == 2 && p.c3cl2_clusters > 0)
            return c3cl_normal(p, 2, x, out, scale, operand, alpha, st);
        if (p.tune_c3 == 3 && p.c3df_ctas > 0)
            return c3df_normal(p, x, out, scale, operand, alpha, st);
        bool done = false;
        PP_TRY(cart3d4_normal(p, x, out, scale, operand, alpha, p.wk_a, st, &done));
        if (done) return PP_OK;
        PP_TRY(lines_cart3d_normal(p, x, out, scale, operand, alpha, p.wk_a, p.c3_chunk, st, &done));
        if (done) return PP_OK;
        // 3-D: per coil, y FFT -> (z FFT, mask, z IFFT) -> y IFFT -> conj accumulate
        for (int c = 0; c < p.C; ++c) {
            const float2* sc = p.sens + (int64_t)c * n;
            PP_TRY(launch_expand(x, sc, p.wk_a, n, st));
            ColArgs ay = col_args(ny, ny, ny, 0, 0, nx, (int64_t)ny * nx, (int64_t)ny * nx, nz, 1.f);
            PP_TRY(launch_cols(p.fy, ay, p.wk_a, p.wk_b, false, st));
            ColArgs az = col_args(nz, nz, nz, 0, 0, ny * nx, 0, 0, 1, 1.f);
            az.mo_q = ny; az.mo_c = 1; az.mo_cdiv = nx;
            PP_TRY(launch_cols_roundtrip(p.fz, az, p.mask_fo, p.wk_b, p.wk_a, st));
            PP_TRY(launch_cols(p.fy, ay, p.wk_a, p.wk_b, true, st));
            PP_TRY(launch_conj_accum(sc, p.wk_b, out, n, c == 0, scale, operand, alpha, c == p.C - 1, st));
        }
        return PP_OK;
    }
    if (p.toep) return toep_normal(p, x, out, scale, operand, alpha, st);
    // non-Cartesian: rows -> cols -> G^T G stencil -> cols^H -> rows^H
    if (use_ci(p))
        return ci_normal(p, x, out, scale, operand, alpha,
                         p.tune_stencil_kind == 9 ? 0 : (p.tune_stencil_kind == 8 ? 2 : 1), st);
    const int Gx = p.G_x, Gy = p.G_y;
    RowArgs rf = row_args(nx, Gx, nx / 2, 0, ny, (int64_t)ny * nx, 1.f);
    PP_TRY(launch_rows_fwd(p, p.gx, rf, x, p.sens, p.deapod_y, p.deapod_x, p.wk_a, p.C, 0, st));
    ColArgs cf = col_args(ny, Gy, Gy, ny / 2, 0, Gx, (int64_t)ny * Gx, (int64_t)Gy * Gx, p.C, 1.f);
    PP_TRY(launch_cols(p.gy, cf, p.wk_a, p.wk_b, false, st));
    PP_TRY(launch_gtg_stencil(p, p.wk_b, p.wk_c, st));
    ColArgs ci = col_args(Gy, ny, Gy, 0, ny / 2, Gx, (int64_t)Gy * Gx, (int64_t)ny * Gx, p.C, 1.f);
    PP_TRY(launch_cols(p.gy, ci, p.wk_c, p.wk_a, true, st));
    RowArgs ra = row_args(nx, Gx, 0, nx / 2, ny, (int64_t)ny * nx, scale);
    if (p.tune_rows_adj_cl == -1) {
        bool done = false;
        PP_TRY(launch_rows4_adj_split(p.gx, ra, p.wk_a, p.sens, p.deapod_y, p.deapod_x, p.wk_c, out,
                                      operand, alpha, p.C, st, &done));
        if (done) return PP_OK;
    }
    return launch_rows_adj(p, p.gx, ra, p.wk_a, p.sens, p.deapod_y, p.deapod_x, out, operand, alpha,
                           p.C, st);
}

// y = A x (unscaled)
static pp_status forward_into(const Plan& p, const float2* x, float2* y, cudaStream_t st) {
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int64_t n = p.nimg;
    if (p.kind == PP_CARTESIAN) {
        // centred orthonormal FFT along x, then y (then z), mask on the last axis pass
        RowArgs rf = row_args(nx, nx, nx / 2, nx / 2, ny * nz, n, (float)(1.0 / sqrt((double)nx)));
        ColArgs ay = col_args(ny, ny, ny, ny / 2, ny / 2, nx, (int64_t)ny * nx, (int64_t)ny * nx,
                              p.C * nz, (float)(1.0 / sqrt((double)ny)));
        if (p.ndim == 2) {
            PP_TRY(launch_rows_fwd(p, p.fx, rf, x, p.sens, nullptr, nullptr, y, p.C, 0, st));
            ay.mul_out = p.mask_c; ay.mo_q = 1; ay.mo_c = 0; ay.mo_cdiv = 1;
            return launch_cols(p.fy, ay, y, y, false, st);
        }
        // a chunk of coils at a time, so that its three passes meet in L2
        for (int c0 = 0; c0 < p.C; c0 += p.c3_chunk) {
            const int nc = std::min(p.c3_chunk, p.C - c0);
            float2* yc = y + (int64_t)c0 * n;
            PP_TRY(launch_rows_fwd(p, p.fx, rf, x, p.sens + (int64_t)c0 * n, nullptr, nullptr, yc, nc, 0, st));
            ay.nbatch = nc * nz;
            PP_TRY(launch_cols(p.fy, ay, yc, yc, false, st));
            ColArgs az = col_args(nz, nz, nz, nz / 2, nz / 2, ny * nx, n, n, nc,
                                  (float)(1.0 / sqrt((double)nz)));
            az.mul_out = p.mask_c; az.mo_q = ny; az.mo_c = 1; az.mo_cdiv = nx;
            PP_TRY(launch_cols(p.fz, az, yc, yc, false, st));
        }
        return PP_OK;
    }
    if (use_ci(p)) {
        PP_TRY(ci_to_grid(p, x, st));
        return launch_nufft_degrid(p, p.ci_b, y, true, st);
    }
    const int Gx = p.G_x, Gy = p.G_y;
    RowArgs rf = row_args(nx, Gx, nx / 2, 0, ny, (int64_t)ny * nx, 1.f);
    PP_TRY(launch_rows_fwd(p, p.gx, rf, x, p.sens, p.deapod_y, p.deapod_x, p.wk_a, p.C, 0, st));
    ColArgs cf = col_args(ny, Gy, Gy, ny / 2, 0, Gx, (int64_t)ny * Gx, (int64_t)Gy * Gx, p.C, 1.f);
    PP_TRY(launch_cols(p.gy, cf, p.wk_a, p.wk_b, false, st));
    return launch_nufft_degrid(p, p.wk_b, y, false, st);
}

// x = A^H y (unscaled) with the intermediates in wa and wb (plan workspace, or the
// library's fixed scratch array for pp_adjoint_apply_static): Cartesian 2-D
// needs C*n elements in wa; 3-D chunk*n in wa; non-Cartesian C*ny*G_x
// in wa and C*G_y*G_x in wb, and optionally the transposed k-space in kt.
pp_status adjoint_ws(const Plan& p, const float2* y, float2* x, float2* wa, float2* wb, float2* kt,
                     int chunk, cudaStream_t st) {
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int64_t n = p.nimg;
    if (p.kind == PP_CARTESIAN && p.ndim == 2) {
        ColArgs ay = col_args(ny, ny, ny, ny / 2, ny / 2, nx, (int64_t)ny * nx, (int64_t)ny * nx, p.C,
                              (float)(1.0 / sqrt((double)ny)));
        ay.mul_in = p.mask_c;   // centred mask indexed by the input row ky
        PP_TRY(launch_cols(p.fy, ay, y, wa, true, st));
        RowArgs ra = row_args(nx, nx, nx / 2, nx / 2, ny, n, (float)(1.0 / sqrt((double)nx)));
        return launch_rows_adj(p, p.fx, ra, wa, p.sens, nullptr, nullptr, x, nullptr, 0.f, p.C, st);
    }
    if (p.kind == PP_CARTESIAN) {
        // 3-D, `chunk` coils at a time (their planes meet in L2): mask and
        // inverse centred FFT along z into wa, then y in place, then the x rows
        // with the conjugate sensitivities, accumulated into x.
        for (int c0 = 0; c0 < p.C; c0 += chunk) {
            const int nc = std::min(chunk, p.C - c0);
            ColArgs az = col_args(nz, nz, nz, nz / 2, nz / 2, ny * nx, n, n, nc,
                                  (float)(1.0 / sqrt((double)nz)));
            az.mul_in = p.mask_c; az.mi_q = ny; az.mi_c = 1; az.mi_cdiv = nx;
            PP_TRY(launch_cols(p.fz, az, y + (int64_t)c0 * n, wa, true, st));
            ColArgs ay = col_args(ny, ny, ny, ny / 2, ny / 2, nx, (int64_t)ny * nx, (int64_t)ny * nx,
                                  nz * nc, (float)(1.0 / sqrt((double)ny)));
            PP_TRY(launch_cols(p.fy, ay, wa, wa, true, st));
            RowArgs ra = row_args(nx, nx, nx / 2, nx / 2, ny * nz, n, (float)(1.0 / sqrt((double)nx)));
            PP_TRY(launch_rows_adj(p, p.fx, ra, wa, p.sens + (int64_t)c0 * n, nullptr, nullptr, x,
                                   c0 == 0 ? nullptr : x, 1.f, nc, st));
        }
        return PP_OK;
    }
    const int Gx = p.G_x, Gy = p.G_y;
    PP_TRY(launch_nufft_spread(p, y, kt, wb, false, st));
    ColArgs ci = col_args(Gy, ny, Gy, 0, ny / 2, Gx, (int64_t)Gy * Gx, (int64_t)ny * Gx, p.C, 1.f);
    PP_TRY(launch_cols(p.gy, ci, wb, wa, true, st));
    RowArgs ra = row_args(nx, Gx, 0, nx / 2, ny, (int64_t)ny * nx, 1.f);
    return launch_rows_adj(p, p.gx, ra, wa, p.sens, p.deapod_y, p.deapod_x, x, nullptr, 0.f,
                           p.C, st);
}

static pp_status adjoint_into(const Plan& p, const float2* y, float2* x, cudaStream_t st) {
    if (use_ci(p)) {
        PP_TRY(launch_nufft_spread(p, y, p.ksp_t, p.ci_c, true, st));
        return ci_from_grid(p, p.ci_c, x, 1.f, nullptr, 0.f, st);
    }
    return adjoint_ws(p, y, x, p.wk_a, p.wk_b, p.ksp_t, p.c3_chunk, st);
}

// ---------------------------------------------------------------------------
// plan construction
// ---------------------------------------------------------------------------
static pp_status build_cartesian(Plan& p, const uint8_t* mask) {
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    // readout invariance: mask[z][y][x] == mask[z][y][0]
    std::vector<float> mc((size_t)nz * ny), mfo((size_t)nz * ny);
    for (int z = 0; z < nz; ++z)
        for (int yy = 0; yy < ny; ++yy) {
            const uint8_t* row = mask + ((size_t)z * ny + yy) * nx;
            const uint8_t m0 = row[0] ? 1 : 0;
            for (int x = 1; x < nx; ++x)
                if ((row[x] ? 1 : 0) != m0) {
                    set_error("Cartesian mask varies along the readout axis x (z=%d, y=%d)", z, yy);
                    return PP_ERR_UNSUPPORTED;
                }
            mc[(size_t)z * ny + yy] = (float)m0;
        }
    // FFT order: centred index q holds frequency q - n/2, stored at (q - n/2) mod n
    const double norm = 1.0 / ((double)ny * (double)nz);
    for (int z = 0; z < nz; ++z)
        for (int yy = 0; yy < ny; ++yy) {
            const int zf = wrap_host(z - nz / 2, nz), yf = wrap_host(yy - ny / 2, ny);
            mfo[(size_t)zf * ny + yf] = (float)(mc[(size_t)z * ny + yy] * norm);
        }
    PP_TRY(upload(p, &p.mask_c, mc));
    PP_TRY(upload(p, &p.mask_fo, mfo));
    PP_TRY(make_fft(p, nx, p.fx));
    PP_TRY(make_fft(p, ny, p.fy));
    if (p.ndim == 3) PP_TRY(make_fft(p, nz, p.fz));
    if (p.external_wk) {
        // workspace set by the owner
    } else if (p.ndim == 2) {
        PP_TRY(alloc_n(p, &p.wk_a, (size_t)p.C * p.nimg));
    } else {
        PP_TRY(alloc_n(p, &p.wk_a, (size_t)p.nimg));   // see widen_c3
        // the passes for axes without compiled stages alternate between two volumes
        if (!lines_have(ny) || !lines_have(nz)) PP_TRY(alloc_n(p, &p.wk_b, (size_t)p.nimg));
    }
    p.nksp = (int64_t)p.C * p.nimg;
    return PP_OK;
}

// 3-D: coils of one launch of each stage, 512 MB of planes, or the half, the quarter ..
// of them where the memory is short.  Planes that fit L2 together (72 MB) leave each
// launch short: the stages read little back from L2 (26 % hits), and every launch ends
// in a part wave and, in the adjoint, adds to the image.  80 x 180 x 200 x 12, forward +
// adjoint / normal: 862 / 502 us at 72 MB, 789 / - at 200, 746 / 429 at 512 and above;
// 128 x 200 x 200 x 9, normal: 1090 -> 650.
static void widen_c3(Plan& p) {
    const int64_t volume = p.nimg * (int64_t)sizeof(float2);
    for (int c = (int)std::min<int64_t>(p.C, (512ll << 20) / volume); c > 1; c = (c + 1) / 2)
        if (void* w = spare_alloc((size_t)(c * volume))) {
            cudaFree(p.wk_a);
            std::replace(p.allocs.begin(), p.allocs.end(), (void*)p.wk_a, w);
            p.wk_a = static_cast<float2*>(w);
            p.c3_chunk = c;
            return;
        }
}

static pp_status build_noncartesian(Plan& p, const pp_sampling* s) {
    const int nx = p.nx, ny = p.ny;
    const int W = s->kb_width;
    const double sigma = s->oversamp;
    if (W != 4) {
        set_error("kb_width must be 4");
        return PP_ERR_UNSUPPORTED;
    }
    if (!(sigma >= 1.125 && sigma <= 2.0)) {
        set_error("oversamp must lie in [1.125, 2]");
        return PP_ERR_INVALID_ARG;
    }
    if (s->K < 1 || s->K > (1 << 26)) {
        set_error("K out of range");
        return PP_ERR_INVALID_ARG;
    }
    const int Gx = (int)ceil(sigma * nx - 1e-9), Gy = (int)ceil(sigma * ny - 1e-9);
    if ((Gx & 1) || (Gy & 1)) {
        set_error("oversampled grid %dx%d must be even", Gy, Gx);
        return PP_ERR_UNSUPPORTED;
    }
    p.G_x = Gx; p.G_y = Gy; p.W = W; p.K = (int)s->K;
    if (Gx < 32 + 2 * W || Gy < 32 + 2 * W) {   // 40 points: see pp_sampling
        set_error("oversampled grid too small for gridding");
        return PP_ERR_UNSUPPORTED;
    }
    PP_TRY(make_fft(p, Gx, p.gx));
    PP_TRY(make_fft(p, Gy, p.gy));
    // Beatty et al. (2005) shape parameter
    const double beta = M_PI * sqrt((W / sigma) * (W / sigma) * (sigma - 0.5) * (sigma - 0.5) - 0.8);
    std::vector<float> dx(nx), dy(ny);
    for (int i = 0; i < nx; ++i)
        dx[i] = (float)(1.0 / (sqrt((double)nx) * kb_psi((double)(i - nx / 2) / Gx, W, beta)));
    for (int i = 0; i < ny; ++i)
        dy[i] = (float)(1.0 / (sqrt((double)ny) * kb_psi((double)(i - ny / 2) / Gy, W, beta)));
    PP_TRY(upload(p, &p.deapod_x, dx));
    PP_TRY(upload(p, &p.deapod_y, dy));
    // per-sample taps: m in (s - W/2, s + W/2], s = kappa * G / n.  The Bessel
    // series of 8 taps per sample dominates plan set-up at tens of thousands
    // of samples, so contiguous sample ranges run on the host's cores (each
    // sample's taps depend on that sample alone: the result is the same for
    // any thread count)
    const int nterms = kb_series_terms(beta);
    double inv_k2[200];
    for (int k = 1; k <= nterms; ++k) inv_k2[k - 1] = 1.0 / ((double)k * k);
    const int K = p.K;
    std::vector<SampleTaps> st(K);
    std::atomic<int> bad(K);   // the first sample outside the grid, if any
    auto taps = [&](int k0, int k1) {
        for (int k = k0; k < k1; ++k) {
            const double kx = s->traj[2 * k], ky = s->traj[2 * k + 1];
            if (!(kx >= -nx / 2.0 && kx < nx / 2.0 && ky >= -ny / 2.0 && ky < ny / 2.0)) {
                int cur = bad.load();
                while (k < cur && !bad.compare_exchange_weak(cur, k)) {
                }
                continue;
            }
            const double sx = kx * Gx / nx, sy = ky * Gy / ny;
            const int ix0 = (int)floor(sx - W / 2.0) + 1, iy0 = (int)floor(sy - W / 2.0) + 1;
            double u[8];
            for (int a = 0; a < 4; ++a) {
                u[a] = sx - (ix0 + a);
                u[4 + a] = sy - (iy0 + a);
            }
            float w[8];
            kb_phi8(u, W, beta, nterms, inv_k2, w);
            st[k].wx = make_float4(w[0], w[1], w[2], w[3]);
            st[k].wy = make_float4(w[4], w[5], w[6], w[7]);
            st[k].ix0 = ix0;
            st[k].iy0 = iy0;
        }
    };
    // runs body(k0, k1) over nth contiguous ranges of [0, K) on host threads
    const int nth = std::max(1, std::min({16, (int)std::thread::hardware_concurrency(), K / 4096 + 1}));
    auto on_threads = [&](auto&& body) {
        std::vector<std::thread> pool;
        size_t handed = 1;
        try {
            for (int t = 1; t < nth; ++t, ++handed)
                pool.emplace_back(body, (int)((int64_t)K * t / nth), (int)((int64_t)K * (t + 1) / nth));
        } catch (const std::exception&) {
            // no more threads: the calling thread takes the ranges not handed out
            for (int t = (int)handed; t < nth; ++t)
                body((int)((int64_t)K * t / nth), (int)((int64_t)K * (t + 1) / nth));
        }
        body(0, (int)((int64_t)K / nth));
        for (auto& th : pool) th.join();
    };
    on_threads(taps);
    if (bad.load() < K) {
        const int k = bad.load();
        set_error("trajectory sample %d (%g, %g) outside [-n/2, n/2)", k, s->traj[2 * k], s->traj[2 * k + 1]);
        return PP_ERR_INVALID_ARG;
    }
    PP_TRY(upload(p, &p.samp, st));
    // samples sorted by the cell of their first tap (stable: trajectory order
    // within a cell), for the spread
    {
        std::vector<int> start((size_t)Gx * Gy + 1, 0), cell(K);
        for (int k = 0; k < K; ++k) {
            cell[k] = wrap_host(st[k].iy0, Gy) * Gx + wrap_host(st[k].ix0, Gx);
            ++start[cell[k] + 1];
        }
        for (size_t i = 0; i < (size_t)Gx * Gy; ++i) start[i + 1] += start[i];
        std::vector<float4> wx(K), wy(K);
        std::vector<int2> kx(K);
        std::vector<int> next(start.begin(), start.end() - 1);
        for (int k = 0; k < K; ++k) {
            const int j = next[cell[k]]++;
            wx[j] = st[k].wx;
            wy[j] = st[k].wy;
            kx[j] = make_int2(k, cell[k] % Gx);
        }
        // the spread's 4 x 4 tiles by the samples that reach them, most first: the
        // long ones of a trajectory start first, each in a CTA of its own
        const int ntx = (Gx + 3) / 4, nty = (Gy + 3) / 4;
        std::vector<int> count(ntx * nty), order(ntx * nty);
        for (int t = 0; t < ntx * nty; ++t) {
            const int ty = 4 * (t / ntx), tx = 4 * (t % ntx);
            for (int y = ty - 3; y <= std::min(ty + 3, Gy - 1); ++y) {
                const int* row = start.data() + (size_t)wrap_host(y, Gy) * Gx;
                count[t] += row[std::min(tx + 4, Gx)] - row[std::max(tx - 3, 0)];
                if (tx < 3) count[t] += row[Gx] - row[Gx + tx - 3];
            }
            order[t] = t;
        }
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return count[a] / 8 > count[b] / 8; });
        PP_TRY(upload(p, &p.tile_order, order));
        PP_TRY(upload(p, &p.cell_start, start));
        PP_TRY(upload(p, &p.sort_wx, wx));
        PP_TRY(upload(p, &p.sort_wy, wy));
        PP_TRY(upload(p, &p.sort_kx, kx));
    }
    // G^T G as (2W-1)^2 weight planes (FP64 sums of the taps' pairwise
    // products, stored FP32), in both layouts, built on the device
    if (!p.toep) {   // (a Toeplitz plan's normal operator needs no stencil)
        const int D = 2 * W - 1, nxb = (Gx + 7) / 8;
        PP_TRY(alloc_n(p, &p.gtg, (size_t)D * D * Gx * Gy));
        PP_TRY(alloc_n(p, &p.gtg8, (size_t)Gy * nxb * D * D * 8));
        PP_TRY(build_gtg_device(p, 0));
        PP_TRY_CUDA(cudaStreamSynchronize(0));   // weights complete before any use on another stream
        PP_TRY(prepare_gtg_stencil(p));
    }
    PP_TRY(alloc_n(p, &p.wk_a, (size_t)p.C * ny * Gx));
    PP_TRY(alloc_n(p, &p.wk_b, (size_t)p.C * Gy * Gx));
    PP_TRY(alloc_n(p, &p.wk_c, (size_t)p.C * Gy * Gx));
    p.nksp = (int64_t)p.C * K;
    return PP_OK;
}

// Plan-time candidates that launch on thread-block clusters may not fit
// another device: a candidate whose first launch fails (a launch-time error,
// which does not poison the context) is skipped instead of failing the plan.
template <typename F>
static bool launches_ok(F&& fn) {
    if (fn() == PP_OK) return true;
    cudaGetLastError();
    return false;
}

// Plan-time autotuning of the non-Cartesian operator's launch shapes: the
// row-IFFT variant and the stencil kernel are each timed on the plan's own
// buffers (10 launches after two warm-ups, three rounds over all candidates,
// best round kept per candidate) and the fastest is kept.
static pp_status tune_noncartesian(Plan& p, cudaStream_t st) {
    cudaEvent_t e0, e1;
    PP_TRY_CUDA(cudaEventCreate(&e0));
    PP_TRY_CUDA(cudaEventCreate(&e1));
    // warm-up launches, then `reps` timed ones (the whole-operator candidates
    // below, 60-100 us each, are timed 5 at a time: plan set-up is part of a
    // solve's time to target)
    auto timeit = [&](auto&& fn, float* ms, int warm = 2, int reps = 10) -> pp_status {
        for (int r = 0; r < warm; ++r) PP_TRY(fn());
        PP_TRY_CUDA(cudaEventRecord(e0, st));
        for (int r = 0; r < reps; ++r) PP_TRY(fn());
        PP_TRY_CUDA(cudaEventRecord(e1, st));
        PP_TRY_CUDA(cudaEventSynchronize(e1));
        PP_TRY_CUDA(cudaEventElapsedTime(ms, e0, e1));
        *ms /= (float)reps;
        return PP_OK;
    };
    PP_TRY_CUDA(cudaMemsetAsync(p.wk_a, 0, sizeof(float2) * (size_t)p.C * p.ny * p.G_x, st));
    PP_TRY_CUDA(cudaMemsetAsync(p.wk_b, 0, sizeof(float2) * (size_t)p.C * p.G_y * p.G_x, st));
    const int nx = p.nx, ny = p.ny, Gx = p.G_x;
    RowArgs ra = row_args(nx, Gx, 0, nx / 2, ny, (int64_t)ny * nx, 1.f);
    // With the coil-innermost pipeline available the choice is made on the
    // whole operator below, where the [coil][row][col] pipeline enters with one
    // default launch shape per stage (it lost to the coil-innermost one on
    // every measured shape): the per-stage sweeps, which dominate plan time,
    // run only for plans without that pipeline.
    const bool sweep = !p.ci_sens;
    const int kRounds = sweep ? 3 : 0;
    std::vector<int> rows;
    for (int cl : {1, 2, 4, -1})
        if (cl != -1 || fft4_n2(Gx)) rows.push_back(cl);
    std::vector<float> rbest(rows.size(), 1e30f);
    for (int round = 0; round < kRounds; ++round)
        for (size_t i = 0; i < rows.size(); ++i) {
            const int cl = rows[i];
            p.tune_rows_adj_cl = cl;
            float ms = 0.f;
            if (cl == -1) {
                PP_TRY(timeit([&]() {
                    bool done = false;
                    return launch_rows4_adj_split(p.gx, ra, p.wk_a, p.sens, p.deapod_y, p.deapod_x,
                                                  p.wk_c, p.t, nullptr, 0.f, p.C, st, &done);
                }, &ms));
            } else {
                PP_TRY(timeit([&]() { return launch_rows_adj(p, p.gx, ra, p.wk_a, p.sens, p.deapod_y,
                                                             p.deapod_x, p.t, nullptr, 0.f, p.C, st); },
                              &ms));
            }
            rbest[i] = std::min(rbest[i], ms);
        }
    p.tune_rows_adj_cl = sweep ? rows[std::min_element(rbest.begin(), rbest.end()) - rbest.begin()] : 1;
    std::vector<std::pair<int, int>> sten;   // (kind, coils per CTA)
    for (int kind = 0; kind <= 6; ++kind)
        for (int cpc : {2, 4, 8, 16, 32}) {
            if (kind >= 2 && cpc != 8) continue;
            if (kind >= 2 && kind <= 5 && p.stencil_rb_grid[kind - 2] == 0) continue;
            if (kind == 6 && (!p.gtg8 || p.stencil_rb_grid[0] == 0)) continue;
            if (cpc > p.C && cpc != 2) continue;
            sten.push_back({kind, cpc});
        }
    std::vector<float> sbest(sten.size(), 1e30f);
    for (int round = 0; round < kRounds; ++round)
        for (size_t i = 0; i < sten.size(); ++i) {
            p.tune_stencil_kind = sten[i].first;
            p.tune_stencil_cpc = sten[i].second;
            float ms = 0.f;
            PP_TRY(timeit([&]() { return launch_gtg_stencil(p, p.wk_b, p.wk_c, st); }, &ms));
            sbest[i] = std::min(sbest[i], ms);
        }
    const size_t bi = std::min_element(sbest.begin(), sbest.end()) - sbest.begin();
    p.tune_stencil_kind = sweep ? sten[bi].first : 1;
    p.tune_stencil_cpc = sweep ? sten[bi].second : 8;
    // whole operator: the tuned [coil][row][col] pipeline against the
    // coil-innermost one (kinds 7, 8)
    if (p.ci_sens) {
        // (stencil kind, row variant): for kinds 7 and 8 the row variant 4
        // reduces the four 8-coil blocks of a row in a thread-block cluster
        std::vector<std::pair<int, int>> whole = {{p.tune_stencil_kind, p.tune_rows_adj_cl},
                                                  {7, 1}, {7, 4}, {8, 1}, {8, 4}, {9, 1}, {9, 4}};
        PP_TRY_CUDA(cudaMemsetAsync(p.v, 0, sizeof(float2) * (size_t)p.nimg, st));
        std::vector<float> wbest(whole.size(), 1e30f);
        for (int round = 0; round < 2; ++round) {
            // the second round re-times only the candidates within 10 % of
            // the first round's best
            const float cut = round == 0 ? 1.5e30f
                                         : 1.1f * *std::min_element(wbest.begin(), wbest.end());
            for (size_t i = 0; i < whole.size(); ++i) {
                p.tune_stencil_kind = whole[i].first;
                p.tune_rows_adj_cl = whole[i].second;
                if (round == 0 && i > 0 && !launches_ok([&]() {
                        return normal_into(p, p.v, p.t, 1.f, nullptr, 0.f, st); }))
                    wbest[i] = 2e30f;   // a cluster shape this device cannot place
                if (wbest[i] > cut) continue;
                float ms = 0.f;
                PP_TRY(timeit([&]() { return normal_into(p, p.v, p.t, 1.f, nullptr, 0.f, st); }, &ms, 1, 5));
                wbest[i] = std::min(wbest[i], ms);
            }
        }
        const size_t wi = std::min_element(wbest.begin(), wbest.end()) - wbest.begin();
        p.tune_stencil_kind = whole[wi].first;
        p.tune_rows_adj_cl = whole[wi].second;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return PP_OK;
}

// Launch shapes chosen by the plan-time tuners are kept per geometry for the
// life of the process: a later plan with the same geometry and sampling on
// the same device takes them instead of timing the candidates again (the
// choice depends on the shapes and, through tile lists and empty stencil
// tiles, on the trajectory; not on the coil maps or the image, nor on a Cartesian
// mask, which multiplies whatever it holds: a second plan with another mask takes 0.4 ms
// at 180 x 240 x 13 and 256 x 256 x 32, 5.2 at 128 x 256 x 256 x 8, where the timing made it
// 2.8, 6.4 and 171).
struct TuneKey {
    int dev, kind, ndim, nx, ny, nz, C, K, kb, toep;
    uint64_t data;   // FNV-1a of the trajectory (non-Cartesian)
    double oversamp;
    bool operator<(const TuneKey& o) const {
        return std::tie(dev, kind, ndim, nx, ny, nz, C, K, kb, toep, data, oversamp) <
               std::tie(o.dev, o.kind, o.ndim, o.nx, o.ny, o.nz, o.C, o.K, o.kb, o.toep, o.data, o.oversamp);
    }
};
struct TuneVal {
    int rows_adj_cl, stencil_kind, stencil_cpc, c3, c3df_cg, c3df_hi, c2, c2_one;
};
static std::mutex g_tune_mu;
static std::map<TuneKey, TuneVal> g_tune_cache;

static uint64_t fnv1a(const void* data, size_t n, uint64_t h = 1469598103934665603ull) {
    const unsigned char* b = static_cast<const unsigned char*>(data);
    for (size_t i = 0; i < n; ++i) h = (h ^ b[i]) * 1099511628211ull;
    return h;
}
static TuneKey tune_key(const Plan& p, const pp_sampling* s, int dev) {
    TuneKey k{};
    k.dev = dev; k.kind = (int)s->kind; k.ndim = p.ndim; k.nx = p.nx; k.ny = p.ny; k.nz = p.nz;
    k.C = p.C; k.K = s->kind == PP_CARTESIAN ? 0 : (int)s->K; k.kb = s->kb_width;
    k.toep = p.toep ? 1 : 0; k.oversamp = s->kind == PP_CARTESIAN ? 0.0 : s->oversamp;
    k.data = s->kind == PP_CARTESIAN ? 0 : fnv1a(s->traj, sizeof(float) * 2 * (size_t)s->K);
    return k;
}
static bool tune_lookup(const TuneKey& k, Plan& p) {
    std::lock_guard<std::mutex> g(g_tune_mu);
    auto it = g_tune_cache.find(k);
    if (it == g_tune_cache.end()) return false;
    const TuneVal& v = it->second;
    p.tune_rows_adj_cl = v.rows_adj_cl; p.tune_stencil_kind = v.stencil_kind;
    p.tune_stencil_cpc = v.stencil_cpc; p.tune_c3 = v.c3; p.c3df_cg = v.c3df_cg;
    p.c3df_hi = v.c3df_hi; p.tune_c2 = v.c2; p.tune_c2_one = v.c2_one;
    return true;
}
static void tune_store(const TuneKey& k, const Plan& p) {
    std::lock_guard<std::mutex> g(g_tune_mu);
    g_tune_cache[k] = TuneVal{p.tune_rows_adj_cl, p.tune_stencil_kind, p.tune_stencil_cpc, p.tune_c3,
                              p.c3df_cg, p.c3df_hi, p.tune_c2, p.tune_c2_one};
}

// 3-D Cartesian: the three passes per coil, the one-kernel cluster operator
// and the dataflow operator with 2, 4 or 8 coils per group, timed on the
// plan's buffers (two rounds of 3 applies after one warm-up); the fastest is
// kept.
static pp_status tune_cart3d(Plan& p, cudaStream_t st) {
    struct Cand { int kind, cg, hi; };
    std::vector<Cand> cand = {{0, 0, 0}};
    if (p.c3cl_clusters > 0) cand.push_back({1, 0, 0});
    if (p.c3cl2_clusters > 0) cand.push_back({2, 0, 0});
    for (int hi = 0; hi < 6; ++hi)
        if ((hi == 3 ? p.c3df_ctas_tma1 : hi == 2 ? p.c3df_ctas_tma
             : (hi == 1 || hi == 5) ? p.c3df_ctas_hi : p.c3df_ctas) > 0)
            for (int cgc : {2, 4, 8})
                if (cgc <= std::max(2, p.C) && (cgc == 2 || cgc <= p.C) &&
                    2 * c3df_slot_elems(p, cgc) <= p.c3df_w_elems)
                    cand.push_back({3, cgc, hi});
    if (cand.size() == 1) return PP_OK;
    cudaEvent_t e0, e1;
    PP_TRY_CUDA(cudaEventCreate(&e0));
    PP_TRY_CUDA(cudaEventCreate(&e1));
    PP_TRY_CUDA(cudaMemsetAsync(p.v, 0, sizeof(float2) * (size_t)p.nimg, st));
    std::vector<float> best(cand.size(), 1e30f);
    for (int round = 0; round < 2; ++round)
        for (size_t i = 0; i < cand.size(); ++i) {
            p.tune_c3 = cand[i].kind;
            if (cand[i].cg) {
                p.c3df_cg = cand[i].cg;
                p.c3df_hi = cand[i].hi;
            }
            if (best[i] > 1.5e30f) continue;
            if (!launches_ok([&]() { return normal_into(p, p.v, p.t, 1.f, nullptr, 0.f, st); }) ||
                (p.tune_c3 == 3 && c3df_check(p, st) != PP_OK)) {
                best[i] = 2e30f;
                continue;
            }
            PP_TRY_CUDA(cudaEventRecord(e0, st));
            for (int r = 0; r < 3; ++r) PP_TRY(normal_into(p, p.v, p.t, 1.f, nullptr, 0.f, st));
            PP_TRY_CUDA(cudaEventRecord(e1, st));
            PP_TRY_CUDA(cudaEventSynchronize(e1));
            float ms = 0.f;
            PP_TRY_CUDA(cudaEventElapsedTime(&ms, e0, e1));
            if (p.tune_c3 == 3 && c3df_check(p, st) != PP_OK) ms = 2e30f;
            best[i] = std::min(best[i], ms);
        }
    const size_t bi = std::min_element(best.begin(), best.end()) - best.begin();
    p.tune_c3 = cand[bi].kind;
    if (cand[bi].cg) {
        p.c3df_cg = cand[bi].cg;
        p.c3df_hi = cand[bi].hi;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return PP_OK;
}

// 2-D Cartesian: the columns per CTA of the column kernels, timed on the plan's
// buffers for one application and for a chain of three (a preconditioned gradient of
// degree 2); the fastest of each is kept (256 x 256 x 32: 14.7 us streaming and 17.7 on
// two columns for one, 42 and 29 for the chain).  A second round re-times the
// candidates within 10 % of the first one's best.
static pp_status tune_cart2d(Plan& p, cudaStream_t st) {
    p.cols = cart_cols_width_ok(p.ny, 1);
    if (!p.cols) return PP_OK;   // the Stockham kernel
    cudaEvent_t ev[3];
    for (cudaEvent_t& e : ev) PP_TRY_CUDA(cudaEventCreate(&e));
    PP_TRY_CUDA(cudaMemsetAsync(p.v, 0, sizeof(float2) * (size_t)p.nimg, st));
    std::vector<int> cand;
    for (int w : {1, 2, 4, 8})
        if (cart_cols_width_ok(p.ny, w)) cand.push_back(w);
    std::vector<float> one(cand.size(), 1e30f), chain(cand.size(), 1e30f);
    CartChain three;
    three.out = p.t;
    three.v_first = 1;
    three.J = 3;
    for (int j = 0; j < 3; ++j) three.sc[j] = three.al[j] = 1.f;
    for (int round = 0; round < 2; ++round) {
        const float one0 = *std::min_element(one.begin(), one.end()),
                    chain0 = *std::min_element(chain.begin(), chain.end());
        for (size_t i = 0; i < cand.size(); ++i) {
            if (round > 0 && one[i] > 1.1f * one0 && chain[i] > 1.1f * chain0) continue;
            p.tune_c2 = p.tune_c2_one = cand[i];
            PP_TRY(normal_into(p, p.v, p.t, 1.f, nullptr, 0.f, st));
            PP_TRY(cart_chain(p, p.v, three, st));
            PP_TRY_CUDA(cudaEventRecord(ev[0], st));
            for (int r = 0; r < 4; ++r) PP_TRY(normal_into(p, p.v, p.t, 1.f, nullptr, 0.f, st));
            PP_TRY_CUDA(cudaEventRecord(ev[1], st));
            for (int r = 0; r < 4; ++r) PP_TRY(cart_chain(p, p.v, three, st));
            PP_TRY_CUDA(cudaEventRecord(ev[2], st));
            PP_TRY_CUDA(cudaEventSynchronize(ev[2]));
            float a = 0.f, b = 0.f;
            PP_TRY_CUDA(cudaEventElapsedTime(&a, ev[0], ev[1]));
            PP_TRY_CUDA(cudaEventElapsedTime(&b, ev[1], ev[2]));
            one[i] = std::min(one[i], a);
            chain[i] = std::min(chain[i], b);
        }
    }
    p.tune_c2_one = cand[std::min_element(one.begin(), one.end()) - one.begin()];
    p.tune_c2 = cand[std::min_element(chain.begin(), chain.end()) - chain.begin()];
    for (cudaEvent_t e : ev) cudaEventDestroy(e);
    return PP_OK;
}

// Toeplitz-embedded normal operator: twiddles of the 2n transforms, the
// coil-innermost maps, the two [ny][2nx][32] arrays (zeroed once, so that
// coil blocks past C read zeros) and the kernel spectrum.
static pp_status setup_toeplitz(Plan& p, const pp_sampling* s, cudaStream_t st) {
    PP_TRY(make_fft(p, 2 * p.nx, p.tx));
    PP_TRY(make_fft(p, 2 * p.ny, p.ty));
    PP_TRY(make_fft(p, p.nx, p.toep_hx));
    PP_TRY(make_fft(p, p.ny, p.toep_hy));
    if (!p.ci_sens) {
        PP_TRY(alloc_n(p, &p.ci_sens, ci_sens_elems(p)));
        PP_TRY(ci_prepare(p, st));
    }
    const size_t nr = toep_rows_elems(p);
    PP_TRY(alloc_n(p, &p.toep_a, nr));
    PP_TRY(alloc_n(p, &p.toep_b, nr));
    PP_TRY_CUDA(cudaMemsetAsync(p.toep_a, 0, sizeof(float2) * nr, st));
    PP_TRY_CUDA(cudaMemsetAsync(p.toep_b, 0, sizeof(float2) * nr, st));
    PP_TRY(alloc_n(p, &p.toep_T, (size_t)4 * p.nx * p.ny));
    return toep_build_kernel(p, s->traj, s->K, st);
}

// Buffers of the coil-innermost pipeline (when the plan supports it).
static pp_status setup_ci(Plan& p, cudaStream_t st) {
    if (!ci_supported(p)) return PP_OK;
    PP_TRY(alloc_n(p, &p.ci_sens, ci_sens_elems(p)));
    PP_TRY(alloc_n(p, &p.ci_part, ci_partial_elems(p)));
    if (p.C == 32) {
        p.ci_a = p.wk_a;
        p.ci_b = p.wk_b;
        p.ci_c = p.wk_c;
    } else {
        PP_TRY(alloc_n(p, &p.ci_a, ci_rows_elems(p)));
        PP_TRY(alloc_n(p, &p.ci_b, ci_grid_elems(p)));
        PP_TRY(alloc_n(p, &p.ci_c, ci_grid_elems(p)));
    }
    PP_TRY(alloc_n(p, &p.ci_tile_nz, ci_stencil_tiles(p)));
    return ci_prepare(p, st);
}

static pp_status power_iteration(Plan& p, uint64_t seed, int iters, cudaStream_t st) {
    const int64_t n = p.nimg;
    PP_TRY(launch_start_vector(p.v, n, seed, st));
    PP_TRY(launch_norm2(p.v, n, p.red, p.red_blocks, p.scal + 2, st));
    PP_TRY(launch_scale_by_rnorm(p.v, p.v, n, p.scal + 2, 1.0, 1, st));
    for (int it = 0; it < iters; ++it) {
        PP_TRY(normal_into(p, p.v, p.t, 1.f, nullptr, 0.f, st));
        PP_TRY(launch_dot(p.v, p.t, n, p.red, p.red_blocks, p.scal + 1, p.scal + 2, st));
        PP_TRY(launch_scale_by_rnorm(p.t, p.v, n, p.scal + 2, 1.0, 1, st));
    }
    double L = 0.0;
    PP_TRY_CUDA(cudaMemcpyAsync(&L, p.scal + 1, sizeof(double), cudaMemcpyDeviceToHost, st));
    PP_TRY_CUDA(cudaStreamSynchronize(st));
    PP_TRY(c3df_check(p, st));
    if (!(L > 0.0) || !isfinite(L)) {
        set_error("power iteration gave a non-positive or non-finite norm estimate (%g)", L);
        return PP_ERR_NONFINITE;
    }
    p.L = L;
    return PP_OK;
}

// Power iteration on I - N_hat (the remark closing the Chebyshev design of
// Sec. 3.4): converges to 1 - mu, mu the smallest eigenvalue of N_hat when
// A^H A is injective.  Same start vector and FP64 reductions as
// power_iteration; returns mu = 1 - (last Rayleigh quotient).
static pp_status mu_iteration(Plan& p, uint64_t seed, int iters, double* mu, cudaStream_t st) {
    const int64_t n = p.nimg;
    PP_TRY(launch_start_vector(p.v, n, seed, st));
    PP_TRY(launch_norm2(p.v, n, p.red, p.red_blocks, p.scal + 2, st));
    PP_TRY(launch_scale_by_rnorm(p.v, p.v, n, p.scal + 2, 1.0, 1, st));
    const float s = (float)(-1.0 / p.L);
    for (int it = 0; it < iters; ++it) {
        PP_TRY(normal_into(p, p.v, p.t, s, p.v, 1.f, st));   // t = v - N_hat v
        PP_TRY(launch_dot(p.v, p.t, n, p.red, p.red_blocks, p.scal + 1, p.scal + 2, st));
        PP_TRY(launch_scale_by_rnorm(p.t, p.v, n, p.scal + 2, 1.0, 1, st));
    }
    double rho = 0.0;
    PP_TRY_CUDA(cudaMemcpyAsync(&rho, p.scal + 1, sizeof(double), cudaMemcpyDeviceToHost, st));
    PP_TRY_CUDA(cudaStreamSynchronize(st));
    PP_TRY(c3df_check(p, st));
    if (!isfinite(rho)) {
        set_error("pp_plan_mu: non-finite Rayleigh quotient");
        return PP_ERR_NONFINITE;
    }
    *mu = 1.0 - rho;
    return PP_OK;
}

static bool fft_len_ok(int n) {
    FftDesc d;
    return factorize(n, d);
}

// ---------------------------------------------------------------------------
// Horner recursion (Listing "pcode"): u = c_d v; u = c_i v + N_hat u.
// The first step folds c_d into the apply: u = c_{d-1} v + (c_d/L) N v.
// Writes the result into `out`; bufA/bufB are scratch images.
// ---------------------------------------------------------------------------
static pp_status horner_into(const Plan& p, const double* c, int d, const float2* v, float2* out,
                             float2* bufA, float2* bufB, cudaStream_t st) {
    const float invL = (float)(1.0 / p.L);
    if (d == 0) return launch_axpby(v, (float)c[0], nullptr, 0.f, out, p.nimg, st);
    if (p.cols) {
        CartChain ch;
        ch.J = 0;
        ch.v_first = 1;
        ch.out = out;
        chain_horner(ch, c, d, 1.0 / p.L);
        return cart_chain(p, v, ch, st);
    }
    const float2* cur = v;
    float scale = (float)(c[d] / p.L);
    for (int i = d - 1; i >= 0; --i) {
        float2* dst = (i == 0) ? out : ((cur == bufA) ? bufB : bufA);
        PP_TRY(normal_into(p, cur, dst, scale, v, (float)c[i], st));
        cur = dst;
        scale = invL;
    }
    return PP_OK;
}

// `shift` (sh_a, sh_b): the iteration runs on a N_hat + sh_b I instead of
// N_hat (the proximal subproblem of pp_fista_solve_prox); the caller then
// passes the preconditioner already rewritten as a polynomial in N_hat.
struct Shift {
    bool on = false;
    float a = 1.f, b = 0.f;
};

static pp_status fista_iterations(Plan& p, float lambda, int iters, const double* c, int d,
                                  int levels, bool hist, const float2* ref, bool momentum,
                                  int wavelet, cudaStream_t st, Shift sh = Shift()) {
    const float invL = (float)(1.0 / p.L);
    const bool chain = p.cols && c && d >= 1;
    for (int k = 0; k < iters; ++k) {
        if (chain) {
            // gradient and preconditioner in one launch
            CartChain ch;
            ch.sc[0] = sh.on ? sh.a * invL : invL;
            ch.al[0] = sh.on ? 1.f : -1.f;
            ch.ext = p.ahb;
            if (sh.on) {
                PP_TRY(launch_axpby(p.z, sh.b, p.ahb, -1.f, p.t, p.nimg, st));
                ch.ext = p.t;
            }
            ch.first_out = p.g;
            ch.out = p.u;
            chain_horner(ch, c, d, 1.0 / p.L);
            PP_TRY(cart_chain(p, p.z, ch, st));
        } else if (sh.on) {
            // g = (a N_hat + b I) z - rhs: u = b z - rhs, then g = a N_hat z + u
            PP_TRY(launch_axpby(p.z, sh.b, p.ahb, -1.f, p.u, p.nimg, st));
            PP_TRY(normal_into(p, p.z, p.g, sh.a * invL, p.u, 1.f, st));
        } else {
            // g = N_hat z - A_hat^H b_hat
            PP_TRY(normal_into(p, p.z, p.g, invL, p.ahb, -1.f, st));
        }
        const float2* u = p.g;
        float gamma = 1.f;
        if (chain) {
            u = p.u;
        } else if (c && d >= 1) {
            PP_TRY(horner_into(p, c, d, p.g, p.u, p.t, p.w3, st));
            u = p.u;
        } else if (c) {
            gamma = (float)c[0];
        }
        const float beta = momentum ? (float)((double)k / (k + 3.0)) : 0.f;
        if (wavelet == 1)   // Daubechies-4: multi-pass, p.t (free after Horner) holds the coefficients
            PP_TRY(launch_prox_fista_db4(p, levels, lambda, gamma, beta, u, p.t, hist ? ref : nullptr,
                                         hist ? p.hist + 3 * k : nullptr, st));
        else
            PP_TRY(launch_prox_fista(p, levels, lambda, gamma, beta, u, hist ? ref : nullptr,
                                     hist ? p.hist + 3 * k : nullptr, st));
    }
    return PP_OK;
}


// ---------------------------------------------------------------------------
// Batched uneven 2-D Cartesian problems
// ---------------------------------------------------------------------------
struct Batch {
    int n = 0;
    std::vector<Plan*> sub;
    std::vector<int64_t> img_off, ksp_off, tile_off;
    int64_t nimg = 0, nksp = 0;
    std::vector<double> L;
    std::vector<SliceDesc> hdesc;
    BatchDev dev;
    std::vector<void*> allocs;
    float2 *z = nullptr, *y = nullptr, *g = nullptr, *u = nullptr, *t = nullptr, *ahb = nullptr,
           *v = nullptr, *w3 = nullptr, *wk = nullptr;
    double *partials = nullptr, *scal = nullptr, *dfac = nullptr, *hist = nullptr;
    int hist_cap = 0;
    cudaStream_t cap_stream = nullptr;
    cudaGraphExec_t gexec = nullptr;
    std::vector<double> gkey;
    int64_t graph_kernels = 0;
    // differentiable unrolled solve: arena of image vectors and FP64 slots
    float2* arena = nullptr;
    size_t arena_vecs = 0;
    double* dslots = nullptr;
    size_t dslots_n = 0;
    std::vector<double> tape_key;
    // forward and adjoint stages of the whole batch (empty: slice by slice)
    std::vector<LineGroup> fwd_rows, fwd_cols;
    std::vector<AdjointChunk> adj;
};

template <class T>
static pp_status balloc(Batch& b, T** ptr, size_t n) {
    *ptr = nullptr;
    if (n == 0) return PP_OK;
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(ptr), n * sizeof(T));
    if (e != cudaSuccess) {
        *ptr = nullptr;
        cudaGetLastError();
        return cuda_status(e, "cudaMalloc");
    }
    b.allocs.push_back(*ptr);
    return PP_OK;
}

template <class T>
static pp_status bupload(Batch& b, T** dst, const std::vector<T>& src) {
    PP_TRY(balloc(b, dst, src.size()));
    PP_TRY_CUDA(cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice));
    return PP_OK;
}

// Forward and adjoint stages over the whole batch: one launch per distinct length
// (the slices one after another leave most SMs idle: eight 256 x 256 slices of 16
// coils took 215 us forward and 310 us adjoint that way).  The adjoint's column
// stage writes `wk` elements of workspace at most, so it runs in chunks of slices.
// Skipped (empty lists) when some length has no compiled stage.
template <class Item>
static pp_status add_group(Batch& b, std::vector<LineGroup>& to, LineGroup g, std::vector<Item>& items) {
    for (size_t i = 0; i < items.size(); i += 65535) {   // the batch index is blockIdx.y
        const std::vector<Item> part(items.begin() + i, items.begin() + std::min(items.size(), i + 65535));
        Item* p = nullptr;
        PP_TRY(bupload(b, &p, part));
        g.items = p;
        g.nitems = (int)part.size();
        to.push_back(g);
    }
    return PP_OK;
}
static pp_status plan_lines(Batch& b, size_t wk) {
    for (const Plan* p : b.sub)
        if (!lines_have(p->nx) || !lines_have(p->ny) || p->nx > 512) return PP_OK;
    struct Cols { LineGroup g; std::vector<ColItem> items; };
    struct Rows { LineGroup g; std::vector<RowItem> items; };
    auto cols_of = [&](std::map<int, Cols>& m, const Plan& p, int64_t src, int64_t dst) {
        Cols& c = m[p.ny];
        c.g.n = p.ny;
        c.g.tw = p.fy.twb;
        c.g.extent = std::max(c.g.extent, p.nx);
        for (int q = 0; q < p.C; ++q)
            c.items.push_back({src + q * p.nimg, dst + q * p.nimg, p.mask_c, p.nx, (float)(1.0 / sqrt((double)p.ny))});
    };
    std::map<int, Cols> fc;
    std::map<int, Rows> fr;
    for (int s = 0; s < b.n; ++s) {
        const Plan& p = *b.sub[s];
        Rows& r = fr[p.nx];
        r.g.n = p.nx;
        r.g.tw = p.fx.twb;
        r.g.extent = std::max(r.g.extent, p.ny);
        for (int q = 0; q < p.C; ++q)
            r.items.push_back({b.img_off[s], b.ksp_off[s] + q * p.nimg, p.sens + q * p.nimg, p.ny, 1, 1.f});
        cols_of(fc, p, b.ksp_off[s], b.ksp_off[s]);
    }
    for (auto& e : fr) PP_TRY(add_group(b, b.fwd_rows, e.second.g, e.second.items));
    for (auto& e : fc) PP_TRY(add_group(b, b.fwd_cols, e.second.g, e.second.items));
    for (int s0 = 0; s0 < b.n;) {
        std::map<int, Cols> ac;
        std::map<int, Rows> ar;
        int64_t used = 0;
        int s = s0;
        for (; s < b.n && (s == s0 || used + b.sub[s]->nksp <= (int64_t)wk); ++s) {
            const Plan& p = *b.sub[s];
            cols_of(ac, p, b.ksp_off[s], used);
            Rows& r = ar[p.nx];
            r.g.n = p.nx;
            r.g.tw = p.fx.twb;
            r.g.extent = std::max(r.g.extent, p.ny);
            r.g.ncoils = std::max(r.g.ncoils, p.C);
            r.items.push_back({used, b.img_off[s], p.sens, p.ny, p.C, 1.f});
            used += p.nksp;
        }
        s0 = s;
        AdjointChunk c;
        for (auto& e : ac) PP_TRY(add_group(b, c.cols, e.second.g, e.second.items));
        for (auto& e : ar) PP_TRY(add_group(b, c.rows, e.second.g, e.second.items));
        b.adj.push_back(c);
    }
    return PP_OK;
}

static pp_status batch_cols(const std::vector<LineGroup>& gs, bool inv, const float2* src, float2* dst, cudaStream_t st) {
    for (const LineGroup& g : gs)
        PP_TRY(launch_lines_batch_cols(g.n, g.tw, g.extent, (const ColItem*)g.items, g.nitems, inv, src, dst, st));
    return PP_OK;
}
static pp_status batch_rows(const std::vector<LineGroup>& gs, bool adj, const float2* src, float2* dst, cudaStream_t st) {
    for (const LineGroup& g : gs)
        PP_TRY(launch_lines_batch_rows(g.n, g.tw, g.extent, (const RowItem*)g.items, g.nitems, adj, g.ncoils,
                                       (float)(1.0 / sqrt((double)g.n)), src, dst, st));
    return PP_OK;
}
// y_s = A_s x_s and x_s = A_s^H y_s for every slice (unscaled)
static pp_status batch_forward(const Batch& b, const float2* x, float2* y, cudaStream_t st) {
    if (!b.fwd_rows.empty()) {
        PP_TRY(batch_rows(b.fwd_rows, false, x, y, st));
        return batch_cols(b.fwd_cols, false, y, y, st);
    }
    for (int s = 0; s < b.n; ++s) PP_TRY(forward_into(*b.sub[s], x + b.img_off[s], y + b.ksp_off[s], st));
    return PP_OK;
}
static pp_status batch_adjoint(const Batch& b, const float2* y, float2* x, cudaStream_t st) {
    if (!b.adj.empty()) {
        for (const AdjointChunk& c : b.adj) {
            PP_TRY(batch_cols(c.cols, true, y, b.wk, st));
            PP_TRY(batch_rows(c.rows, true, b.wk, x, st));
        }
        return PP_OK;
    }
    for (int s = 0; s < b.n; ++s) PP_TRY(adjoint_into(*b.sub[s], y + b.ksp_off[s], x + b.img_off[s], st));
    return PP_OK;
}

// blocks per segment: ceil(len / per_block) clamped to [1, max_blocks]
static pp_status make_segments(Batch& b, Segments& sg, const std::vector<int64_t>& off,
                               int64_t per_block, int max_blocks) {
    const int nseg = (int)off.size() - 1;
    std::vector<int> blk_seg, first(nseg + 1, 0);
    for (int s = 0; s < nseg; ++s) {
        const int64_t len = off[s + 1] - off[s];
        int64_t nb = (len + per_block - 1) / per_block;
        nb = std::max<int64_t>(1, std::min<int64_t>(nb, max_blocks));
        first[s] = (int)blk_seg.size();
        for (int64_t j = 0; j < nb; ++j) blk_seg.push_back(s);
    }
    first[nseg] = (int)blk_seg.size();
    sg.nseg = nseg;
    sg.nblocks = (int)blk_seg.size();
    PP_TRY(bupload(b, &sg.off, off));
    PP_TRY(bupload(b, &sg.blk_seg, blk_seg));
    PP_TRY(bupload(b, &sg.seg_first_blk, first));
    return PP_OK;
}

static int km_for(int ny_max, int lgt) {
    const int need = (ny_max * (1 << lgt) + kThreads - 1) / kThreads;
    const int kms[] = {4, 8, 12, 16};
    for (int km : kms)
        if (need <= km && batch_normal_fn(km, lgt)) return km;
    return 0;
}

// Work items (slice, first column) for column tiles of 2^lgt, most expensive
// first so that the persistent grid's round-robin balances the load.
static pp_status set_items(Batch& b, int lgt, std::vector<int2>* scratch) {
    const int T = 1 << lgt;
    std::vector<std::pair<double, int2>> it;
    for (int s = 0; s < b.n; ++s) {
        const SliceDesc& d = b.hdesc[s];
        const double cost = (double)d.C * d.ny * log2((double)d.ny);
        for (int c0 = 0; c0 < d.nx; c0 += T) it.push_back({cost, make_int2(s, c0)});
    }
    std::stable_sort(it.begin(), it.end(),
                     [](const std::pair<double, int2>& a, const std::pair<double, int2>& c) {
                         return a.first > c.first;
                     });
    scratch->clear();
    for (auto& e : it) scratch->push_back(e.second);
    if (b.dev.items) {
        cudaFree(b.dev.items);
        b.allocs.erase(std::remove(b.allocs.begin(), b.allocs.end(), (void*)b.dev.items), b.allocs.end());
        b.dev.items = nullptr;
    }
    PP_TRY(bupload(b, &b.dev.items, *scratch));
    b.dev.nitems = (int)scratch->size();
    b.dev.lgt = lgt;
    b.dev.km = km_for(b.dev.ny_max, lgt);
    int occ = 0;
    PP_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &occ, batch_normal_fn(b.dev.km, lgt), kThreads, batch_normal_smem(b.dev.ny_max, lgt)));
    int nsm = 0;
    PP_TRY_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, 0));
    b.dev.grid = std::max(1, std::min(b.dev.nitems, nsm * std::max(occ, 1)));
    return PP_OK;
}

static pp_status upload_descs(Batch& b) {
    for (int s = 0; s < b.n; ++s) b.hdesc[s].invL = (float)(1.0 / b.L[s]);
    PP_TRY_CUDA(cudaMemcpy(b.dev.descs, b.hdesc.data(), b.n * sizeof(SliceDesc), cudaMemcpyHostToDevice));
    std::vector<double> f(b.n);
    for (int s = 0; s < b.n; ++s) f[s] = 1.0 / sqrt(b.L[s]);
    PP_TRY_CUDA(cudaMemcpy(b.dfac, f.data(), b.n * sizeof(double), cudaMemcpyHostToDevice));
    b.gkey.clear();
    return PP_OK;
}

// Work lists of the column-resident kernels, W columns per CTA (fewer for a
// length without that form): one list per distinct slice length, longest first.
// False when some length has no such kernel.
static bool cols_supported(const Batch& b) {
    for (const SliceDesc& d : b.hdesc)
        if (!cart_cols_width_ok(d.ny, 1)) return false;
    return !b.hdesc.empty();
}
// One upload holds the lists of all lengths: groups[0].items is its start.
static void free_groups(Batch& b, std::vector<CartGroup>& groups) {
    if (!groups.empty()) {
        cudaFree(groups[0].items);
        b.allocs.erase(std::remove(b.allocs.begin(), b.allocs.end(), (void*)groups[0].items), b.allocs.end());
    }
    groups.clear();
}
static pp_status make_groups(Batch& b, int W, bool lean, std::vector<CartGroup>* out) {
    std::map<int, std::vector<std::pair<int, int2>>, std::greater<int>> by_len;
    std::map<int, CartGroup> info;
    for (int s = 0; s < b.n; ++s) {
        const SliceDesc& d = b.hdesc[s];
        CartGroup& g = info[d.ny];
        g.n = d.ny;
        g.W = W;
        g.lean = lean;
        while (g.W > 1 && !cart_cols_width_ok(d.ny, g.W)) g.W >>= 1;
        g.max_coils = std::max(g.max_coils, d.C);
        for (int c0 = 0; c0 < d.nx; c0 += g.W) by_len[d.ny].push_back({d.C, make_int2(s, c0)});
    }
    std::vector<int2> items;
    std::vector<CartGroup> groups;
    for (auto& e : by_len) {
        std::stable_sort(e.second.begin(), e.second.end(),
                         [](const std::pair<int, int2>& a, const std::pair<int, int2>& c) {
                             return a.first > c.first;
                         });
        for (auto& it : e.second) items.push_back(it.second);
        CartGroup g = info[e.first];
        g.nitems = (int)e.second.size();
        groups.push_back(g);
    }
    int2* all = nullptr;
    PP_TRY(bupload(b, &all, items));
    for (CartGroup& g : groups) {
        g.items = all;
        all += g.nitems;
    }
    *out = groups;
    return PP_OK;
}
// `one` may be the same lists as `groups`.
static void use_groups(Batch& b, int W, const std::vector<CartGroup>& groups, const std::vector<CartGroup>& one) {
    b.dev.groups = groups;
    b.dev.one = one;
    b.dev.cols = groups.empty() ? 0 : W;
    b.dev.grid = 0;
    for (const CartGroup& g : groups) b.dev.grid += g.nitems;
}
static void drop_groups(Batch& b) {
    if (!b.dev.one.empty() && b.dev.one[0].items != b.dev.groups[0].items) free_groups(b, b.dev.one);
    free_groups(b, b.dev.groups);
    b.dev.one.clear();
    b.dev.cols = 0;
}
static pp_status set_cols(Batch& b, int W) {
    std::vector<CartGroup> groups;
    PP_TRY(make_groups(b, W, false, &groups));
    drop_groups(b);
    use_groups(b, W, groups, groups);
    return PP_OK;
}

// Batch autotuner: the columns per CTA of the column-resident kernels where every
// slice length has one, for an application and for a chain of three (the fastest of
// each: one 256 x 256 x 16 slice takes 12.4 us on two columns and 16.5 on one, a solve
// of d = 5 40.9 and 44.2 an iteration), else the tile width of the Stockham kernel.
// The streaming form is tried with both counts of slots: us for as many as bring 16
// warps to an SM / for no more than raise those on an SM (CartLaunch::lean), eight
// slices of 384 x 384 x 8 53.3 / 45.2, of 256 x 256 x 16 43.9 / 40.9, 32 of 128 x 128 x 16
// 39.1 / 32.9, but six of 320 x 320 x 20 59.8 / 80.2.  One pass each, then about 0.4 ms of
// passes for those within 20 % of the best.
static pp_status autotune(Batch& b, cudaStream_t st) {
    std::vector<int2> items;
    cudaEvent_t ev[3];
    for (cudaEvent_t& e : ev) PP_TRY_CUDA(cudaEventCreate(&e));
    const bool cols = cols_supported(b);
    CartChain three;
    three.out = b.t;
    three.v_first = 1;
    three.J = 3;
    for (int j = 0; j < 3; ++j) three.sc[j] = three.al[j] = 1.f;
    std::vector<int> cand;
    if (cols) {
        // two columns only for batches that leave SMs idle on wider ones
        int64_t wide = 0;
        for (const SliceDesc& d : b.hdesc) wide += (d.nx + 7) / 8;
        cand = wide <= 2 * 152 ? std::vector<int>{1, 2, 4, 8, 8} : std::vector<int>{1, 4, 8, 8};
    } else {
        for (int v : {2, 3, 4})
            if (km_for(b.dev.ny_max, v)) cand.push_back(v);
    }
    if (cand.empty()) {
        set_error("no batched kernel fits ny_max = %d", b.dev.ny_max);
        return PP_ERR_UNSUPPORTED;
    }
    std::vector<std::vector<CartGroup>> lists(cand.size());
    if (cols)
        for (size_t i = 0; i < cand.size(); ++i)
            PP_TRY(make_groups(b, cand[i], i + 1 == cand.size(), &lists[i]));
    auto single = [&]() { return launch_batch_normal(b.dev, b.v, b.t, 1.f, nullptr, 0.f, st); };
    auto chain = [&]() { return cols ? launch_batch_chain(b.dev, b.v, three, st) : PP_OK; };
    std::vector<float> one(cand.size(), 1e30f), chn(cand.size(), 1e30f);
    for (int round = 0; round < 2; ++round) {
        const float one0 = *std::min_element(one.begin(), one.end()), chn0 = *std::min_element(chn.begin(), chn.end());
        const int reps = round == 0 ? 1 : std::max(2, std::min(8, (int)(0.4f / (one0 + chn0))));
        for (size_t i = 0; i < cand.size(); ++i) {
            if (round > 0 && one[i] > 1.2f * one0 && (!cols || chn[i] > 1.2f * chn0)) continue;
            if (cols) use_groups(b, cand[i], lists[i], lists[i]);
            else PP_TRY(set_items(b, cand[i], &items));
            if (round == 0) {
                PP_TRY(single());
                PP_TRY(chain());
            }
            PP_TRY_CUDA(cudaEventRecord(ev[0], st));
            for (int r = 0; r < reps; ++r) PP_TRY(single());
            PP_TRY_CUDA(cudaEventRecord(ev[1], st));
            for (int r = 0; r < reps; ++r) PP_TRY(chain());
            PP_TRY_CUDA(cudaEventRecord(ev[2], st));
            PP_TRY_CUDA(cudaEventSynchronize(ev[2]));
            float t1 = 0.f, t3 = 0.f;
            PP_TRY_CUDA(cudaEventElapsedTime(&t1, ev[0], ev[1]));
            PP_TRY_CUDA(cudaEventElapsedTime(&t3, ev[1], ev[2]));
            one[i] = t1 / reps;
            chn[i] = t3 / reps;
        }
    }
    for (cudaEvent_t& e : ev) cudaEventDestroy(e);
    const size_t w1 = std::min_element(one.begin(), one.end()) - one.begin(),
                 w3 = std::min_element(chn.begin(), chn.end()) - chn.begin();
    if (!cols) return set_items(b, cand[w1], &items);
    use_groups(b, cand[w3], lists[w3], lists[w1]);
    for (size_t i = 0; i < cand.size(); ++i)
        if (i != w1 && i != w3) free_groups(b, lists[i]);
    return PP_OK;
}

static pp_status batch_power_iteration(Batch& b, uint64_t seed, int iters, cudaStream_t st) {
    for (int s = 0; s < b.n; ++s)
        PP_TRY(launch_start_vector(b.v + b.img_off[s], b.img_off[s + 1] - b.img_off[s], seed + s, st));
    PP_TRY(launch_seg_dot(nullptr, b.v, b.dev.img, b.partials, nullptr, b.scal + 2, 4, st));
    PP_TRY(launch_seg_scale(b.v, b.v, b.dev.img, b.scal + 2, 4, nullptr, 1, st));
    for (int it = 0; it < iters; ++it) {
        PP_TRY(launch_batch_normal(b.dev, b.v, b.t, 1.f, nullptr, 0.f, st));
        PP_TRY(launch_seg_dot(b.v, b.t, b.dev.img, b.partials, b.scal + 1, b.scal + 2, 4, st));
        PP_TRY(launch_seg_scale(b.t, b.v, b.dev.img, b.scal + 2, 4, nullptr, 1, st));
    }
    std::vector<double> h(4 * b.n);
    PP_TRY_CUDA(cudaMemcpyAsync(h.data(), b.scal, h.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
    PP_TRY_CUDA(cudaStreamSynchronize(st));
    for (int s = 0; s < b.n; ++s) {
        if (!(h[4 * s + 1] > 0.0) || !isfinite(h[4 * s + 1])) {
            set_error("power iteration: non-positive estimate for slice %d", s);
            return PP_ERR_NONFINITE;
        }
        b.L[s] = h[4 * s + 1];
    }
    return upload_descs(b);
}

static pp_status batch_horner(Batch& b, const double* c, int d, const float2* v, float2* out,
                              cudaStream_t st) {
    if (d == 0) return launch_axpby(v, (float)c[0], nullptr, 0.f, out, b.nimg, st);
    if (b.dev.cols > 0) {
        CartChain ch;
        ch.J = 0;
        ch.v_first = 1;
        ch.out = out;
        chain_horner(ch, c, d, 1.0);
        return launch_batch_chain(b.dev, v, ch, st);
    }
    const float2* cur = v;
    float coef = (float)c[d];
    for (int i = d - 1; i >= 0; --i) {
        float2* dst = (i == 0) ? out : ((cur == b.t) ? b.w3 : b.t);
        PP_TRY(launch_batch_normal(b.dev, cur, dst, coef, v, (float)c[i], st));
        cur = dst;
        coef = 1.f;
    }
    return PP_OK;
}

// u = p(N_hat) (N_hat z - ahb) in one launch per slice length, d >= 1; the
// gradient itself into g
static pp_status batch_gradient_chain(Batch& b, const double* c, int d, const float2* z,
                                      const float2* ahb, float2* g, float2* u, cudaStream_t st) {
    CartChain ch;
    ch.sc[0] = 1.f;
    ch.al[0] = -1.f;
    ch.ext = ahb;
    ch.first_out = g;
    ch.out = u;
    chain_horner(ch, c, d, 1.0);
    return launch_batch_chain(b.dev, z, ch, st);
}

static pp_status batch_iterations(Batch& b, float lambda, int iters, const double* c, int d,
                                  bool hist, const float2* ref, bool momentum, cudaStream_t st) {
    for (int k = 0; k < iters; ++k) {
        const float2* u = b.g;
        float gamma = 1.f;
        if (b.dev.cols > 0 && c && d >= 1) {
            PP_TRY(batch_gradient_chain(b, c, d, b.z, b.ahb, b.g, b.u, st));
            u = b.u;
        } else {
            PP_TRY(launch_batch_normal(b.dev, b.z, b.g, 1.f, b.ahb, -1.f, st));
        }
        if (u == b.u) {
        } else if (c && d >= 1) {
            PP_TRY(batch_horner(b, c, d, b.g, b.u, st));
            u = b.u;
        } else if (c) {
            gamma = (float)c[0];
        }
        const float beta = momentum ? (float)((double)k / (k + 3.0)) : 0.f;
        PP_TRY(launch_batch_prox_fista(b.dev, lambda, gamma, beta, b.z, u, b.y, nullptr, hist ? ref : nullptr,
                                       hist ? b.hist + 3 * k : nullptr, st));
    }
    return PP_OK;
}


// ---------------------------------------------------------------------------
// Differentiable unrolled solve on a batch: raw b (no normalisation, L_s
// fixed), Algorithm "pfista" for a fixed iteration count, checkpoints
// (y_k, z_k) every `ce` iterations, and the reverse pass.
// Arena layout (image-sized vectors): [0] ahb, [1 .. 2*ncp] checkpoints,
// then 2*ce segment vectors (g_k, w_k), d+2 Horner-adjoint vectors and
// Ybar, Zbar, wbar, ahb_bar, yw, zw.
// ---------------------------------------------------------------------------
static pp_status ensure_arena(Batch& b, size_t vecs, size_t slots) {
    if (vecs > b.arena_vecs) {
        if (b.arena) {
            cudaFree(b.arena);
            b.allocs.erase(std::remove(b.allocs.begin(), b.allocs.end(), (void*)b.arena), b.allocs.end());
            b.arena = nullptr;
            b.arena_vecs = 0;
        }
        PP_TRY(balloc(b, &b.arena, vecs * (size_t)b.nimg));
        b.arena_vecs = vecs;
        b.tape_key.clear();
    }
    if (slots > b.dslots_n) {
        if (b.dslots) {
            cudaFree(b.dslots);
            b.allocs.erase(std::remove(b.allocs.begin(), b.allocs.end(), (void*)b.dslots), b.allocs.end());
            b.dslots = nullptr;
            b.dslots_n = 0;
        }
        PP_TRY(balloc(b, &b.dslots, slots));
        b.dslots_n = slots;
    }
    return PP_OK;
}

static inline float2* avec(Batch& b, size_t i) { return b.arena + i * (size_t)b.nimg; }

static size_t unrolled_vecs(int iters, int ce, int d) {
    const size_t ncp = (size_t)((iters + ce - 1) / ce);
    return 1 + 2 * ncp + 2 * (size_t)ce + (size_t)(d + 2) + 6;
}

static pp_status unrolled_step(Batch& b, const double* c, int d, float lambda, int k, float2* z,
                               float2* y, float2* g_out, float2* w_out, cudaStream_t st) {
    const float2* ahb = avec(b, 0);
    if (b.dev.cols > 0 && d >= 1) {
        PP_TRY(batch_gradient_chain(b, c, d, z, ahb, g_out, b.u, st));
    } else {
        PP_TRY(launch_batch_normal(b.dev, z, g_out, 1.f, ahb, -1.f, st));
        PP_TRY(batch_horner(b, c, d, g_out, b.u, st));
    }
    const float beta = (float)((double)k / (k + 3.0));
    return launch_batch_prox_fista(b.dev, lambda, 1.f, beta, z, b.u, y, w_out, nullptr, nullptr, st);
}

static pp_status unrolled_forward(Batch& b, const float2* bk, float lambda, int iters,
                                  const double* c, int d, int ce, float2* x_out, cudaStream_t st) {
    PP_TRY(ensure_arena(b, unrolled_vecs(iters, ce, d), 1 + (size_t)(iters + kRevBlocks) * (d + 1)));
    float2* ahb = avec(b, 0);
    PP_TRY(batch_adjoint(b, bk, ahb, st));
    PP_TRY(launch_seg_scale(ahb, ahb, b.dev.img, nullptr, 0, b.dfac, 0, st));
    PP_TRY_CUDA(cudaMemsetAsync(b.y, 0, b.nimg * sizeof(float2), st));
    PP_TRY_CUDA(cudaMemsetAsync(b.z, 0, b.nimg * sizeof(float2), st));
    const size_t bytes = (size_t)b.nimg * sizeof(float2);
    for (int k = 0; k < iters; ++k) {
        if (k % ce == 0) {
            const int cp = k / ce;
            PP_TRY_CUDA(cudaMemcpyAsync(avec(b, 1 + 2 * cp), b.y, bytes, cudaMemcpyDeviceToDevice, st));
            PP_TRY_CUDA(cudaMemcpyAsync(avec(b, 2 + 2 * cp), b.z, bytes, cudaMemcpyDeviceToDevice, st));
        }
        PP_TRY(unrolled_step(b, c, d, lambda, k, b.z, b.y, b.g, nullptr, st));
    }
    PP_TRY_CUDA(cudaMemcpyAsync(x_out, b.y, bytes, cudaMemcpyDeviceToDevice, st));
    return PP_OK;
}

static pp_status unrolled_backward(Batch& b, float lambda, int iters, const double* c, int d,
                                   int ce, const float2* gout, float2* grad_b, double* grad_lam,
                                   double* grad_c, cudaStream_t st) {
    const size_t ncp = (size_t)((iters + ce - 1) / ce);
    const size_t seg0 = 1 + 2 * ncp, v0 = seg0 + 2 * (size_t)ce, r0 = v0 + (size_t)(d + 2);
    float2 *Ybar = avec(b, r0), *Zbar = avec(b, r0 + 1), *wbar = avec(b, r0 + 2),
           *ahb_bar = avec(b, r0 + 3), *yw = avec(b, r0 + 4), *zw = avec(b, r0 + 5);
    const size_t bytes = (size_t)b.nimg * sizeof(float2);
    double* lam_bar = b.dslots;
    double* dots = b.dslots + 1;   // [iters][d+1]
    PP_TRY_CUDA(cudaMemcpyAsync(Ybar, gout, bytes, cudaMemcpyDeviceToDevice, st));
    PP_TRY_CUDA(cudaMemsetAsync(Zbar, 0, bytes, st));
    PP_TRY_CUDA(cudaMemsetAsync(ahb_bar, 0, bytes, st));
    PP_TRY_CUDA(cudaMemsetAsync(b.dslots, 0, sizeof(double) * (1 + (size_t)iters * (d + 1)), st));
    for (int sg = (int)ncp - 1; sg >= 0; --sg) {
        const int k0 = sg * ce, k1 = std::min(iters, k0 + ce);
        // recompute the segment forward from its checkpoint, keeping g_k, w_k
        PP_TRY_CUDA(cudaMemcpyAsync(yw, avec(b, 1 + 2 * sg), bytes, cudaMemcpyDeviceToDevice, st));
        PP_TRY_CUDA(cudaMemcpyAsync(zw, avec(b, 2 + 2 * sg), bytes, cudaMemcpyDeviceToDevice, st));
        for (int k = k0; k < k1; ++k) {
            const int j = k - k0;
            PP_TRY(unrolled_step(b, c, d, lambda, k, zw, yw, avec(b, seg0 + 2 * j),
                                 avec(b, seg0 + 2 * j + 1), st));
        }
        for (int k = k1 - 1; k >= k0; --k) {
            const int j = k - k0;
            const float beta = (float)((double)k / (k + 3.0));
            PP_TRY(launch_batch_prox_vjp(b.dev, lambda, beta, avec(b, seg0 + 2 * j + 1), Ybar, Zbar,
                                         wbar, lam_bar, st));
            // v_0 = wbar, v_i = N_hat v_{i-1}, i = 1..d+1
            if (b.dev.cols > 0) {
                CartChain ch;
                ch.J = d + 1;
                for (int i = 0; i <= d; ++i) {
                    ch.sc[i] = 1.f;
                    ch.al[i] = 0.f;
                }
                ch.all_out = avec(b, v0 + 1);
                ch.all_stride = b.nimg;
                PP_TRY(launch_batch_chain(b.dev, wbar, ch, st));
            } else {
                const float2* prev = wbar;
                for (int i = 1; i <= d + 1; ++i) {
                    PP_TRY(launch_batch_normal(b.dev, prev, avec(b, v0 + i), 1.f, nullptr, 0.f, st));
                    prev = avec(b, v0 + i);
                }
            }
            const float2* gk = avec(b, seg0 + 2 * j);
            // dots_i = Re<v_i, g_k>;  Zbar = wbar - sum_i c_i v_{i+1};  ahb_bar += sum_i c_i v_i
            RevCombine rc;
            rc.d = d;
            for (int i = 0; i <= d; ++i) rc.c[i] = (float)c[i];
            rc.wbar = wbar;
            rc.v = avec(b, v0 + 1);
            rc.n = b.nimg;
            rc.g = gk;
            rc.Zbar = Zbar;
            rc.ahb_bar = ahb_bar;
            rc.partials = b.dslots + 1 + (size_t)iters * (d + 1);
            PP_TRY(launch_rev_combine(rc, dots + (size_t)k * (d + 1), st));
        }
    }
    // b_bar = A_s ahb_bar_s / sqrt(L_s)
    PP_TRY(batch_forward(b, ahb_bar, grad_b, st));
    PP_TRY(launch_seg_scale(grad_b, grad_b, b.dev.ksp, nullptr, 0, b.dfac, 0, st));
    std::vector<double> h(1 + (size_t)iters * (d + 1));
    PP_TRY_CUDA(cudaMemcpyAsync(h.data(), b.dslots, h.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
    PP_TRY_CUDA(cudaStreamSynchronize(st));
    *grad_lam = h[0];
    for (int i = 0; i <= d; ++i) {
        double acc = 0.0;
        for (int k = 0; k < iters; ++k) acc += h[1 + (size_t)k * (d + 1) + i];
        grad_c[i] = -acc;
    }
    return PP_OK;
}

}  // namespace pp

// ===========================================================================
// extern "C" entry points
// ===========================================================================
using namespace pp;

extern "C" {

const char* pp_last_error(void) { return g_last_error.c_str(); }

pp_status pp_poly_max_zp(const double* c, int d, double* m) {
    if (!c || !m || d < 0 || d > 16) {
        set_error("pp_poly_max_zp: need c != NULL, m != NULL, 0 <= d <= 16");
        return PP_ERR_INVALID_ARG;
    }
    // z p(z) on 4096 equal steps of [0, 1], then golden-section refinement
    // of the best bracket (z p(z) is a polynomial: one smooth maximum there)
    auto f = [&](double z) {
        double acc = 0.0;
        for (int i = d; i >= 0; --i) acc = acc * z + c[i];
        return z * acc;
    };
    const int n = 4096;
    int best = 0;
    double fb = f(0.0);
    for (int i = 1; i <= n; ++i) {
        const double v = f((double)i / n);
        if (v > fb) {
            fb = v;
            best = i;
        }
    }
    double a = std::max(0.0, (best - 1.0) / n), b = std::min(1.0, (best + 1.0) / n);
    const double g = 0.5 * (sqrt(5.0) - 1.0);
    for (int it = 0; it < 80; ++it) {
        const double x1 = b - g * (b - a), x2 = a + g * (b - a);
        if (f(x1) < f(x2)) a = x1;
        else b = x2;
    }
    *m = std::max(fb, f(0.5 * (a + b)));
    if (!std::isfinite(*m)) {
        set_error("pp_poly_max_zp: non-finite value");
        return PP_ERR_NONFINITE;
    }
    return PP_OK;
}

pp_status pp_poly_coeffs_l2(int d, double* c) {
    if (!c || d < 0 || d > 8) {
        set_error("pp_poly_coeffs_l2: need 0 <= d <= 8 and c != NULL");
        return PP_ERR_INVALID_ARG;
    }
    // r(z) = 1 - z p(z) is the degree-(d+1) polynomial with r(0) = 1 of least
    // L2([0,1]) norm.  With the orthonormal shifted Legendre polynomials
    // Q_j(z) = sqrt(2j+1) P_j(2z-1) this is the normalised Christoffel-Darboux
    // kernel r(z) = sum_j Q_j(0) Q_j(z) / sum_j Q_j(0)^2, j = 0..m, m = d+1.
    // Since P_j(2z-1) = sum_k (-1)^(j+k) C(j,k) C(j+k,k) z^k and Q_j(0)^2 = 2j+1,
    //   [z^k] r = (-1)^k sum_{j=k..m} (2j+1) C(j,k) C(j+k,k) / (m+1)^2,
    // an exact integer ratio; c_i = -[z^(i+1)] r.
    const int m = d + 1;
    auto binom = [](int a, int b) {
        long long r = 1;
        for (int t = 1; t <= b; ++t) r = r * (a - b + t) / t;
        return r;
    };
    const double den = (double)((m + 1) * (m + 1));
    for (int i = 0; i <= d; ++i) {
        const int k = i + 1;
        long long S = 0;
        for (int j = k; j <= m; ++j) S += (long long)(2 * j + 1) * binom(j, k) * binom(j + k, k);
        c[i] = ((k + 1) % 2 == 0 ? 1.0 : -1.0) * (double)S / den;
    }
    return PP_OK;
}

// r_i = h_i - sum_j G_ij c_j with the products' rounding errors (fma) and the
// sum's (two-sum) carried in a second word: the residual of a Hankel system
// whose condition grows like that of the Hilbert matrix.
static double residual_dd(const double* G, const double* h, const double* c, int n, int i) {
    double hi = h[i], lo = 0.0;
    for (int j = 0; j < n; ++j) {
        const double p = G[i * n + j] * c[j];
        const double pe = std::fma(G[i * n + j], c[j], -p);
        const double s = hi - p;
        const double bb = s - hi;
        lo += ((hi - (s - bb)) + (-p - bb)) - pe;
        hi = s;
    }
    return hi + lo;
}

pp_status pp_poly_coeffs_wl2(int d, const double* moments, double* c) {
    if (!c || !moments || d < 0 || d > 8) {
        set_error("pp_poly_coeffs_wl2: need 0 <= d <= 8 and non-NULL moments, c");
        return PP_ERR_INVALID_ARG;
    }
    for (int k = 0; k <= 2 * d + 2; ++k)
        if (!std::isfinite(moments[k])) {
            set_error("pp_poly_coeffs_wl2: moment %d is not finite", k);
            return PP_ERR_INVALID_ARG;
        }
    // normal equations of int_0^1 w (1 - z p)^2: sum_j m_{i+j+2} c_j = m_{i+1}
    const int n = d + 1;
    double G[81], h[9], LU[81];
    int piv[9];
    for (int i = 0; i < n; ++i) {
        h[i] = moments[i + 1];
        for (int j = 0; j < n; ++j) G[i * n + j] = LU[i * n + j] = moments[i + j + 2];
    }
    double gmax = 0.0;
    for (int i = 0; i < n * n; ++i) gmax = std::max(gmax, std::fabs(G[i]));
    // LU with partial pivoting
    for (int k = 0; k < n; ++k) {
        int p = k;
        for (int r = k + 1; r < n; ++r)
            if (std::fabs(LU[r * n + k]) > std::fabs(LU[p * n + k])) p = r;
        piv[k] = p;
        if (!(std::fabs(LU[p * n + k]) > 1e-15 * gmax)) {
            set_error("pp_poly_coeffs_wl2: the moments do not define a positive weight "
                      "(singular normal equations)");
            return PP_ERR_INVALID_ARG;
        }
        if (p != k)
            for (int j = 0; j < n; ++j) std::swap(LU[k * n + j], LU[p * n + j]);
        for (int r = k + 1; r < n; ++r) {
            LU[r * n + k] /= LU[k * n + k];
            for (int j = k + 1; j < n; ++j) LU[r * n + j] -= LU[r * n + k] * LU[k * n + j];
        }
    }
    auto lu_solve = [&](double* x) {
        for (int k = 0; k < n; ++k) std::swap(x[k], x[piv[k]]);
        for (int i = 0; i < n; ++i)
            for (int j = 0; j < i; ++j) x[i] -= LU[i * n + j] * x[j];
        for (int i = n - 1; i >= 0; --i) {
            for (int j = i + 1; j < n; ++j) x[i] -= LU[i * n + j] * x[j];
            x[i] /= LU[i * n + i];
        }
    };
    for (int i = 0; i < n; ++i) c[i] = h[i];
    lu_solve(c);
    // iterative refinement with compensated residuals: each step multiplies
    // the error by about cond(G) * 2^-53, which stays below 1 up to d = 8 for
    // weights that are not extremely concentrated; stop once the correction
    // no longer changes c
    for (int it = 0; it < 60; ++it) {
        double r[9], dmax = 0.0, cmax = 0.0;
        for (int i = 0; i < n; ++i) r[i] = residual_dd(G, h, c, n, i);
        lu_solve(r);
        for (int i = 0; i < n; ++i) {
            c[i] += r[i];
            dmax = std::max(dmax, std::fabs(r[i]));
            cmax = std::max(cmax, std::fabs(c[i]));
        }
        if (!(dmax > 1e-17 * cmax)) break;
    }
    for (int i = 0; i < n; ++i)
        if (!std::isfinite(c[i])) {
            set_error("pp_poly_coeffs_wl2: non-finite coefficients");
            return PP_ERR_NONFINITE;
        }
    return PP_OK;
}

pp_status pp_poly_coeffs_cheb(int d, double mu, double* c) {
    if (!c || d < 0 || d > 8 || !(mu > 0.0 && mu < 1.0)) {
        set_error("pp_poly_coeffs_cheb: need 0 <= d <= 8, 0 < mu < 1, c != NULL");
        return PP_ERR_INVALID_ARG;
    }
    // T_k(a + b z) as monomial coefficients in z by T_{k+1} = 2 (a + b z) T_k - T_{k-1}
    const double a = (1.0 + mu) / (1.0 - mu), bz = -2.0 / (1.0 - mu);
    const int m = d + 1;
    double Tm1[10] = {0}, T0[10] = {0}, T1[10] = {0};
    T0[0] = 1.0;                         // T_0
    T1[0] = a; T1[1] = bz;               // T_1
    if (m == 1) {
        for (int i = 0; i < 10; ++i) Tm1[i] = T1[i];
    } else {
        double prev[10], cur[10];
        for (int i = 0; i < 10; ++i) { prev[i] = T0[i]; cur[i] = T1[i]; }
        for (int k = 1; k < m; ++k) {
            double next[10] = {0};
            for (int i = 0; i <= k; ++i) {
                next[i] += 2.0 * a * cur[i];
                next[i + 1] += 2.0 * bz * cur[i];
            }
            for (int i = 0; i < 10; ++i) next[i] -= prev[i];
            for (int i = 0; i < 10; ++i) { prev[i] = cur[i]; cur[i] = next[i]; }
        }
        for (int i = 0; i < 10; ++i) Tm1[i] = cur[i];
    }
    // r = T_m(a + b z) / T_m(a); T_m(a) is the constant term
    const double t0 = Tm1[0];
    for (int i = 0; i <= d; ++i) c[i] = -Tm1[i + 1] / t0;
    return PP_OK;
}

pp_status pp_plan_create(pp_plan** out, pp_dims dims, int coils, const pp_c64* sens,
                         const pp_sampling* s, uint64_t seed, int power_iters, pp_stream stream) {
    if (!out) {
        set_error("pp_plan_create: out is NULL");
        return PP_ERR_INVALID_ARG;
    }
    *out = nullptr;
    if (!sens || !s) {
        set_error("pp_plan_create: sens and sampling must be non-NULL");
        return PP_ERR_INVALID_ARG;
    }
    if ((uintptr_t)sens & 15) {
        set_error("pp_plan_create: sens must be 16-byte aligned");
        return PP_ERR_INVALID_ARG;
    }
    if (dims.ndim != 2 && dims.ndim != 3) {
        set_error("pp_plan_create: ndim must be 2 or 3");
        return PP_ERR_UNSUPPORTED;
    }
    const int nx = dims.n[0], ny = dims.n[1], nz = dims.ndim == 3 ? dims.n[2] : 1;
    if (nx < 4 || ny < 4 || nz < 1 || (dims.ndim == 3 && nz < 4) || nx > 512 || ny > 512 ||
        nz > 512) {
        set_error("pp_plan_create: image size out of range (4..512 per axis)");
        return PP_ERR_INVALID_ARG;
    }
    if ((nx % 4) || (ny % 4) || (dims.ndim == 3 && (nz % 4))) {
        set_error("pp_plan_create: every image axis must be a multiple of 4");
        return PP_ERR_UNSUPPORTED;
    }
    if (coils < 1 || coils > 64) {
        set_error("pp_plan_create: coils must be in 1..64");
        return PP_ERR_INVALID_ARG;
    }
    if (power_iters < 0 || power_iters > 100000) {
        set_error("pp_plan_create: power_iters out of range");
        return PP_ERR_INVALID_ARG;
    }
    if (s->kind == PP_CARTESIAN) {
        if (!s->mask) {
            set_error("pp_plan_create: Cartesian sampling needs a mask");
            return PP_ERR_INVALID_ARG;
        }
        if (!fft_len_ok(nx) || !fft_len_ok(ny) || (dims.ndim == 3 && !fft_len_ok(nz))) {
            set_error("pp_plan_create: FFT lengths need prime factors <= 5");
            return PP_ERR_UNSUPPORTED;
        }
    } else if (s->kind == PP_NONCARTESIAN || s->kind == PP_NONCARTESIAN_TOEPLITZ) {
        if (!s->traj) {
            set_error("pp_plan_create: non-Cartesian sampling needs a trajectory");
            return PP_ERR_INVALID_ARG;
        }
        if (dims.ndim != 2) {
            set_error("pp_plan_create: non-Cartesian plans are 2-D only");
            return PP_ERR_UNSUPPORTED;
        }
        if (s->kind == PP_NONCARTESIAN_TOEPLITZ && !toep_supported(nx, ny, coils)) {
            set_error("pp_plan_create: the Toeplitz normal operator needs coils <= 32 and "
                      "nx, ny in {64, 96, 128, 160, 192, 256}");
            return PP_ERR_UNSUPPORTED;
        }
    } else {
        set_error("pp_plan_create: unknown sampling kind %d", s->kind);
        return PP_ERR_INVALID_ARG;
    }
    static PerDevice configured;
    pp_status cfg = PP_OK;
    configured.get(current_device(), [&] { return (cfg = configure_kernels()) == PP_OK ? 0 : -1; });
    if (cfg != PP_OK) return cfg;

    pp_plan* h = new pp_plan();
    Plan& p = h->impl;
    p.ndim = dims.ndim; p.nx = nx; p.ny = ny; p.nz = nz; p.C = coils;
    p.kind = s->kind == PP_NONCARTESIAN_TOEPLITZ ? PP_NONCARTESIAN : s->kind;
    p.toep = s->kind == PP_NONCARTESIAN_TOEPLITZ;
    p.nimg = (int64_t)nx * ny * nz;
    p.sens = reinterpret_cast<const float2*>(sens);
    cudaGetDevice(&p.dev);
    cudaStream_t st = (cudaStream_t)stream;
    pp_status rc = (s->kind == PP_CARTESIAN) ? build_cartesian(p, s->mask) : build_noncartesian(p, s);
    if (rc == PP_OK && s->kind == PP_CARTESIAN && p.ndim == 2) p.cols = cart_cols_width_ok(p.ny, 1);
    if (rc == PP_OK) {
        const size_t n = (size_t)p.nimg;
        p.red_blocks = 2 * 152;
        if ((rc = alloc_n(p, &p.z, n)) == PP_OK && (rc = alloc_n(p, &p.y, n)) == PP_OK &&
            (rc = alloc_n(p, &p.g, n)) == PP_OK && (rc = alloc_n(p, &p.u, n)) == PP_OK &&
            (rc = alloc_n(p, &p.t, n)) == PP_OK && (rc = alloc_n(p, &p.ahb, n)) == PP_OK &&
            (rc = alloc_n(p, &p.v, n)) == PP_OK && (rc = alloc_n(p, &p.w3, n)) == PP_OK &&
            (rc = alloc_n(p, &p.red, (size_t)3 * p.red_blocks)) == PP_OK &&
            (rc = alloc_n(p, &p.scal, 8)) == PP_OK) {
            cudaError_t e = cudaStreamCreateWithFlags(&p.cap_stream, cudaStreamNonBlocking);
            if (e != cudaSuccess) rc = cuda_status(e, "cudaStreamCreate");
        }
    }
    int dev_now = 0;
    cudaGetDevice(&dev_now);
    const TuneKey tkey = tune_key(p, s, dev_now);
    bool tuned = false;   // launch shapes taken from an earlier plan of the same geometry
    if (rc == PP_OK && p.kind == PP_CARTESIAN && p.ndim == 2 && !(tuned = tune_lookup(tkey, p)))
        rc = tune_cart2d(p, st);
    if (rc == PP_OK && p.kind == PP_CARTESIAN && p.ndim == 3) {
        p.c3cl_clusters = c3cl_prepare(p, 4);
        p.c3cl2_clusters = c3cl_prepare(p, 2);
        p.c3df_ctas = c3df_prepare(p, 0);
        p.c3df_ctas_hi = c3df_prepare(p, 1);
        p.c3df_ctas_tma = (p.c3df_ctas > 0 && c3df_make_tensor_map(p)) ? c3df_prepare(p, 2) : 0;
        p.c3df_ctas_tma1 = p.c3df_ctas_tma > 0 ? c3df_prepare(p, 3) : 0;
        if (p.c3df_ctas > 0) {
            // two phase slots for up to 8 coils per group; counters for 1
            p.c3df_w_elems = 2 * c3df_slot_elems(p, std::min(8, std::max(2, p.C)));
            p.c3df_cnt_ints = 0;
            for (int cgc = 1; cgc <= 8; ++cgc)
                p.c3df_cnt_ints = std::max(p.c3df_cnt_ints, c3df_counter_ints(p, cgc));
            if ((rc = alloc_n(p, &p.c3df_w, p.c3df_w_elems)) == PP_OK &&
                (rc = alloc_n(p, &p.c3df_cnt, p.c3df_cnt_ints)) == PP_OK)
                rc = cudaMemsetAsync(p.c3df_cnt, 0, sizeof(int) * p.c3df_cnt_ints, st) == cudaSuccess
                         ? PP_OK : cuda_status(cudaGetLastError(), "cudaMemsetAsync");
            p.c3df_cg = std::min(4, p.C);
        }
        if (rc == PP_OK) widen_c3(p);
        if (rc == PP_OK && !(tuned = tune_lookup(tkey, p))) rc = tune_cart3d(p, st);
    }
    if (rc == PP_OK && p.kind == PP_NONCARTESIAN) rc = setup_ci(p, st);
    if (rc == PP_OK && p.toep) rc = setup_toeplitz(p, s, st);
    if (rc == PP_OK && p.kind == PP_NONCARTESIAN) {
        // the spread's transposed k-space; without it the spread reads [C][K] in place
        if (void* w = spare_alloc(nufft_transposed_elems(p) * sizeof(float2))) {
            p.allocs.push_back(w);
            p.ksp_t = static_cast<float2*>(w);
        }
    }
    if (rc == PP_OK && p.kind == PP_NONCARTESIAN && !p.toep && !(tuned = tune_lookup(tkey, p)))
        rc = tune_noncartesian(p, st);
    if (rc == PP_OK && !tuned) tune_store(tkey, p);
    if (rc == PP_OK && power_iters > 0) rc = power_iteration(p, seed, power_iters, st);
    if (rc != PP_OK) {
        cudaStreamSynchronize(st);
        for (void* a : p.allocs) cudaFree(a);
        if (p.cap_stream) cudaStreamDestroy(p.cap_stream);
        delete h;
        return rc;
    }
    *out = h;
    return PP_OK;
}

pp_status pp_plan_destroy(pp_plan* plan) {
    if (!plan) return PP_OK;
    Plan& p = plan->impl;
    if (p.gexec) cudaGraphExecDestroy(p.gexec);
    if (p.cap_stream) cudaStreamDestroy(p.cap_stream);
    for (void* a : p.allocs) cudaFree(a);
    delete plan;
    return PP_OK;
}

pp_status pp_plan_scale(const pp_plan* plan, double* L) {
    if (!plan || !L) {
        set_error("pp_plan_scale: NULL argument");
        return PP_ERR_INVALID_ARG;
    }
    *L = plan->impl.L;
    return PP_OK;
}

pp_status pp_plan_set_scale(pp_plan* plan, double L) {
    if (!plan || !(L > 0.0) || !isfinite(L)) {
        set_error("pp_plan_set_scale: need a plan and a finite L > 0");
        return PP_ERR_INVALID_ARG;
    }
    if (plan->impl.L != L) {
        plan->impl.L = L;
        plan->impl.gkey.clear();   // captured graphs bake 1/L into their kernels
    }
    return PP_OK;
}

pp_status pp_plan_tuning(const pp_plan* plan, int* row_ifft_variant, int* stencil_kind,
                         int* stencil_coils) {
    if (!plan) {
        set_error("pp_plan_tuning: NULL plan");
        return PP_ERR_INVALID_ARG;
    }
    if (row_ifft_variant) {
        const Plan& p = plan->impl;
        if (p.kind == PP_CARTESIAN && p.ndim == 3)
            *row_ifft_variant = p.tune_c3 == 1 ? 16 : (p.tune_c3 == 2 ? -16 : (p.tune_c3 == 3 ? 3 : 1));
        else if (p.kind == PP_CARTESIAN)
            *row_ifft_variant = p.tune_c2;
        else
            *row_ifft_variant = p.tune_rows_adj_cl ? p.tune_rows_adj_cl : 1;
    }
    if (stencil_kind) {
        const Plan& p = plan->impl;
        *stencil_kind = (p.kind == PP_CARTESIAN && p.ndim == 3 && p.tune_c3 == 3) ? p.c3df_hi
                                                                                  : p.tune_stencil_kind;
    }
    if (stencil_coils) {
        const Plan& p = plan->impl;
        *stencil_coils = (p.kind == PP_CARTESIAN && p.ndim == 3 && p.tune_c3 == 3)
                             ? p.c3df_cg : (p.tune_stencil_cpc ? p.tune_stencil_cpc : 8);
    }
    return PP_OK;
}

pp_status pp_plan_set_tuning(pp_plan* plan, int row_ifft_variant, int stencil_kind, int stencil_coils) {
    if (!plan || !(row_ifft_variant == 1 || row_ifft_variant == 2 || row_ifft_variant == 4 ||
                   row_ifft_variant == -1 || row_ifft_variant == 8 || row_ifft_variant == 16 ||
                   row_ifft_variant == -16 || row_ifft_variant == 3) ||
        stencil_kind < 0 || stencil_kind > 9 || stencil_coils < 1 || stencil_coils > 64) {
        set_error("pp_plan_set_tuning: row variant must be 1, 2, 3, 4, 8, -1, 16 or -16; stencil "
                  "kind 0..9; stencil coils 1..64");
        return PP_ERR_INVALID_ARG;
    }
    Plan& p = plan->impl;
    if (row_ifft_variant == 3) {
        const int cgv = std::min(stencil_coils, std::max(1, p.C));   // the kernel's group size
        if (!(p.kind == PP_CARTESIAN && p.ndim == 3) || p.c3df_ctas <= 0 ||
            2 * c3df_slot_elems(p, cgv) > p.c3df_w_elems ||
            c3df_counter_ints(p, cgv) > p.c3df_cnt_ints) {
            set_error("pp_plan_set_tuning: row variant 3 (the 3-D dataflow operator) needs a 3-D "
                      "Cartesian plan with register-FFT lengths ny, nz and at most 8 coils per group");
            return PP_ERR_UNSUPPORTED;
        }
        if (stencil_kind < 0 || stencil_kind > 5 || ((stencil_kind == 1 || stencil_kind == 5) && p.c3df_ctas_hi <= 0) ||
            (stencil_kind == 2 && p.c3df_ctas_tma <= 0) || (stencil_kind == 3 && p.c3df_ctas_tma1 <= 0)) {
            set_error("pp_plan_set_tuning: the 3-D dataflow operator takes stencil kind 0 (two "
                      "blocks per SM), 1 (three), 2 (map tiles staged by TMA), 3 (staged by TMA "
                      "into one buffer, three blocks per SM), 4 or 5 (0 or 1 with two z planes "
                      "per y-FFT item and two line units per z item)");
            return PP_ERR_UNSUPPORTED;
        }
        p.tune_c3 = 3;
        p.c3df_cg = stencil_coils;
        p.c3df_hi = stencil_kind;
        p.gkey.clear();
        return PP_OK;
    }
    if ((row_ifft_variant == 16 && p.c3cl_clusters <= 0) ||
        (row_ifft_variant == -16 && p.c3cl2_clusters <= 0)) {
        set_error("pp_plan_set_tuning: the one-kernel cluster operator needs a 3-D Cartesian plan "
                  "with nz = 128, ny in {128, 192, 256} and a device that fits 16-CTA clusters");
        return PP_ERR_UNSUPPORTED;
    }
    if (row_ifft_variant == 8 && !(p.kind == PP_CARTESIAN && p.ndim == 2)) {
        set_error("pp_plan_set_tuning: row variant 8 (the streaming form on 8 columns) applies to "
                  "2-D Cartesian plans");
        return PP_ERR_UNSUPPORTED;
    }
    if (p.kind == PP_CARTESIAN && p.ndim == 3)
        p.tune_c3 = row_ifft_variant == 16 ? 1 : (row_ifft_variant == -16 ? 2 : 0);
    if (p.kind == PP_CARTESIAN && p.ndim == 2) {
        if (row_ifft_variant == -1 || row_ifft_variant == 16 || row_ifft_variant == -16) {
            set_error("pp_plan_set_tuning: 2-D Cartesian plans take row variant 1, 2, 4 or 8 (image "
                      "columns per CTA)");
            return PP_ERR_UNSUPPORTED;
        }
        p.tune_c2 = p.tune_c2_one = row_ifft_variant;
        p.gkey.clear();
        return PP_OK;
    }
    if (row_ifft_variant == -1 && (p.kind != PP_NONCARTESIAN || !fft4_n2(p.G_x))) {
        set_error("pp_plan_set_tuning: the split row IFFT needs a non-Cartesian plan with a "
                  "register-FFT grid length");
        return PP_ERR_UNSUPPORTED;
    }
    if (stencil_kind >= 2 && (p.kind != PP_NONCARTESIAN || p.stencil_rb_grid[0] == 0 ||
                              (stencil_kind <= 5 && p.stencil_rb_grid[stencil_kind - 2] == 0))) {
        set_error("pp_plan_set_tuning: register-blocked stencil kinds need a non-Cartesian plan "
                  "whose 49 weight planes hold fewer than 2^31 values");
        return PP_ERR_UNSUPPORTED;
    }
    if (stencil_kind >= 7 && !p.ci_sens) {
        set_error("pp_plan_set_tuning: the coil-innermost pipeline needs at most 32 coils and "
                  "register-FFT grid lengths");
        return PP_ERR_UNSUPPORTED;
    }
    p.tune_rows_adj_cl = row_ifft_variant;
    p.tune_stencil_kind = stencil_kind;
    p.tune_stencil_cpc = stencil_coils;
    p.gkey.clear();
    return PP_OK;
}

pp_status pp_plan_mu(pp_plan* plan, int iters, uint64_t seed, double* mu, pp_stream stream) {
    if (!plan || !mu || iters < 1 || iters > 1000000) {
        set_error("pp_plan_mu: bad argument");
        return PP_ERR_INVALID_ARG;
    }
    return mu_iteration(plan->impl, seed, iters, mu, (cudaStream_t)stream);
}

pp_status pp_prox_llr(pp_dims dims, int T, int block, const int* shift, float lambda,
                      const pp_c64* in, pp_c64* out, pp_stream stream) {
    if (!in || !out || !(lambda >= 0.f) || !isfinite(lambda) || (dims.ndim != 2 && dims.ndim != 3)) {
        set_error("pp_prox_llr: bad argument");
        return PP_ERR_INVALID_ARG;
    }
    const int nz = dims.ndim == 3 ? dims.n[2] : 1;
    if (T < 1 || T > 8 || !(block == 4 || block == 8 || (block == 16 && dims.ndim == 2)) ||
        dims.n[0] < 1 || dims.n[1] < 1 || nz < 1 || dims.n[0] % block || dims.n[1] % block ||
        (dims.ndim == 3 && nz % block)) {
        set_error("pp_prox_llr: need 1 <= T <= 8, block 4 or 8 (16 in 2-D) dividing every axis");
        return PP_ERR_UNSUPPORTED;
    }
    return launch_prox_llr(dims.ndim, dims.n[0], dims.n[1], nz, T, block, shift, lambda,
                           reinterpret_cast<const float2*>(in), reinterpret_cast<float2*>(out),
                           (cudaStream_t)stream);
}

pp_status pp_selftest_wait(int64_t limit_ns, pp_stream stream) {
    if (limit_ns < 1000000 || limit_ns > 1000000000) {
        set_error("pp_selftest_wait: limit must be 1 ms .. 1 s");
        return PP_ERR_INVALID_ARG;
    }
    return selftest_wait((long long)limit_ns, (cudaStream_t)stream);
}

pp_status pp_plan_sizes(const pp_plan* plan, int64_t* image_elems, int64_t* kspace_elems) {
    if (!plan) {
        set_error("pp_plan_sizes: NULL plan");
        return PP_ERR_INVALID_ARG;
    }
    if (image_elems) *image_elems = plan->impl.nimg;
    if (kspace_elems) *kspace_elems = plan->impl.nksp;
    return PP_OK;
}

pp_status pp_forward_apply(const pp_plan* plan, const pp_c64* x, pp_c64* y, pp_stream stream) {
    if (!plan || !x || !y) {
        set_error("pp_forward_apply: NULL argument");
        return PP_ERR_INVALID_ARG;
    }
    return forward_into(plan->impl, reinterpret_cast<const float2*>(x), reinterpret_cast<float2*>(y),
                        (cudaStream_t)stream);
}

pp_status pp_adjoint_apply(const pp_plan* plan, const pp_c64* y, pp_c64* x, pp_stream stream) {
    if (!plan || !x || !y) {
        set_error("pp_adjoint_apply: NULL argument");
        return PP_ERR_INVALID_ARG;
    }
    return adjoint_into(plan->impl, reinterpret_cast<const float2*>(y), reinterpret_cast<float2*>(x),
                        (cudaStream_t)stream);
}

pp_status pp_normal_apply(const pp_plan* plan, const pp_c64* x, pp_c64* y, pp_stream stream) {
    if (!plan || !x || !y || (const void*)x == (const void*)y) {
        set_error("pp_normal_apply: NULL or aliased argument");
        return PP_ERR_INVALID_ARG;
    }
    const Plan& p = plan->impl;
    return normal_into(p, reinterpret_cast<const float2*>(x), reinterpret_cast<float2*>(y),
                       (float)(1.0 / p.L), nullptr, 0.f, (cudaStream_t)stream);
}

pp_status pp_poly_apply(const pp_plan* plan, const double* c, int d, const pp_c64* v, pp_c64* out,
                        pp_stream stream) {
    if (!plan || !c || !v || !out || d < 0 || d > 16 || (const void*)v == (const void*)out) {
        set_error("pp_poly_apply: bad argument (NULL, aliased, or d outside 0..16)");
        return PP_ERR_INVALID_ARG;
    }
    Plan& p = const_cast<Plan&>(plan->impl);
    return horner_into(p, c, d, reinterpret_cast<const float2*>(v), reinterpret_cast<float2*>(out),
                       p.t, p.w3, (cudaStream_t)stream);
}

pp_status pp_prox_l1_haar(pp_dims dims, int levels, float lambda, const pp_c64* in, pp_c64* out,
                          pp_stream stream) {
    if (!in || !out || (dims.ndim != 2 && dims.ndim != 3) || !(lambda >= 0.f) || !isfinite(lambda)) {
        set_error("pp_prox_l1_haar: bad argument");
        return PP_ERR_INVALID_ARG;
    }
    if (levels < 1 || levels > 2) {
        set_error("pp_prox_l1_haar: levels must be 1 or 2");
        return PP_ERR_UNSUPPORTED;
    }
    const int ts = 1 << levels;
    const int nx = dims.n[0], ny = dims.n[1], nz = dims.ndim == 3 ? dims.n[2] : 1;
    if (nx <= 0 || ny <= 0 || nz <= 0 || nx % ts || ny % ts || (dims.ndim == 3 && nz % ts)) {
        set_error("pp_prox_l1_haar: every axis must be a positive multiple of 2^levels");
        return PP_ERR_UNSUPPORTED;
    }
    return launch_prox(dims.ndim, nx, ny, nz, levels, lambda, reinterpret_cast<const float2*>(in),
                       reinterpret_cast<float2*>(out), (cudaStream_t)stream);
}

pp_status pp_prox_l1_db4(pp_dims dims, int levels, float lambda, const pp_c64* in, pp_c64* out,
                         pp_stream stream) {
    if (!in || !out || (dims.ndim != 2 && dims.ndim != 3) || !(lambda >= 0.f) || !isfinite(lambda)) {
        set_error("pp_prox_l1_db4: bad argument");
        return PP_ERR_INVALID_ARG;
    }
    if (!db4_supported(dims.ndim, dims.n[0], dims.n[1], levels)) {
        set_error("pp_prox_l1_db4: 2-D only, levels 1..4, axes <= 512 and multiples of 2^levels");
        return PP_ERR_UNSUPPORTED;
    }
    return launch_prox_db4(dims.n[0], dims.n[1], levels, lambda, reinterpret_cast<const float2*>(in),
                           reinterpret_cast<float2*>(out), (cudaStream_t)stream);
}

// After a synchronising solve: a NaN or infinite ||b||^2 (first slice's for
// a batch) or history entry means the input held a non-finite value.
static pp_status check_history(const char* who, double bn2, const double* h, int iters) {
    bool ok = std::isfinite(bn2);
    for (int i = 0; ok && i < 3 * iters; ++i) ok = std::isfinite(h[i]);
    if (!ok) {
        set_error("%s: non-finite value in b (||b||^2 = %g) or in the iterates", who, bn2);
        return PP_ERR_NONFINITE;
    }
    return PP_OK;
}

// info->safe_scale: c divided by max_{z in [0, 1]} z p(z), in buf
static pp_status safe_coeffs(const pp_solve_info* info, const double*& c, int d, std::vector<double>& buf) {
    if (!info || !info->safe_scale || !c) return PP_OK;
    double m = 0.0;
    PP_TRY(pp_poly_max_zp(c, d, &m));
    if (!(m > 0.0)) {
        set_error("safe_scale: max of z p(z) on [0, 1] is not positive");
        return PP_ERR_INVALID_ARG;
    }
    buf.assign(c, c + d + 1);
    for (double& v : buf) v /= m;
    c = buf.data();
    return PP_OK;
}

pp_status pp_fista_solve(pp_plan* plan, const pp_c64* b, float lambda, int iters, const double* c,
                         int d, pp_c64* x_out, pp_solve_info* info, pp_stream stream) {
    if (!plan || !b || !x_out || iters < 0 || iters > 1000000 || !(lambda >= 0.f) ||
        !isfinite(lambda) || d < 0 || d > 16 || (!c && d != 0)) {
        set_error("pp_fista_solve: bad argument");
        return PP_ERR_INVALID_ARG;
    }
    Plan& p = plan->impl;
    cudaStream_t st = (cudaStream_t)stream;
    std::vector<double> c_safe;
    PP_TRY(safe_coeffs(info, c, d, c_safe));
    const int levels = (info && info->levels) ? info->levels : 2;
    const int wavelet = info ? info->wavelet : 0;
    if (wavelet != 0 && wavelet != 1) {
        set_error("pp_fista_solve: wavelet must be 0 (Haar) or 1 (Daubechies-4)");
        return PP_ERR_INVALID_ARG;
    }
    if (wavelet == 1 && !db4_supported(p.ndim, p.nx, p.ny, levels)) {
        set_error("pp_fista_solve: the Daubechies-4 prox is 2-D with levels 1..4 and axes "
                  "multiples of 2^levels");
        return PP_ERR_UNSUPPORTED;
    }
    if (wavelet == 0 && (levels < 1 || levels > 2 || p.nx % (1 << levels) || p.ny % (1 << levels) ||
                         (p.ndim == 3 && p.nz % (1 << levels)))) {
        set_error("pp_fista_solve: unsupported Haar levels");
        return PP_ERR_UNSUPPORTED;
    }
    const bool hist = info && info->history;
    const bool momentum = !(info && info->no_momentum);
    const float2* ref = info ? reinterpret_cast<const float2*>(info->ref) : nullptr;
    const int64_t n = p.nimg;
    const int64_t launches0 = g_launches;
    // A_hat^H b_hat = A^H b / (sqrt(L) ||b||)
    PP_TRY(launch_norm2(reinterpret_cast<const float2*>(b), p.nksp, p.red, p.red_blocks, p.scal + 0, st));
    PP_TRY(adjoint_into(p, reinterpret_cast<const float2*>(b), p.ahb, st));
    PP_TRY(launch_scale_by_rnorm(p.ahb, p.ahb, n, p.scal + 0, 1.0 / sqrt(p.L), 1, st));
    PP_TRY_CUDA(cudaMemsetAsync(p.y, 0, n * sizeof(float2), st));
    PP_TRY_CUDA(cudaMemsetAsync(p.z, 0, n * sizeof(float2), st));
    if (hist) {
        if (p.hist_cap < iters) {
            if (p.hist) {
                cudaStreamSynchronize(st);
                cudaFree(p.hist);
                p.allocs.erase(std::remove(p.allocs.begin(), p.allocs.end(), (void*)p.hist), p.allocs.end());
                p.hist = nullptr;
            }
            PP_TRY(alloc_n(p, &p.hist, (size_t)3 * std::max(iters, 1)));
            p.hist_cap = iters;
            p.gkey.clear();
        }
        PP_TRY_CUDA(cudaMemsetAsync(p.hist, 0, sizeof(double) * 3 * std::max(iters, 1), st));
    }
    if (iters > 0) {
        std::vector<double> key = {0.0 /* normalised solve */, (double)iters, (double)d,
                                   (double)lambda, (double)levels, hist ? 1.0 : 0.0, c ? 1.0 : 0.0, p.L,
                                   (double)(uintptr_t)p.hist, (double)(uintptr_t)ref,
                                   momentum ? 1.0 : 0.0, (double)wavelet};
        if (c)
            for (int i = 0; i <= d; ++i) key.push_back(c[i]);
        if (!p.gexec || key != p.gkey) {
            if (p.gexec) {
                cudaGraphExecDestroy(p.gexec);
                p.gexec = nullptr;
            }
            p.gkey.clear();
            cudaGraph_t graph = nullptr;
            PP_TRY_CUDA(cudaStreamBeginCapture(p.cap_stream, cudaStreamCaptureModeThreadLocal));
            const int64_t before = g_launches;
            pp_status rc = fista_iterations(p, lambda, iters, c, d, levels, hist, ref, momentum,
                                            wavelet, p.cap_stream);
            cudaError_t e = cudaStreamEndCapture(p.cap_stream, &graph);
            p.graph_kernels = g_launches - before;
            g_launches = before;
            if (rc != PP_OK) {
                if (graph) cudaGraphDestroy(graph);
                return rc;
            }
            if (e != cudaSuccess) return cuda_status(e, "cudaStreamEndCapture");
            e = cudaGraphInstantiate(&p.gexec, graph, 0);
            cudaGraphDestroy(graph);
            if (e != cudaSuccess) {
                p.gexec = nullptr;
                return cuda_status(e, "cudaGraphInstantiate");
            }
            p.gkey = key;
        }
        PP_TRY_CUDA(cudaGraphLaunch(p.gexec, st));
    }
    float2* xo = reinterpret_cast<float2*>(x_out);
    if (info && info->rescale)
        PP_TRY(launch_scale_by_rnorm(p.y, xo, n, p.scal + 0, 1.0 / sqrt(p.L), 0, st));
    else
        PP_TRY_CUDA(cudaMemcpyAsync(xo, p.y, n * sizeof(float2), cudaMemcpyDeviceToDevice, st));
    if (info) {
        info->L = p.L;
        info->launches = (g_launches - launches0) + (iters > 0 ? p.graph_kernels : 0);
        if (hist) {
            double bn2 = 0.0;
            PP_TRY_CUDA(cudaMemcpyAsync(&bn2, p.scal + 0, sizeof(double), cudaMemcpyDeviceToHost, st));
            PP_TRY_CUDA(cudaMemcpyAsync(info->history, p.hist, sizeof(double) * 3 * iters,
                                        cudaMemcpyDeviceToHost, st));
            PP_TRY_CUDA(cudaStreamSynchronize(st));
            info->bnorm = sqrt(bn2);
            PP_TRY(c3df_check(p, st));
            PP_TRY(check_history("pp_fista_solve", bn2, info->history, iters));
        }
    }
    return PP_OK;
}

pp_status pp_fista_solve_prox(pp_plan* plan, const pp_c64* b, const pp_c64* v, double sigma,
                              float lambda, int iters, const double* c, int d, pp_c64* x_out,
                              pp_solve_info* info, pp_stream stream) {
    if (!plan || !x_out || iters < 0 || iters > 1000000 || !(lambda >= 0.f) || !isfinite(lambda) ||
        !(sigma >= 0.0) || !isfinite(sigma) || d < 0 || d > 16 || (!c && d != 0)) {
        set_error("pp_fista_solve_prox: bad argument");
        return PP_ERR_INVALID_ARG;
    }
    Plan& p = plan->impl;
    cudaStream_t st = (cudaStream_t)stream;
    const int levels = (info && info->levels) ? info->levels : 2;
    const int wavelet = info ? info->wavelet : 0;
    if (wavelet != 0 && wavelet != 1) {
        set_error("pp_fista_solve_prox: wavelet must be 0 (Haar) or 1 (Daubechies-4)");
        return PP_ERR_INVALID_ARG;
    }
    if ((wavelet == 1 && !db4_supported(p.ndim, p.nx, p.ny, levels)) ||
        (wavelet == 0 && (levels < 1 || levels > 2 || p.nx % (1 << levels) || p.ny % (1 << levels) ||
                          (p.ndim == 3 && p.nz % (1 << levels))))) {
        set_error("pp_fista_solve_prox: unsupported wavelet levels for this image");
        return PP_ERR_UNSUPPORTED;
    }
    const bool hist = info && info->history;
    const bool momentum = !(info && info->no_momentum);
    const float2* ref = info ? reinterpret_cast<const float2*>(info->ref) : nullptr;
    const int64_t n = p.nimg;
    const int64_t launches0 = g_launches;
    // L' = L + sigma; the iteration runs on N_hat' = a N_hat + b I with
    // a = L/L', b = sigma/L', gradient constant rhs = (A^H b + sigma v)/L'
    // and threshold lambda/L'; p(N_hat') = q(N_hat) with
    // q_j = sum_{i >= j} c_i C(i, j) a^j b^(i-j) (binomial expansion, FP64)
    const double Lp = p.L + sigma, sa = p.L / Lp, sb = sigma / Lp;
    std::vector<double> q;
    if (c) {
        q.assign(d + 1, 0.0);
        std::vector<double> binom(d + 1, 0.0);
        for (int i = 0; i <= d; ++i) {
            // binom[j] = C(i, j), row i of Pascal's triangle
            for (int j = i; j >= 1; --j) binom[j] += binom[j - 1];
            binom[0] = 1.0;
            for (int j = 0; j <= i; ++j) q[j] += c[i] * binom[j] * std::pow(sa, j) * std::pow(sb, i - j);
        }
    }
    if (b) {
        PP_TRY(launch_norm2(reinterpret_cast<const float2*>(b), p.nksp, p.red, p.red_blocks, p.scal + 0, st));
        PP_TRY(adjoint_into(p, reinterpret_cast<const float2*>(b), p.ahb, st));
        PP_TRY(launch_axpby(p.ahb, (float)(1.0 / Lp), reinterpret_cast<const float2*>(v),
                            (float)(sigma / Lp), p.ahb, n, st));
    } else if (v) {
        PP_TRY(launch_axpby(reinterpret_cast<const float2*>(v), (float)(sigma / Lp), nullptr, 0.f, p.ahb,
                            n, st));
    } else {
        PP_TRY_CUDA(cudaMemsetAsync(p.ahb, 0, n * sizeof(float2), st));
    }
    if (!b) PP_TRY_CUDA(cudaMemsetAsync(p.scal, 0, sizeof(double), st));
    PP_TRY_CUDA(cudaMemsetAsync(p.y, 0, n * sizeof(float2), st));
    PP_TRY_CUDA(cudaMemsetAsync(p.z, 0, n * sizeof(float2), st));
    if (hist) {
        if (p.hist_cap < iters) {
            if (p.hist) {
                cudaStreamSynchronize(st);
                cudaFree(p.hist);
                p.allocs.erase(std::remove(p.allocs.begin(), p.allocs.end(), (void*)p.hist), p.allocs.end());
                p.hist = nullptr;
            }
            PP_TRY(alloc_n(p, &p.hist, (size_t)3 * std::max(iters, 1)));
            p.hist_cap = iters;
            p.gkey.clear();
        }
        PP_TRY_CUDA(cudaMemsetAsync(p.hist, 0, sizeof(double) * 3 * std::max(iters, 1), st));
    }
    Shift sh;
    sh.on = true;
    sh.a = (float)sa;
    sh.b = (float)sb;
    const float lam_hat = (float)(lambda / Lp);
    if (iters > 0) {
        // the graph cache is shared with pp_fista_solve: the key tells the two apart
        std::vector<double> key = {1.0 /* proximal subproblem */, (double)iters, (double)d,
                                   (double)lam_hat, (double)levels, hist ? 1.0 : 0.0, c ? 1.0 : 0.0,
                                   p.L, (double)(uintptr_t)p.hist, (double)(uintptr_t)ref,
                                   momentum ? 1.0 : 0.0, (double)wavelet, sa, sb};
        for (double qj : q) key.push_back(qj);
        if (!p.gexec || key != p.gkey) {
            if (p.gexec) {
                cudaGraphExecDestroy(p.gexec);
                p.gexec = nullptr;
            }
            p.gkey.clear();
            cudaGraph_t graph = nullptr;
            PP_TRY_CUDA(cudaStreamBeginCapture(p.cap_stream, cudaStreamCaptureModeThreadLocal));
            const int64_t before = g_launches;
            pp_status rc = fista_iterations(p, lam_hat, iters, c ? q.data() : nullptr, d, levels, hist,
                                            ref, momentum, wavelet, p.cap_stream, sh);
            cudaError_t e = cudaStreamEndCapture(p.cap_stream, &graph);
            p.graph_kernels = g_launches - before;
            g_launches = before;
            if (rc != PP_OK) {
                if (graph) cudaGraphDestroy(graph);
                return rc;
            }
            if (e != cudaSuccess) return cuda_status(e, "cudaStreamEndCapture");
            e = cudaGraphInstantiate(&p.gexec, graph, 0);
            cudaGraphDestroy(graph);
            if (e != cudaSuccess) {
                p.gexec = nullptr;
                return cuda_status(e, "cudaGraphInstantiate");
            }
            p.gkey = key;
        }
        PP_TRY_CUDA(cudaGraphLaunch(p.gexec, st));
    }
    PP_TRY_CUDA(cudaMemcpyAsync(x_out, p.y, n * sizeof(float2), cudaMemcpyDeviceToDevice, st));
    if (info) {
        info->L = p.L;
        info->launches = (g_launches - launches0) + (iters > 0 ? p.graph_kernels : 0);
        if (hist) {
            double bn2 = 0.0;
            PP_TRY_CUDA(cudaMemcpyAsync(&bn2, p.scal + 0, sizeof(double), cudaMemcpyDeviceToHost, st));
            PP_TRY_CUDA(cudaMemcpyAsync(info->history, p.hist, sizeof(double) * 3 * iters,
                                        cudaMemcpyDeviceToHost, st));
            PP_TRY_CUDA(cudaStreamSynchronize(st));
            info->bnorm = sqrt(bn2);
            PP_TRY(c3df_check(p, st));
            PP_TRY(check_history("pp_fista_solve_prox", bn2, info->history, iters));
        }
    }
    return PP_OK;
}

pp_status pp_profile_normal(const pp_plan* plan, const pp_c64* x, pp_c64* y, int reps,
                            int max_stages, char* names, double* ms, int* nstages,
                            pp_stream stream) {
    if (!plan || !x || !y || reps < 1 || max_stages < 1 || !names || !ms || !nstages ||
        (const void*)x == (const void*)y) {
        set_error("pp_profile_normal: bad argument");
        return PP_ERR_INVALID_ARG;
    }
    const Plan& p = plan->impl;
    cudaStream_t st = (cudaStream_t)stream;
    Profiler prof;
    prof.st = st;
    cudaEvent_t start;
    PP_TRY_CUDA(cudaEventCreate(&start));
    PP_TRY_CUDA(cudaEventRecord(start, st));
    g_profiler = &prof;
    pp_status rc = PP_OK;
    for (int r = 0; r < reps && rc == PP_OK; ++r)
        rc = normal_into(p, reinterpret_cast<const float2*>(x), reinterpret_cast<float2*>(y),
                         (float)(1.0 / p.L), nullptr, 0.f, st);
    g_profiler = nullptr;
    cudaError_t e = cudaStreamSynchronize(st);
    std::vector<std::string> uniq;
    std::vector<double> tot;
    if (rc == PP_OK && e == cudaSuccess) {
        cudaEvent_t prev = start;
        for (size_t i = 0; i < prof.events.size(); ++i) {
            float t = 0.f;
            cudaEventElapsedTime(&t, prev, prof.events[i]);
            prev = prof.events[i];
            size_t j = std::find(uniq.begin(), uniq.end(), prof.names[i]) - uniq.begin();
            if (j == uniq.size()) {
                uniq.push_back(prof.names[i]);
                tot.push_back(0.0);
            }
            tot[j] += t;
        }
    }
    for (cudaEvent_t ev : prof.events) cudaEventDestroy(ev);
    cudaEventDestroy(start);
    if (rc != PP_OK) return rc;
    if (e != cudaSuccess) return cuda_status(e, "pp_profile_normal sync");
    const int ns = std::min((int)uniq.size(), max_stages);
    for (int i = 0; i < ns; ++i) {
        strncpy(names + 48 * i, uniq[i].c_str(), 47);
        names[48 * i + 47] = 0;
        ms[i] = tot[i] / reps;
    }
    *nstages = ns;
    return PP_OK;
}

struct pp_batch {
    Batch impl;
};

pp_status pp_batch_create(pp_batch** out, int nslices, const pp_dims* dims, const int* coils,
                          const pp_c64* const* sens, const uint8_t* const* masks, uint64_t seed,
                          int power_iters, pp_stream stream) {
    if (!out) {
        set_error("pp_batch_create: out is NULL");
        return PP_ERR_INVALID_ARG;
    }
    *out = nullptr;
    if (nslices < 1 || nslices > 4096 || !dims || !coils || !sens || !masks || power_iters < 0) {
        set_error("pp_batch_create: bad argument");
        return PP_ERR_INVALID_ARG;
    }
    for (int s = 0; s < nslices; ++s) {
        const pp_dims& d = dims[s];
        if (d.ndim != 2) {
            set_error("pp_batch_create: slice %d is not 2-D", s);
            return PP_ERR_UNSUPPORTED;
        }
        const int nx = d.n[0], ny = d.n[1];
        if (nx < 4 || ny < 4 || nx > 512 || ny > 512 || (nx % 4) || (ny % 4) || coils[s] < 1 ||
            coils[s] > 64 || !sens[s] || ((uintptr_t)sens[s] & 15) || !masks[s]) {
            set_error("pp_batch_create: slice %d has a bad size, coil count or pointer", s);
            return PP_ERR_INVALID_ARG;
        }
        if (!fft_len_ok(nx) || !fft_len_ok(ny)) {
            set_error("pp_batch_create: slice %d FFT length has a prime factor above 5", s);
            return PP_ERR_UNSUPPORTED;
        }
    }
    static PerDevice configured;
    pp_status cfg = PP_OK;
    configured.get(current_device(), [&] {
        cfg = configure_kernels();
        if (cfg == PP_OK) cfg = configure_batch_kernels();
        return cfg == PP_OK ? 0 : -1;
    });
    if (cfg != PP_OK) return cfg;
    cudaStream_t st = (cudaStream_t)stream;
    pp_batch* h = new pp_batch();
    Batch& b = h->impl;
    b.n = nslices;
    b.img_off.assign(nslices + 1, 0);
    b.ksp_off.assign(nslices + 1, 0);
    b.tile_off.assign(nslices + 1, 0);
    b.L.assign(nslices, 1.0);
    b.hdesc.resize(nslices);
    pp_status rc = PP_OK;
    size_t wk_max = 0;
    for (int s = 0; s < nslices && rc == PP_OK; ++s) {
        Plan* p = new Plan();
        b.sub.push_back(p);
        p->ndim = 2; p->nx = dims[s].n[0]; p->ny = dims[s].n[1]; p->nz = 1; p->C = coils[s];
        p->kind = PP_CARTESIAN;
        p->nimg = (int64_t)p->nx * p->ny;
        p->sens = reinterpret_cast<const float2*>(sens[s]);
        p->external_wk = true;
        rc = build_cartesian(*p, masks[s]);
        if (rc != PP_OK) break;
        wk_max = std::max(wk_max, (size_t)p->C * p->nimg);
        b.img_off[s + 1] = b.img_off[s] + p->nimg;
        b.ksp_off[s + 1] = b.ksp_off[s] + p->nksp;
        b.tile_off[s + 1] = b.tile_off[s] + p->nimg / 16;
        SliceDesc& d = b.hdesc[s];
        d.fd = p->fy.d; d.tw = p->fy.tw; d.twb = p->fy.twb; d.sens = p->sens; d.mask_fo = p->mask_fo;
        d.ny = p->ny; d.nx = p->nx; d.C = p->C; d.img_off = b.img_off[s];
        d.invL = 1.f;
        b.dev.ny_max = std::max(b.dev.ny_max, p->ny);
    }
    b.nimg = b.img_off[nslices];
    b.nksp = b.ksp_off[nslices];
    const size_t n = (size_t)b.nimg;
    if (rc == PP_OK && (rc = balloc(b, &b.z, n)) == PP_OK && (rc = balloc(b, &b.y, n)) == PP_OK &&
        (rc = balloc(b, &b.g, n)) == PP_OK && (rc = balloc(b, &b.u, n)) == PP_OK &&
        (rc = balloc(b, &b.t, n)) == PP_OK && (rc = balloc(b, &b.ahb, n)) == PP_OK &&
        (rc = balloc(b, &b.v, n)) == PP_OK && (rc = balloc(b, &b.w3, n)) == PP_OK &&
        (rc = balloc(b, &b.scal, (size_t)4 * nslices)) == PP_OK &&
        (rc = balloc(b, &b.dfac, (size_t)nslices)) == PP_OK &&
        (rc = balloc(b, &b.dev.descs, (size_t)nslices)) == PP_OK &&
        (rc = make_segments(b, b.dev.img, b.img_off, (int64_t)kThreads * 8, 64)) == PP_OK &&
        (rc = make_segments(b, b.dev.ksp, b.ksp_off, (int64_t)kThreads * 8, 64)) == PP_OK &&
        (rc = make_segments(b, b.dev.tiles, b.tile_off, kTileThreads / 4, 1 << 30)) == PP_OK) {
        const int nb = std::max(b.dev.img.nblocks, b.dev.ksp.nblocks);
        rc = balloc(b, &b.partials, (size_t)3 * nb);
    }
    if (rc == PP_OK) {
        cudaError_t e = cudaStreamCreateWithFlags(&b.cap_stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) rc = cuda_status(e, "cudaStreamCreate");
    }
    if (rc == PP_OK) rc = upload_descs(b);
    if (rc == PP_OK) {
        cudaError_t e = cudaMemsetAsync(b.v, 0, n * sizeof(float2), st);
        if (e != cudaSuccess) rc = cuda_status(e, "cudaMemsetAsync");
    }
    // adjoint workspace: as many slices as fit half of the L2 together, where there is
    // memory for them, but at least the largest
    size_t wk = std::max(wk_max, std::min((size_t)b.nksp, (size_t)(72 << 20) / sizeof(float2)));
    if (rc == PP_OK) {
        if (void* w = wk > wk_max ? spare_alloc(wk * sizeof(float2)) : nullptr) {
            b.allocs.push_back(w);
            b.wk = static_cast<float2*>(w);
        } else {
            wk = wk_max;
            rc = balloc(b, &b.wk, wk);
        }
        for (Plan* p : b.sub) p->wk_a = b.wk;
    }
    if (rc == PP_OK) rc = plan_lines(b, wk);
    if (rc == PP_OK) rc = autotune(b, st);
    if (rc == PP_OK && power_iters > 0) rc = batch_power_iteration(b, seed, power_iters, st);
    if (rc != PP_OK) {
        cudaStreamSynchronize(st);
        if (b.gexec) cudaGraphExecDestroy(b.gexec);
        if (b.cap_stream) cudaStreamDestroy(b.cap_stream);
        for (Plan* p : b.sub) {
            for (void* a : p->allocs) cudaFree(a);
            delete p;
        }
        for (void* a : b.allocs) cudaFree(a);
        delete h;
        return rc;
    }
    *out = h;
    return PP_OK;
}

pp_status pp_batch_destroy(pp_batch* batch) {
    if (!batch) return PP_OK;
    Batch& b = batch->impl;
    if (b.gexec) cudaGraphExecDestroy(b.gexec);
    if (b.cap_stream) cudaStreamDestroy(b.cap_stream);
    for (Plan* p : b.sub) {
        for (void* a : p->allocs) cudaFree(a);
        delete p;
    }
    for (void* a : b.allocs) cudaFree(a);
    delete batch;
    return PP_OK;
}

pp_status pp_batch_offsets(const pp_batch* batch, int64_t* image_off, int64_t* kspace_off) {
    if (!batch) {
        set_error("pp_batch_offsets: NULL batch");
        return PP_ERR_INVALID_ARG;
    }
    const Batch& b = batch->impl;
    for (int s = 0; s <= b.n; ++s) {
        if (image_off) image_off[s] = b.img_off[s];
        if (kspace_off) kspace_off[s] = b.ksp_off[s];
    }
    return PP_OK;
}

pp_status pp_batch_scales(const pp_batch* batch, double* L) {
    if (!batch || !L) {
        set_error("pp_batch_scales: NULL argument");
        return PP_ERR_INVALID_ARG;
    }
    for (int s = 0; s < batch->impl.n; ++s) L[s] = batch->impl.L[s];
    return PP_OK;
}

pp_status pp_batch_set_scales(pp_batch* batch, const double* L) {
    if (!batch || !L) {
        set_error("pp_batch_set_scales: NULL argument");
        return PP_ERR_INVALID_ARG;
    }
    Batch& b = batch->impl;
    for (int s = 0; s < b.n; ++s)
        if (!(L[s] > 0.0) || !isfinite(L[s])) {
            set_error("pp_batch_set_scales: L[%d] must be finite and > 0", s);
            return PP_ERR_INVALID_ARG;
        }
    for (int s = 0; s < b.n; ++s) {
        b.L[s] = L[s];
        b.sub[s]->L = L[s];
    }
    b.tape_key.clear();   // checkpoints taken under the old L_s are stale
    return upload_descs(b);
}

pp_status pp_batch_tile(const pp_batch* batch, int* cols_per_cta, int* persistent_ctas) {
    if (!batch) {
        set_error("pp_batch_tile: NULL batch");
        return PP_ERR_INVALID_ARG;
    }
    if (cols_per_cta)
        {
        const int w = batch->impl.dev.cols;
        *cols_per_cta = w ? (w == 8 ? -8 : (w == 1 ? -16 : -32)) : 1 << batch->impl.dev.lgt;
    }
    if (persistent_ctas) *persistent_ctas = batch->impl.dev.grid;
    return PP_OK;
}

pp_status pp_batch_set_tile(pp_batch* batch, int cols_per_cta) {
    if (!batch) {
        set_error("pp_batch_set_tile: NULL batch");
        return PP_ERR_INVALID_ARG;
    }
    Batch& b = batch->impl;
    std::vector<int2> items;
    if (cols_per_cta == -8 || cols_per_cta == -16 || cols_per_cta == -32) {
        for (const SliceDesc& d : b.hdesc)
            if (!cart_cols_width_ok(d.ny, 1)) {
                set_error("pp_batch_set_tile: slice length %d has no compiled column chain", d.ny);
                return PP_ERR_UNSUPPORTED;
            }
        PP_TRY(set_cols(b, cols_per_cta == -8 ? 8 : (cols_per_cta == -16 ? 1 : 4)));
    } else {
        const int lgt = cols_per_cta == 4 ? 2 : cols_per_cta == 8 ? 3 : cols_per_cta == 16 ? 4 : -1;
        if (lgt < 0 || !km_for(b.dev.ny_max, lgt)) {
            set_error("pp_batch_set_tile: unsupported tile width %d", cols_per_cta);
            return PP_ERR_UNSUPPORTED;
        }
        drop_groups(b);
        PP_TRY(set_items(b, lgt, &items));
    }
    b.gkey.clear();
    b.tape_key.clear();
    return PP_OK;
}

pp_status pp_batch_forward_apply(const pp_batch* batch, const pp_c64* x, pp_c64* y, pp_stream stream) {
    if (!batch || !x || !y) {
        set_error("pp_batch_forward_apply: NULL argument");
        return PP_ERR_INVALID_ARG;
    }
    return batch_forward(batch->impl, reinterpret_cast<const float2*>(x), reinterpret_cast<float2*>(y),
                         (cudaStream_t)stream);
}

pp_status pp_batch_adjoint_apply(const pp_batch* batch, const pp_c64* y, pp_c64* x, pp_stream stream) {
    if (!batch || !x || !y) {
        set_error("pp_batch_adjoint_apply: NULL argument");
        return PP_ERR_INVALID_ARG;
    }
    return batch_adjoint(batch->impl, reinterpret_cast<const float2*>(y), reinterpret_cast<float2*>(x),
                         (cudaStream_t)stream);
}

pp_status pp_batch_normal_apply(const pp_batch* batch, const pp_c64* x, pp_c64* y, pp_stream stream) {
    if (!batch || !x || !y || (const void*)x == (const void*)y) {
        set_error("pp_batch_normal_apply: NULL or aliased argument");
        return PP_ERR_INVALID_ARG;
    }
    return launch_batch_normal(batch->impl.dev, reinterpret_cast<const float2*>(x),
                               reinterpret_cast<float2*>(y), 1.f, nullptr, 0.f, (cudaStream_t)stream);
}

pp_status pp_batch_fista_solve(pp_batch* batch, const pp_c64* bk, float lambda, int iters,
                               const double* c, int d, pp_c64* x_out, pp_solve_info* info,
                               pp_stream stream) {
    if (!batch || !bk || !x_out || iters < 0 || iters > 1000000 || !(lambda >= 0.f) ||
        !isfinite(lambda) || d < 0 || d > 16 || (!c && d != 0)) {
        set_error("pp_batch_fista_solve: bad argument");
        return PP_ERR_INVALID_ARG;
    }
    if (info && info->levels && info->levels != 2) {
        set_error("pp_batch_fista_solve: batched prox supports 2 Haar levels only");
        return PP_ERR_UNSUPPORTED;
    }
    if (info && info->wavelet) {
        set_error("pp_batch_fista_solve: the batched prox is the 2-level Haar");
        return PP_ERR_UNSUPPORTED;
    }
    std::vector<double> c_safe;
    PP_TRY(safe_coeffs(info, c, d, c_safe));
    Batch& b = batch->impl;
    cudaStream_t st = (cudaStream_t)stream;
    const bool hist = info && info->history;
    const bool momentum = !(info && info->no_momentum);
    const float2* ref = info ? reinterpret_cast<const float2*>(info->ref) : nullptr;
    const int64_t launches0 = g_launches;
    const float2* bd = reinterpret_cast<const float2*>(bk);
    PP_TRY(launch_seg_dot(nullptr, bd, b.dev.ksp, b.partials, nullptr, b.scal + 0, 4, st));
    PP_TRY(batch_adjoint(b, bd, b.ahb, st));
    PP_TRY(launch_seg_scale(b.ahb, b.ahb, b.dev.img, b.scal + 0, 4, b.dfac, 1, st));
    PP_TRY_CUDA(cudaMemsetAsync(b.y, 0, b.nimg * sizeof(float2), st));
    PP_TRY_CUDA(cudaMemsetAsync(b.z, 0, b.nimg * sizeof(float2), st));
    if (hist) {
        if (b.hist_cap < iters) {
            if (b.hist) {
                cudaStreamSynchronize(st);
                cudaFree(b.hist);
                b.allocs.erase(std::remove(b.allocs.begin(), b.allocs.end(), (void*)b.hist), b.allocs.end());
                b.hist = nullptr;
            }
            PP_TRY(balloc(b, &b.hist, (size_t)3 * std::max(iters, 1)));
            b.hist_cap = iters;
            b.gkey.clear();
        }
        PP_TRY_CUDA(cudaMemsetAsync(b.hist, 0, sizeof(double) * 3 * std::max(iters, 1), st));
    }
    if (iters > 0) {
        std::vector<double> key = {(double)iters, (double)d, (double)lambda, hist ? 1.0 : 0.0,
                                   c ? 1.0 : 0.0, (double)(uintptr_t)b.hist, (double)(uintptr_t)ref,
                                   (double)b.dev.lgt, (double)b.dev.cols, momentum ? 1.0 : 0.0};
        if (c)
            for (int i = 0; i <= d; ++i) key.push_back(c[i]);
        if (!b.gexec || key != b.gkey) {
            if (b.gexec) {
                cudaGraphExecDestroy(b.gexec);
                b.gexec = nullptr;
            }
            b.gkey.clear();
            cudaGraph_t graph = nullptr;
            PP_TRY_CUDA(cudaStreamBeginCapture(b.cap_stream, cudaStreamCaptureModeThreadLocal));
            const int64_t before = g_launches;
            pp_status rc = batch_iterations(b, lambda, iters, c, d, hist, ref, momentum, b.cap_stream);
            cudaError_t e = cudaStreamEndCapture(b.cap_stream, &graph);
            b.graph_kernels = g_launches - before;
            g_launches = before;
            if (rc != PP_OK) {
                if (graph) cudaGraphDestroy(graph);
                return rc;
            }
            if (e != cudaSuccess) return cuda_status(e, "cudaStreamEndCapture");
            e = cudaGraphInstantiate(&b.gexec, graph, 0);
            cudaGraphDestroy(graph);
            if (e != cudaSuccess) {
                b.gexec = nullptr;
                return cuda_status(e, "cudaGraphInstantiate");
            }
            b.gkey = key;
        }
        PP_TRY_CUDA(cudaGraphLaunch(b.gexec, st));
    }
    float2* xo = reinterpret_cast<float2*>(x_out);
    if (info && info->rescale)
        PP_TRY(launch_seg_scale(b.y, xo, b.dev.img, b.scal + 0, 4, b.dfac, 0, st));
    else
        PP_TRY_CUDA(cudaMemcpyAsync(xo, b.y, b.nimg * sizeof(float2), cudaMemcpyDeviceToDevice, st));
    if (info) {
        info->L = b.L[0];
        info->launches = (g_launches - launches0) + (iters > 0 ? b.graph_kernels : 0);
        if (hist) {
            double bn2 = 0.0;
            PP_TRY_CUDA(cudaMemcpyAsync(&bn2, b.scal + 0, sizeof(double), cudaMemcpyDeviceToHost, st));
            PP_TRY_CUDA(cudaMemcpyAsync(info->history, b.hist, sizeof(double) * 3 * iters,
                                        cudaMemcpyDeviceToHost, st));
            PP_TRY_CUDA(cudaStreamSynchronize(st));
            PP_TRY(check_history("pp_batch_fista_solve", bn2, info->history, iters));
        }
    }
    return PP_OK;
}

static bool unrolled_args_ok(const pp_batch* batch, const void* bk, int iters, const double* c,
                             int d, int ce, float lambda) {
    return batch && bk && c && iters >= 1 && iters <= 100000 && d >= 0 && d <= 10 && ce >= 1 &&
           ce <= iters && lambda >= 0.f && isfinite(lambda);
}

// What the checkpoints of an unrolled forward depend on besides the contents
// of b: b's address, lambda, the iteration count, the polynomial, the
// checkpoint spacing and every slice's L_s.
static std::vector<double> tape_key_of(const Batch& B, const void* bk, float lambda, int iters,
                                       const double* c, int d, int ce) {
    std::vector<double> key = {(double)(uintptr_t)bk, (double)lambda, (double)iters, (double)d,
                               (double)ce};
    for (int i = 0; i <= d; ++i) key.push_back(c[i]);
    key.insert(key.end(), B.L.begin(), B.L.end());
    return key;
}

pp_status pp_batch_unrolled_forward(pp_batch* batch, const pp_c64* b, float lambda, int iters,
                                    const double* c, int d, int checkpoint_every, pp_c64* x_out,
                                    pp_stream stream) {
    if (!unrolled_args_ok(batch, b, iters, c, d, checkpoint_every, lambda) || !x_out) {
        set_error("pp_batch_unrolled_forward: bad argument");
        return PP_ERR_INVALID_ARG;
    }
    Batch& B = batch->impl;
    pp_status rc = unrolled_forward(B, reinterpret_cast<const float2*>(b), lambda, iters, c, d,
                                    checkpoint_every, reinterpret_cast<float2*>(x_out),
                                    (cudaStream_t)stream);
    if (rc != PP_OK) return rc;
    B.tape_key = tape_key_of(B, b, lambda, iters, c, d, checkpoint_every);
    return PP_OK;
}

pp_status pp_batch_unrolled_backward(pp_batch* batch, const pp_c64* b, float lambda, int iters,
                                     const double* c, int d, int checkpoint_every,
                                     const pp_c64* grad_out, pp_c64* grad_b, double* grad_lambda,
                                     double* grad_c, pp_stream stream) {
    if (!unrolled_args_ok(batch, b, iters, c, d, checkpoint_every, lambda) || !grad_out ||
        !grad_b || !grad_lambda || !grad_c) {
        set_error("pp_batch_unrolled_backward: bad argument");
        return PP_ERR_INVALID_ARG;
    }
    Batch& B = batch->impl;
    cudaStream_t st = (cudaStream_t)stream;
    const std::vector<double> key = tape_key_of(B, b, lambda, iters, c, d, checkpoint_every);
    if (key != B.tape_key) {
        // no matching forward on the tape: run it (its output goes to the solve buffer)
        PP_TRY(unrolled_forward(B, reinterpret_cast<const float2*>(b), lambda, iters, c, d,
                                checkpoint_every, B.w3, st));
        B.tape_key = key;
    }
    return unrolled_backward(B, lambda, iters, c, d, checkpoint_every,
                             reinterpret_cast<const float2*>(grad_out), reinterpret_cast<float2*>(grad_b),
                             grad_lambda, grad_c, st);
}

}  // extern "C"
