// Choice and launch of the compiled row and column FFT stages (pp_lines.cuh).
#include <algorithm>

#include "pp_lines.h"
#include "pp_lines_lengths.h"

namespace pp {
namespace {

struct Len {
    int n, n1, n2;
    cudaError_t (*launch)(LineOp, const LineUnion&, dim3, cudaStream_t);
};
#define PP_LINE_ROW(n, a, b) {n, a, b, line_launch<a, b>},
const Len kLens[] = {PP_LINE_LENGTHS(PP_LINE_ROW)};
#undef PP_LINE_ROW

const Len* find(int n) {
    for (const Len& l : kLens)
        if (l.n == n) return &l;
    return nullptr;
}

pp_status go(const char* what, int n, LineOp op, const LineUnion& u, dim3 grid, cudaStream_t st) {
    cudaError_t e = find(n)->launch(op, u, grid, st);
    if (e != cudaSuccess) return cuda_status(e, what);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_status(e, what);
    ++g_launches;
    if (g_profiler) g_profiler->mark(what);
    return PP_OK;
}

pp_status go_cols(LineOp op, const LineCols& L, int nbatch, cudaStream_t st) {
    LineUnion u;
    u.cols = &L;
    return go("line_cols_kernel", L.a.G, op, u, dim3((L.a.ncols + TXG - 1) / TXG, nbatch), st);
}

// Rows per CTA of the adjoint row stage: whole rows where they fill the GPU (152
// SMs, several CTAs each), else one row with its coils side by side.
int rows_per_cta(int64_t nrows, int ncoils) {
    int rb = RBG;
    while (rb > 1 && (nrows + rb - 1) / rb < 4 * 152 && RBG / rb * 2 <= std::max(1, ncoils)) rb >>= 1;
    return rb;
}

}  // namespace

bool lines_have(int n) { return find(n) != nullptr; }

GenSplit gen_split_of(int n) {
    GenSplit g;
    if (const Len* l = find(n)) {
        g.n1 = l->n1;
        g.n2 = l->n2;
    }
    return g;
}

pp_status launch_lines_cols(const DevFft& f, const ColArgs& a, const float2* src, float2* dst, bool inv,
                            const float2* ximg, int nimgs, cudaStream_t st, bool* done) {
    *done = false;
    // 32-bit offsets in a batch; the batch index is blockIdx.y
    if (!find(a.G) || (int64_t)a.G * a.ncols >= (1ll << 31) || a.nbatch > 65535) return PP_OK;
    *done = true;
    const LineCols L{f.twb, a, nullptr, src, dst, ximg, nimgs};
    return go_cols(ximg ? LineOp::ColsFwdImg : (inv ? LineOp::ColsInv : LineOp::ColsFwd), L, a.nbatch, st);
}

pp_status launch_lines_roundtrip(const DevFft& f, const ColArgs& a, const float* mask_fo,
                                 const float2* src, float2* dst, cudaStream_t st, bool* done) {
    *done = false;
    if (!find(a.G) || (int64_t)a.G * a.ncols >= (1ll << 31)) return PP_OK;
    *done = true;
    LineCols L{f.twb, a, nullptr, src, dst, nullptr, 1};
    L.a.mul_out = mask_fo;
    return go_cols(LineOp::RoundTrip, L, a.nbatch, st);
}

pp_status launch_lines_rows_fwd(const DevFft& f, const RowArgs& a, const float2* x, const float2* sens,
                                const float* wrow, const float* wcol, float2* out, int ncoils,
                                int64_t img_batch_stride, cudaStream_t st, bool* done) {
    *done = false;
    if (!find(a.G)) return PP_OK;
    *done = true;
    const LineRows L{f.twb, a, nullptr, x, img_batch_stride, sens, wrow, wcol, out, nullptr, 0.f, ncoils, RBG};
    LineUnion u;
    u.rows = &L;
    return go("line_rows_fwd_kernel", a.G, LineOp::RowsFwd, u, dim3((a.nrows + RBG - 1) / RBG, ncoils), st);
}

pp_status launch_lines_rows_adj(const DevFft& f, const RowArgs& a, const float2* src, const float2* sens,
                                const float* wrow, const float* wcol, float2* out, const float2* operand,
                                float alpha, int ncoils, cudaStream_t st, bool* done) {
    *done = false;
    if (!find(a.G) || a.n > 512) return PP_OK;
    *done = true;
    const int rb = rows_per_cta(a.nrows, ncoils);
    const LineRows L{f.twb, a, nullptr, src, 0, sens, wrow, wcol, out, operand, alpha, ncoils, rb};
    LineUnion u;
    u.rows = &L;
    return go("line_rows_adj_kernel", a.G, LineOp::RowsAdj, u, dim3((a.nrows + rb - 1) / rb), st);
}

// The stages over slices of one transform length n: columns (ncols of the widest
// slice, one item a batch) and rows (nrows of the tallest slice).
pp_status launch_lines_batch_cols(int n, const float2* tw, int ncols, const ColItem* items, int nitems,
                                  bool inv, const float2* src, float2* dst, cudaStream_t st) {
    LineCols L{};
    L.tw = tw;
    L.a.Hin = L.a.Hout = L.a.G = n;
    L.a.off_in = L.a.off_out = n / 2;
    L.a.ncols = ncols;
    L.a.scale = 1.f;
    L.a.mi_q = L.a.mo_q = L.a.mi_cdiv = L.a.mo_cdiv = 1;
    L.items = items;
    L.src = src;
    L.dst = dst;
    return go_cols(inv ? LineOp::ColsInv : LineOp::ColsFwd, L, nitems, st);
}

pp_status launch_lines_batch_rows(int n, const float2* tw, int nrows, const RowItem* items, int nitems,
                                  bool adj, int ncoils, float scale, const float2* src, float2* dst,
                                  cudaStream_t st) {
    LineRows L{};
    L.tw = tw;
    L.a.n = L.a.G = n;
    L.a.off_in = L.a.off_out = n / 2;
    L.a.nrows = nrows;
    L.a.scale = scale;
    L.items = items;
    L.src = src;
    L.dst = dst;
    L.ncoils = ncoils;
    L.rb = adj ? rows_per_cta((int64_t)nrows * nitems, ncoils) : RBG;
    LineUnion u;
    u.rows = &L;
    return go(adj ? "line_rows_adj_kernel" : "line_rows_fwd_kernel", n, adj ? LineOp::RowsAdj : LineOp::RowsFwd, u,
              dim3((nrows + L.rb - 1) / L.rb, nitems), st);
}

// 3-D normal operator, `chunk` coils at a time: y FFT of S_c x into W, z round
// trip in place, inverse y FFT with the coil sum.  W: chunk * nimg elements.
pp_status lines_cart3d_normal(const Plan& p, const float2* x, float2* out, float scale,
                              const float2* operand, float alpha, float2* W, int chunk, cudaStream_t st,
                              bool* done) {
    *done = false;
    if (!find(p.ny) || !find(p.nz) || p.nimg >= (1ll << 31)) return PP_OK;
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int64_t n = p.nimg;
    for (int c0 = 0; c0 < p.C; c0 += chunk) {
        const int nc = std::min(chunk, p.C - c0);
        const float2* S = p.sens + (int64_t)c0 * n;
        LineCols L{};
        L.tw = p.fy.twb;
        L.a.Hin = L.a.Hout = L.a.G = ny;
        L.a.ncols = nx;
        L.a.scale = 1.f;
        L.a.in_batch_stride = L.a.out_batch_stride = (int64_t)ny * nx;
        L.a.mi_cdiv = L.a.mo_cdiv = 1;
        L.src = S;
        L.dst = W;
        L.ximg = x;
        L.nimgs = nz;
        PP_TRY(go_cols(LineOp::ColsFwdImg, L, nc * nz, st));
        LineCols Z{};
        Z.tw = p.fz.twb;
        Z.a.Hin = Z.a.Hout = Z.a.G = nz;
        Z.a.ncols = ny * nx;
        Z.a.scale = 1.f;
        Z.a.in_batch_stride = Z.a.out_batch_stride = n;
        Z.a.mi_cdiv = 1;
        Z.a.mul_out = p.mask_fo;
        Z.a.mo_q = ny;
        Z.a.mo_c = 1;
        Z.a.mo_cdiv = nx;
        Z.src = W;
        Z.dst = W;
        PP_TRY(go_cols(LineOp::RoundTrip, Z, nc, st));
        const LineYinv Y{p.fy.twb, nx, n, nc, W, S, out, c0 == 0, c0 + nc == p.C, scale, operand, alpha};
        LineUnion u;
        u.yinv = &Y;
        PP_TRY(go("line_yinv_kernel", ny, LineOp::Yinv, u, dim3((nx + TXG - 1) / TXG, nz), st));
    }
    *done = true;
    return PP_OK;
}

}  // namespace pp
