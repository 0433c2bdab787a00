// Batched uneven 2-D Cartesian problems: device descriptors and launchers.
#pragma once
#include <vector>

#include "pp_internal.h"

namespace pp {

// Per-slice view used by the batched kernels.
struct SliceDesc {
    FftDesc fd;              // FFT along ky (length ny)
    const float2* tw;        // its twiddle table
    const float2* twb;       //   and the balanced one of the two-factor kernels
    const float2* sens;      // [C][ny][nx] (borrowed)
    const float* mask_fo;    // [ny], FFT order, times 1/ny
    int ny, nx, C;
    int64_t img_off;         // offset of the slice in concatenated images
    float invL;
};

// A partition of a concatenated array into segments (one per slice), and
// of a launch's blocks over those segments.  Device arrays.
struct Segments {
    int nseg = 0, nblocks = 0;
    int64_t* off = nullptr;        // [nseg + 1]
    int* blk_seg = nullptr;        // [nblocks]
    int* seg_first_blk = nullptr;  // [nseg + 1]
};

constexpr int kCartMaxChain = 18;
constexpr int kCartSmem = 220 * 1024;   // dynamic shared memory a CTA may take

// The chain of applications.  op_j = `ext` for j = 0 of a chain that starts with a
// gradient (v_first = 0), else v: the input (v_first = 1) or the first result.
struct CartChain {
    int J = 1;
    int v_first = 0;
    float sc[kCartMaxChain], al[kCartMaxChain];
    const float2* ext = nullptr;     // operand of the first application (NULL: none)
    float2* out = nullptr;           // last result
    float2* first_out = nullptr;     // result of the first application (needed by the streaming form
                                     //   of a longer chain with v_first = 0), or NULL
    float2* all_out = nullptr;       // result j at all_out + j * all_stride, or NULL
    int64_t all_stride = 0;
};

struct CartLaunch {
    SliceDesc one;                   // single slice (items == NULL)
    const SliceDesc* descs = nullptr;
    const int2* items = nullptr;     // (slice, first column)
    int nitems = 0;
    int W = 1;                       // columns per CTA: 1, 2, 4 (column-resident) or 8 (streaming)
    int slots = 1;                   // coils side by side in a streaming CTA
    int split = 1;                   // CTAs of a cluster that share a streaming item's coils
    int beside = 0;                  // items of the launches that run beside this one
    int max_coils = 1;               // largest coil count of the slices
    int resident = 1;                // maps of all coil groups in shared memory
    bool lean = false;               // a streaming CTA takes no more slots than raise those on an SM
    bool pdl = false;
    bool follows = false;            // runs beside the launch before it (same input)
};

// The slices of one length ny in a batch: column groups of W columns.
struct CartGroup {
    int n = 0, W = 1, max_coils = 1, nitems = 0;
    bool lean = false;       // see CartLaunch
    int2* items = nullptr;   // (slice, first column), most expensive first
};

// One launch of a row or column stage over a batch: the slices (and coils) of one
// transform length.
struct LineGroup {
    int n = 0, extent = 0, ncoils = 1, nitems = 0;   // extent: most columns or rows of a slice
    const float2* tw = nullptr;
    void* items = nullptr;   // ColItem or RowItem
};
// Slices whose k-space fits the workspace together: column stage into it, row
// stage out of it.
struct AdjointChunk {
    std::vector<LineGroup> cols, rows;
};

struct BatchDev {
    SliceDesc* descs = nullptr;
    int2* items = nullptr;   // (slice, first column), most expensive first
    int nitems = 0, ny_max = 0, km = 0, lgt = 3, grid = 0;
    int cols = 0;            // > 0: the column-resident kernels run, one launch per length, a
                             //   chain on `cols` columns per CTA (fewer where a length has no such
                             //   form)
    std::vector<CartGroup> groups, one;   // of chains, of a single application (or the same lists)
    Segments img, ksp, tiles;
};

// One iteration of the reverse pass at the Horner recursion, v_0 = wbar and
// v_i = v + (i - 1) * n, i = 1 .. d + 1.
constexpr int kTileThreads = 128;   // threads per CTA of the 4 x 4 tile kernels, four a tile
constexpr int kRevBlocks = 4 * 152;
struct RevCombine {
    int d;
    float c[11];
    const float2 *wbar, *v, *g;
    int64_t n;
    float2 *Zbar, *ahb_bar;
    double* partials;   // [kRevBlocks][d + 1]
};

size_t batch_normal_smem(int ny_max, int lgt);
void* batch_normal_fn(int km, int lgt);
pp_status configure_batch_kernels();
// Columns per CTA that are compiled: 4 where the tile of one coil group leaves
// room for two map buffers (n <= 256).
// 8: the streaming form.
constexpr bool cart_width_ok(int n, int W) { return W == 1 || W == 2 || W == 8 || (W == 4 && n <= 256); }
// One launch for the length of (N1, N2); defined in that length's unit.
template <int N1, int N2>
cudaError_t cart_cols_launch(const CartLaunch& L, const float2* x, const CartChain& ch, cudaStream_t st);
// Whether the column-resident kernel is compiled for length n and W columns.
bool cart_cols_width_ok(int n, int W);
pp_status launch_cart_cols(int n, CartLaunch L, const float2* x, const CartChain& ch, cudaStream_t st);
// a chain of applications on every slice (b.cols > 0)
pp_status launch_batch_chain(const BatchDev& b, const float2* x, const CartChain& ch, cudaStream_t st);
pp_status launch_batch_normal(const BatchDev& b, const float2* x, float2* out, float coef,
                              const float2* operand, float alpha, cudaStream_t st);
pp_status launch_seg_dot(const float2* a, const float2* bv, const Segments& sg, double* partials,
                         double* out_re, double* out_nb, int stride, cudaStream_t st);
pp_status launch_seg_scale(const float2* in, float2* out, const Segments& sg, const double* norm2,
                           int stride, const double* factor, int invert, cudaStream_t st);
pp_status launch_batch_prox_fista(const BatchDev& b, float lam, float gamma, float beta,
                                  float2* z, const float2* u, float2* y, float2* w_out, const float2* ref,
                                  double* hist, cudaStream_t st);

pp_status launch_batch_prox_vjp(const BatchDev& b, float lam, float beta, const float2* w,
                                float2* Ybar, const float2* Zbar, float2* wbar, double* lam_bar,
                                cudaStream_t st);
// dots[0 .. d] = Re<v_i, g> and the two linear combinations
pp_status launch_rev_combine(const RevCombine& r, double* dots, cudaStream_t st);

}  // namespace pp
