// Arguments and launcher of the compiled row and column FFT stages (pp_lines.cuh).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "pp_internal.h"

namespace pp {

constexpr int TXG = 8;   // columns per CTA
constexpr int RBG = 8;   // lines (rows, or rows x coils) per CTA in the row stages

struct LineCols {
    const float2* tw;
    ColArgs a;
    const ColItem* items;     // one per batch, or NULL: a's strides
    const float2* src;
    float2* dst;
    const float2* ximg;       // XIMG: image multiplied into the input (batch b: image b % nimgs)
    int nimgs;
};
struct LineRows {
    const float2* tw;
    RowArgs a;
    const RowItem* items;     // one per (slice, coil) (forward) or slice (adjoint), or NULL
    const float2* src;
    int64_t src_batch_stride;
    const float2* sens;
    const float* wrow;
    const float* wcol;
    float2* dst;
    const float2* operand;
    float alpha;
    int ncoils, rb;
};
struct LineYinv {
    const float2* tw;
    int nx;
    int64_t nimg;
    int ncoils;
    const float2* W;
    const float2* S;
    float2* out;
    int first, last;
    float scale;
    const float2* operand;
    float alpha;
};

enum class LineOp { ColsFwd, ColsInv, ColsFwdImg, RoundTrip, Yinv, RowsFwd, RowsAdj };
union LineUnion {
    const LineCols* cols;
    const LineRows* rows;
    const LineYinv* yinv;
};
// One launch of a stage for the length of (N1, N2); defined in that length's unit.
template <int N1, int N2>
cudaError_t line_launch(LineOp op, const LineUnion& u, dim3 grid, cudaStream_t st);

}  // namespace pp
