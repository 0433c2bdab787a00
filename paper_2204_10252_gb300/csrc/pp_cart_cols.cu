// Choice and launch of the column-resident Cartesian kernels (pp_cart_cols.cuh).
#include <algorithm>

#include "pp_batch.h"
#include "pp_lines_lengths.h"

namespace pp {

namespace {

struct Len {
    int n, n1, n2;
    cudaError_t (*launch)(const CartLaunch&, const float2*, const CartChain&, cudaStream_t);
};
#define PP_LEN_ROW(n, a, b) {n, a, b, cart_cols_launch<a, b>},
const Len kLens[] = {PP_CART_LENGTHS(PP_LEN_ROW)};
#undef PP_LEN_ROW

const Len* find(int n) {
    for (const Len& l : kLens)
        if (l.n == n) return &l;
    return nullptr;
}

size_t smem_of(const Len& l, int W, int NB) {
    const size_t n = l.n;
    return sizeof(float2) * (n + n / 2 + 2 * n * W + (size_t)l.n1 * (l.n2 | 1) * 8 * W + (size_t)NB * n * 8 * W);
}

}  // namespace

bool cart_cols_width_ok(int n, int W) {
    const Len* l = find(n);
    if (!l || !cart_width_ok(n, W)) return false;
    return W == 8 || smem_of(*l, W, 2) <= (size_t)kCartSmem;
}

pp_status launch_cart_cols(int n, CartLaunch L, const float2* x, const CartChain& ch, cudaStream_t st) {
    const Len* l = find(n);
    // The maps of all coil groups stay in shared memory for a chain of several
    // applications while every CTA that an SM would run then (its share of the
    // grid, four at most) still fits; otherwise they stream through two buffers.
    const int groups = (L.max_coils + 7) / 8;
    const int grid = L.items ? L.nitems : (L.one.nx + L.W - 1) / L.W;
    const int per_sm = std::min(4, (grid + 151) / 152);
    L.resident = groups <= 2 || (ch.J > 1 && l && per_sm * (smem_of(*l, L.W, groups) + 1024) <= (size_t)kCartSmem);
    // Streaming: the coils of an item over a cluster of up to four CTAs, while those of
    // all launches side by side still get an SM each and two coils are left to each
    // (256 x 256, us for 1 / 2 / 4 / 8 CTAs, when one rank still added up the last sum:
    // 18.4 / 12.7 / 10.7 / 38.6 at 16 coils, 63 / 36 / 22.4 / 52 at 64; more CTAs than SMs,
    // 320 x 320 x 12: 17.9 / 11.9 / 21.9; eight CTAs also where they fit, 128 x 128 x 32:
    // 18.1 / 11.6 / 8.0 / 15.0).  Then as many slots as bring 16 warps to every SM (what
    // 128 registers a thread allow), while two coils are left to each, or one where the
    // coils are split.  A lean launch stops where more slots only take the place of
    // CTAs (see the batch's timing).
    if (l && L.W == 8) {
        const int items = L.items ? L.nitems : (L.one.nx + 7) / 8;
        while (L.split < 4 && 2 * items * L.split + L.beside <= 152 && L.max_coils >= 4 * L.split) L.split *= 2;
        const int ctas = items * L.split, coils = L.max_coils / L.split, left = L.split > 1 ? 2 : 4;
        auto in_flight = [&](int slots) {   // slots on the fullest SM
            return std::min((ctas + 151) / 152, std::max(1, 512 / (8 * l->n2 * slots))) * slots;
        };
        while (L.slots < 4 && ctas * L.slots * 8 * l->n2 < 152 * 512 && coils >= left * L.slots &&
               (!L.lean || in_flight(2 * L.slots) > in_flight(L.slots)))
            L.slots *= 2;
    }
    cudaError_t e = l ? l->launch(L, x, ch, st) : cudaErrorInvalidValue;
    if (e != cudaSuccess) return cuda_status(e, "cart_cols_kernel launch");
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_status(e, "cart_cols_kernel");
    ++g_launches;
    if (g_profiler) g_profiler->mark("cart_cols_kernel");
    return PP_OK;
}

}  // namespace pp
