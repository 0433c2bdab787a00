// Locally-low-rank prox (the LLR regulariser of the MRF experiment, Sec. 5.3):
// for every block of block^ndim voxels (non-overlapping, after a circular
// shift of the volume), the Casorati matrix M (one row per voxel, one column
// per coefficient image) is replaced by U max(S - lambda, 0) V^H, its
// singular values soft-thresholded.
//
// One CTA per block, the matrix in registers (RPT rows of T columns a thread).
// The SVD goes through the T x T Gram matrix twice:
//   H  = M^H M   (one block reduction), Jacobi eigenvectors V0, M1 = M V0;
//   H1 = M1^H M1 (one block reduction), Jacobi eigenvectors V1, V = V0 V1;
//   out = M1 Q,  Q = V1 diag(max(0, 1 - lambda / s_i)) V^H,  s_i^2 the
//   eigenvalues of H1.
// The rounding of H is relative to its largest eigenvalue, so V0 leaves the
// columns of M1 orthogonal only to about 2^-24 s_1^2 / (s_i s_j).  H1 is formed
// from those columns themselves: each of its entries is accurate relative to
// |a_i| |a_j|, and Jacobi with a relative threshold keeps that accuracy, as
// one-sided Jacobi on M does (its rotations leave the same 2^-24 s_1 in every
// column).  Rows meet in two block reductions instead of one for each of the
// T'-1 rounds of every sweep, and are rotated twice instead of in every round:
// five images of 128 x 256 x 256 with 8^3 blocks (0.67 GB in and out) took
// 877 us with one-sided Jacobi over the rows (issue bound: 60 % of issue slots)
// and take 348 us (1930 GB/s).
//
// The T x T eigenproblems run in one warp, a lane per matrix element: the
// rounds of disjoint pairs (round-robin schedule, T' = T rounded up to even)
// are exact in either order, so a round updates A <- J^H A J and V <- V J out
// of one shared buffer into another with one warp barrier.  Their serial chain
// (about 25 rounds) is hidden by the other CTAs of the SM.
#include <cuda_runtime.h>
#include <stdint.h>

#include "pp_fft.cuh"
#include "pp_internal.h"

namespace pp {
namespace {

constexpr int kLlrSweeps = 12;

struct LlrArgs {
    const float2* in;
    float2* out;
    int64_t nimg;          // voxels per coefficient image
    int nx, ny, nz, ndim;
    int block, lb;         // block edge and log2
    int sx, sy, sz;        // circular shift of the block grid
    int nbx, nby;          // blocks per axis (x, y)
    int R;                 // voxels per block
    float lam;
};

// Partner of index i in round r of the round-robin schedule (circle method) of
// TP players: r and TP - 1 meet, the others pair to a sum of 2r mod (TP - 1).
template <int TP>
__device__ __forceinline__ int rr_partner(int r, int i) {
    if (i == TP - 1) return r;
    if (i == r) return TP - 1;
    int j = 2 * r - i;
    j += j < 0 ? TP - 1 : 0;
    return j >= TP - 1 ? j - (TP - 1) : j;
}

// The T^2 floats of the Gram matrix of the block's rows, as a T x T array:
// |a_i|^2 at (i, i), Re a_i^H a_j at (i, j) and Im a_i^H a_j at (j, i), i < j; one row
// a warp in `buf`.  Within a warp a butterfly reduce-scatter halves the values each
// step (31 shuffles for 32 values instead of 5 for each), which leaves value l of a
// chunk with lane l; the 1 or 4 values of one or two images go to the lowest lanes,
// and the others' sums are added (5 or 6 shuffles).
template <int T, int RPT, int NT>
__device__ __forceinline__ void gram_partials(const float2 (&m)[RPT][T], float (*buf)[64]) {
    constexpr int NV = T <= 2 ? T * T : 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int base = 0; base < T * T; base += NV) {
        float t[NV];
#pragma unroll
        for (int e = 0; e < NV; ++e) {
            const int i = (base + e) / T, j = (base + e) % T;
            float acc = 0.f;
            if (base + e < T * T && i <= j) {
                float2 p = make_float2(0.f, 0.f);
#pragma unroll
                for (int q = 0; q < RPT; ++q) p = __ffma2_rn(m[q][i], m[q][j], p);
                acc = p.x + p.y;
            } else if (base + e < T * T) {
#pragma unroll
                for (int q = 0; q < RPT; ++q)
                    acc = fmaf(m[q][j].x, m[q][i].y, fmaf(-m[q][j].y, m[q][i].x, acc));
            }
            t[e] = acc;
        }
#pragma unroll
        for (int h = NV / 2; h >= 1; h >>= 1) {
            const bool up = (lane & h) != 0;
#pragma unroll
            for (int i = 0; i < h; ++i) {
                const float send = up ? t[i] : t[i + h];
                const float keep = up ? t[i + h] : t[i];
                t[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
            }
        }
#pragma unroll
        for (int h = NV; h < 32; h <<= 1) t[0] += __shfl_xor_sync(0xffffffffu, t[0], h);
        if (lane < NV) buf[w][base + lane] = t[0];
    }
}

__device__ __forceinline__ float2 shfl2(float2 v, int src) {
    return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// 1 / sqrt(x) with one Newton step, so that rotations do not stretch: relative
// errors of 2^-22 in their lengths would add up over the rounds.  Error of the prox
// against 64 bits: 2.4e-7 for five images, 4.2e-7 without the step (3.9e-7 with
// one-sided Jacobi); 4e-7, 1.0e-6 (9.5e-7) for eight.  It costs 12 us of the 369.
__device__ __forceinline__ float rsqrt_nr(float x) {
    const float r = rsqrtf(x);
    return fmaf(0.5f * r, fmaf(-x * r, r, 1.f), r);
}

// Column k's share of the rotation that makes columns k and k2 of the Hermitian
// A orthogonal: new column k = alpha * column k + beta * column k2.  Returns
// |a_k^H a_k2| / (|a_k| |a_k2|), 0 where it is at most tol.
template <int T>
__device__ __forceinline__ float jacobi_pair(const float2 (*A)[T], int k, int k2, float tol,
                                             float2* alpha, float2* beta) {
    *alpha = make_float2(1.f, 0.f);
    *beta = make_float2(0.f, 0.f);
    if (k2 >= T) return 0.f;
    const int i = min(k, k2), j = max(k, k2);
    const float al = A[i][i].x, be = A[j][j].x;
    const float2 gm = A[i][j];
    const float g2 = gm.x * gm.x + gm.y * gm.y, lim = tol * tol * al * be;
    if (!(g2 > fmaxf(lim, 1e-38f))) return 0.f;
    // real symmetric Schur rotation of [[al, g], [g, be]] after the phase
    // conj(gamma)/|gamma| on column j that makes gamma real; any t serves, c and
    // sn follow from it
    const float rg = rsqrt_nr(g2), g = g2 * rg;
    const float zeta = 0.5f * (be - al) * rg;
    const float z1 = fminf(fmaf(zeta, zeta, 1.f), 1e30f);
    const float t = __fdividef(copysignf(1.f, zeta), fabsf(zeta) + z1 * rsqrtf(z1));
    const float c = rsqrt_nr(fmaf(t, t, 1.f)), sn = c * t;
    const float2 ph = make_float2(gm.x * rg, -gm.y * rg);
    const bool up = k == i;
    *alpha = make_float2(up ? c : c * ph.x, up ? 0.f : c * ph.y);
    *beta = make_float2(up ? -sn * ph.x : sn, up ? -sn * ph.y : 0.f);
    // al * be <= 0 only through rounding: count it as not yet orthogonal
    return lim > 0.f ? g * rsqrtf(al * be) : 1.f;
}

// Eigenvectors of the Hermitian T x T matrix A[0] by Jacobi rotations in one
// warp; sweeps until every |a_ij| <= tol sqrt(a_ii a_jj) before its rotation,
// or `last` at the start of the sweep.  Returns the buffer (0 or 1) that holds
// the result; V[that] holds the eigenvectors in its columns.
template <int T>
__device__ __forceinline__ int warp_jacobi(float2 (*A)[T][T], float2 (*V)[T][T], float tol,
                                           float last) {
    constexpr int TP = T + (T & 1), NE = (T * T + 31) / 32;
    const int lane = threadIdx.x & 31;
    int cur = 0;
#pragma unroll
    for (int q = 0; q < NE; ++q) {
        const int e = lane + 32 * q;
        if (e < T * T) V[0][e / T][e % T] = make_float2(e / T == e % T ? 1.f : 0.f, 0.f);
    }
    __syncwarp();
    const int kc = min(lane, T - 1);
    for (int sweep = 0; T > 1 && sweep < kLlrSweeps; ++sweep) {
        float off = 0.f;
#pragma unroll 1
        for (int r = 0; r < TP - 1; ++r) {
            const float2(*Ac)[T] = A[cur];
            const float2(*Vc)[T] = V[cur];
            // lane k < T works out column k's rotation, the others ask for it
            float2 al, be;
            off = fmaxf(off, jacobi_pair<T>(Ac, kc, rr_partner<TP>(r, kc), tol, &al, &be));
#pragma unroll
            for (int q = 0; q < NE; ++q) {
                const int e = lane + 32 * q, i = min(e / T, T - 1), k = e % T;
                const float2 ai = shfl2(al, i), bi = shfl2(be, i), ak = shfl2(al, k), bk = shfl2(be, k);
                if (e < T * T) {
                    const int i2 = rr_partner<TP>(r, i), k2 = rr_partner<TP>(r, k);
                    const int i3 = i2 < T ? i2 : i, k3 = k2 < T ? k2 : k;   // idle: beta = 0
                    const float2 s0 = cadd(cmul(Ac[i][k], ak), cmul(Ac[i][k3], bk));
                    const float2 s1 = cadd(cmul(Ac[i3][k], ak), cmul(Ac[i3][k3], bk));
                    A[cur ^ 1][i][k] = cadd(cmulc(ai, s0), cmulc(bi, s1));
                    V[cur ^ 1][i][k] = cadd(cmul(Vc[i][k], ak), cmul(Vc[i][k3], bk));
                }
            }
            cur ^= 1;
            __syncwarp();
        }
        off = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(off)));
        if (off <= last) break;
    }
    return cur;
}

// Offset of voxel `row` of block `b` in one coefficient image.
__device__ __forceinline__ int64_t llr_voxel(const LlrArgs& a, int b, int row) {
    const int m = a.block - 1;
    const int bx = b % a.nbx, byz = b / a.nbx, by = byz % a.nby, bz = byz / a.nby;
    const int dx = row & m, dy = (row >> a.lb) & m, dz = row >> (2 * a.lb);
    int x = bx * a.block + dx + a.sx, y = by * a.block + dy + a.sy;
    x -= x >= a.nx ? a.nx : 0;
    y -= y >= a.ny ? a.ny : 0;
    if (a.ndim == 2) return (int64_t)y * a.nx + x;
    int z = bz * a.block + dz + a.sz;
    z -= z >= a.nz ? a.nz : 0;
    return ((int64_t)z * a.ny + y) * a.nx + x;
}

// At most 80 registers a thread: 6 CTAs of 128 threads an SM.  One-warp CTAs are
// left uncapped (up to 103 registers).  Capped, their results are the same; a few
// blocks take longer (256 x 240 in 8 x 8 blocks: 30.7 -> 32.9 us for seven images,
// 32.9 -> 35.0 for eight) and many are faster (64 x 256 x 256 in 4^3 blocks: 1004 ->
// 935 us for seven, 1008 -> 910 for eight).
__host__ __device__ constexpr int llr_min_ctas(int nt) { return nt > 32 ? 65536 / (nt * 80) : 0; }

// A trace of the Gram matrix whose reciprocal, or whose terms, leave the range of
// FP32: the first product only scales the rows, by this, and the second Gram matrix
// is the only one.  2^100: no |x| is above 1e-14 there, and the squares of the
// smallest FP32 numbers become 2^-98; 2^-80: the largest become 2^96.  A trace of 0
// needs nothing (every output is 0), and a NaN stays one.  All of it is the first
// warp's: forming the Gram matrix once more instead cost 3 to 15 % of the prox
// (registers), this nothing to 2 % (five images 128 x 256 x 256: 355 -> 348 us, two
// images 64 x 256 x 256: 57.4 -> 58.9).
__device__ __forceinline__ float llr_unit(float trace) {
    if (trace > 0.f && trace < 1e-28f) return 0x1p100f;
    return trace == __int_as_float(0x7f800000) ? 0x1p-80f : 1.f;
}

// The same for one or two images, whose T x T problem is at most one rotation: every
// thread solves it in its own registers, so that no warp waits for the first one's and
// a pass has one barrier, and one image takes one pass.  us, one-sided Jacobi over the
// rows / llr_prox_kernel / here: 64 x 256 x 256 in 8^3 blocks, one image 20.2 / 35.2 / 21.1,
// two 41.6 / 58.1 / 41.7; in 4^3 blocks 37.5 / 48.7 / 37.8 and 74.0 / 91.2 / 54.1; 1024 x 1024
// in 4 x 4 blocks, two 37.3 / 66.2 / 39.5.  Error against 64 bits: 1.1e-7 to 1.4e-7 for
// two images (1.1e-7 to 1.6e-7 before).  Three images so (with sweeps): 102 -> 174 us in
// 8^3 blocks, 190 -> 238 in 4 x 4; these, alone, stay slower than with one-sided
// Jacobi in 4 x 4 blocks (136 us), whose error was 2.8e-7 against 2.3e-7.
template <int T> struct LlrSmall {
    float2 A[T][T], V[T][T];   // Hermitian matrix; its eigenvectors in V's columns

    __device__ __forceinline__ void set(const float (&g)[T * T], float sc) {
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int k = i; k < T; ++k) {
                const float2 v = make_float2(g[i * T + k] * sc, i == k ? 0.f : g[k * T + i] * sc);
                A[i][k] = v;
                A[k][i] = make_float2(v.x, -v.y);
            }
        identity();
    }
    __device__ __forceinline__ void identity() {
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int k = 0; k < T; ++k) V[i][k] = make_float2(i == k ? 1.f : 0.f, 0.f);
    }
    // A <- J^H A J, V = J for the rotation that makes a 2 x 2 matrix diagonal
    __device__ __forceinline__ void rotate(float tol) {
        constexpr int j = T - 1;
        float2 ai, bi, aj, bj;
        jacobi_pair<T>(A, 0, j, tol, &ai, &bi);
        jacobi_pair<T>(A, j, 0, tol, &aj, &bj);
        V[0][0] = ai;
        V[j][0] = bi;
        V[0][j] = bj;
        V[j][j] = aj;
#pragma unroll
        for (int k = 0; k < T; ++k) {
            const float2 p = A[k][0], q = A[k][j];
            A[k][0] = cadd(cmul(p, ai), cmul(q, bi));
            A[k][j] = cadd(cmul(q, aj), cmul(p, bj));
        }
#pragma unroll
        for (int k = 0; k < T; ++k) {
            const float2 p = A[0][k], q = A[j][k];
            A[0][k] = cadd(cmulc(ai, p), cmulc(bi, q));
            A[j][k] = cadd(cmulc(aj, q), cmulc(bj, p));
        }
    }
};

template <int T, int RPT, int NT>
__device__ __forceinline__ void gram_sums(const float2 (&m)[RPT][T], float (*part)[64], float (&g)[T * T]) {
    gram_partials<T, RPT, NT>(m, part);
    __syncthreads();
#pragma unroll
    for (int e = 0; e < T * T; ++e) {
        g[e] = part[0][e];
#pragma unroll
        for (int w = 1; w < NT / 32; ++w) g[e] += part[w][e];
    }
}

template <int T, int RPT, int NT>
__global__ void __launch_bounds__(NT) llr_small_kernel(LlrArgs a) {
    __shared__ float part[2][NT / 32][64];
    float2 m[RPT][T];
    int64_t off[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int row = threadIdx.x + q * NT;
        off[q] = row < a.R ? llr_voxel(a, blockIdx.x, row) : -1;
#pragma unroll
        for (int t = 0; t < T; ++t)
            m[q][t] = off[q] >= 0 ? a.in[t * a.nimg + off[q]] : make_float2(0.f, 0.f);
    }
    const float tol = sqrtf((float)a.R) * 5.9604645e-8f;
    auto trace_of = [](const float (&g)[T * T]) {
        float tr = g[0];
#pragma unroll
        for (int i = 1; i < T; ++i) tr += g[i * T + i];
        return tr;
    };
    auto inverse = [](float tr) { return tr > 0.f ? 1.f / tr : (tr == 0.f ? 0.f : tr); };
    float g[T * T];
    gram_sums<T, RPT, NT>(m, part[0], g);
    float tr = trace_of(g);
    const float unit = llr_unit(tr);
    LlrSmall<T> H;
    float2 V0[T][T];
    H.set(g, inverse(tr));
    if (unit != 1.f) {   // the first pass only scales, as in llr_prox_kernel
#pragma unroll
        for (int q = 0; q < RPT; ++q)
#pragma unroll
            for (int k = 0; k < T; ++k) m[q][k] = cscale(m[q][k], unit);
    } else if (T > 1) {
        H.rotate(tol);
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            float2 y[T];
#pragma unroll
            for (int k = 0; k < T; ++k) {
                y[k] = cmul(m[q][0], H.V[0][k]);
#pragma unroll
                for (int i = 1; i < T; ++i) y[k] = cadd(y[k], cmul(m[q][i], H.V[i][k]));
            }
#pragma unroll
            for (int k = 0; k < T; ++k) m[q][k] = y[k];
        }
    }
#pragma unroll
    for (int i = 0; i < T; ++i)
#pragma unroll
        for (int k = 0; k < T; ++k) V0[i][k] = H.V[i][k];
    if (T > 1 || unit != 1.f) {
        gram_sums<T, RPT, NT>(m, part[1], g);
        tr = trace_of(g);
        H.set(g, inverse(tr));
        if (T > 1) H.rotate(tol);
    }
    const float lam = a.lam * unit, back = 1.f / unit;
    float2 Q[T][T];   // V1 F V^H with V = V0 V1
    float f[T];
#pragma unroll
    for (int l = 0; l < T; ++l) {
        // s <= lambda (also s = 0) -> 0; a NaN fails the test and stays NaN
        const float d = H.A[l][l].x * tr;
        const float sg = d < 0.f ? 0.f : sqrtf(d);
        f[l] = sg <= lam ? 0.f : (1.f - lam / sg) * back;
    }
#pragma unroll
    for (int k = 0; k < T; ++k) {
        float2 v[T];
#pragma unroll
        for (int l = 0; l < T; ++l) {
            v[l] = cmul(V0[k][0], H.V[0][l]);
#pragma unroll
            for (int i = 1; i < T; ++i) v[l] = cadd(v[l], cmul(V0[k][i], H.V[i][l]));
        }
#pragma unroll
        for (int i = 0; i < T; ++i) {
            Q[i][k] = cscale(cmulc(v[0], H.V[i][0]), f[0]);
#pragma unroll
            for (int l = 1; l < T; ++l) Q[i][k] = cadd(Q[i][k], cscale(cmulc(v[l], H.V[i][l]), f[l]));
        }
    }
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        if (off[q] < 0) continue;
#pragma unroll
        for (int k = 0; k < T; ++k) {
            float2 y = cmul(m[q][0], Q[0][k]);
#pragma unroll
            for (int i = 1; i < T; ++i) y = cadd(y, cmul(m[q][i], Q[i][k]));
            a.out[k * a.nimg + off[q]] = y;
        }
    }
}

template <int T, int RPT, int NT>
__global__ void __launch_bounds__(NT, llr_min_ctas(NT)) llr_prox_kernel(LlrArgs a) {
    __shared__ float part[NT / 32][64];
    __shared__ float2 A[2][T][T], V0[2][T][T], V1[2][T][T];
    __shared__ float4 W[T][T];   // (x, x, -y, y) of the T x T factor applied to the rows
    __shared__ float trace, unit;
    const int b = blockIdx.x;
    const int lane = threadIdx.x & 31;
    float2 m[RPT][T];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int row = threadIdx.x + q * NT;
        const bool live = row < a.R;
        const int64_t off = live ? llr_voxel(a, b, row) : 0;
#pragma unroll
        for (int t = 0; t < T; ++t)
            m[q][t] = live ? a.in[t * a.nimg + off] : make_float2(0.f, 0.f);
    }
    const float tol = sqrtf((float)a.R) * 5.9604645e-8f;
    int c0 = 0;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        gram_partials<T, RPT, NT>(m, part);
        __syncthreads();
        if (threadIdx.x < 32) {
            // sum the warps' rows; scale by 1 / trace (pass 0's) against over- and underflow
            float g[(T * T + 31) / 32];
            float tr = 0.f;
#pragma unroll
            for (int q = 0; q < (T * T + 31) / 32; ++q) {
                const int e = lane + 32 * q;
                float acc = 0.f;
                if (e < T * T)
#pragma unroll
                    for (int w = 0; w < NT / 32; ++w) acc += part[w][e];
                g[q] = acc;
                if (e < T * T && e / T == e % T) tr += acc;
            }
            if (pass == 0 || unit != 1.f) {
#pragma unroll
                for (int o = 16; o; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
                __syncwarp();
                if (lane == 0) {
                    trace = tr;
                    if (pass == 0) unit = llr_unit(tr);
                }
                __syncwarp();
            }
            tr = trace;
            const float sc = tr > 0.f ? 1.f / tr : (tr == 0.f ? 0.f : tr);
            const bool skip = pass == 0 && unit != 1.f;   // A = 0: no rotations, V0 = I
#pragma unroll
            for (int q = 0; q < (T * T + 31) / 32; ++q) {
                const int e = lane + 32 * q, i = e / T, k = e - i * T;
                if (e < T * T) {
                    const float v = skip ? 0.f : g[q] * sc;
                    if (i == k) {
                        A[0][i][i] = make_float2(v, 0.f);
                    } else if (i < k) {
                        A[0][i][k].x = v;
                        A[0][k][i].x = v;
                    } else {
                        A[0][k][i].y = v;
                        A[0][i][k].y = -v;
                    }
                }
            }
            __syncwarp();
            if (pass == 0) {
                // near-orthogonal columns are enough here: stop after the sweep
                // that met nothing above 0.03 (its rotations leave the square)
                c0 = warp_jacobi<T>(A, V0, tol, 3e-2f);
#pragma unroll
                for (int q = 0; q < (T * T + 31) / 32; ++q) {
                    const int e = lane + 32 * q;
                    if (e < T * T) {
                        const float2 v = cscale((&V0[c0][0][0])[e], unit);
                        (&W[0][0])[e] = make_float4(v.x, v.x, -v.y, v.y);
                    }
                }
            } else {
                const int c1 = warp_jacobi<T>(A, V1, tol, 1e-3f);
                const float lam = a.lam * unit, back = 1.f / unit;
                // W = V1 F V^H with V = V0 V1; V goes to the buffer of A not in use
#pragma unroll
                for (int q = 0; q < (T * T + 31) / 32; ++q) {
                    const int e = lane + 32 * q, i = e / T, k = e - i * T;
                    if (e < T * T) {
                        float2 s = make_float2(0.f, 0.f);
#pragma unroll
                        for (int l = 0; l < T; ++l) s = cadd(s, cmul(V0[c0][i][l], V1[c1][l][k]));
                        A[c1 ^ 1][i][k] = s;
                    }
                }
                __syncwarp();
#pragma unroll
                for (int q = 0; q < (T * T + 31) / 32; ++q) {
                    const int e = lane + 32 * q, i = e / T, k = e - i * T;
                    if (e < T * T) {
                        float2 s = make_float2(0.f, 0.f);
#pragma unroll
                        for (int l = 0; l < T; ++l) {
                            // s <= lambda (also s = 0) -> 0; a NaN fails the test and stays NaN
                            const float d = A[c1][l][l].x * tr;
                            const float sg = d < 0.f ? 0.f : sqrtf(d);
                            const float f = sg <= lam ? 0.f : (1.f - lam / sg) * back;
                            const float2 v = A[c1 ^ 1][k][l];
                            s = cadd(s, cscale(cmulc(v, V1[c1][i][l]), f));
                        }
                        W[i][k] = make_float4(s.x, s.x, -s.y, s.y);
                    }
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            float2 y[T];
#pragma unroll
            for (int k = 0; k < T; ++k) y[k] = make_float2(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < T; ++i) {
                const float2 u = m[q][i], us = make_float2(u.y, u.x);
#pragma unroll
                for (int k = 0; k < T; ++k) {
                    const float4 w = W[i][k];
                    y[k] = __ffma2_rn(u, make_float2(w.x, w.y), y[k]);
                    y[k] = __ffma2_rn(us, make_float2(w.z, w.w), y[k]);
                }
            }
#pragma unroll
            for (int k = 0; k < T; ++k) m[q][k] = y[k];
        }
    }
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int row = threadIdx.x + q * NT;
        if (row >= a.R) continue;
        const int64_t off = llr_voxel(a, b, row);
#pragma unroll
        for (int k = 0; k < T; ++k) a.out[k * a.nimg + off] = m[q][k];
    }
}

template <int T>
cudaError_t llr_launch_t(const LlrArgs& a, int nblocks, cudaStream_t st) {
    if constexpr (T <= 2) {
        if (a.R > 256) llr_small_kernel<T, 4, 128><<<nblocks, 128, 0, st>>>(a);
        else if (a.R > 64) llr_small_kernel<T, 4, 64><<<nblocks, 64, 0, st>>>(a);
        else if (a.R > 32) llr_small_kernel<T, 2, 32><<<nblocks, 32, 0, st>>>(a);
        else llr_small_kernel<T, 1, 32><<<nblocks, 32, 0, st>>>(a);
        return cudaGetLastError();
    } else {
        // R = 512, 256, 64 or 16 rows: few warps a block, so that few wait for the
        // one that solves the eigenproblems; up to 20 matrix elements a thread
        if (a.R > 256) {
            if constexpr (T <= 5) llr_prox_kernel<T, 4, 128><<<nblocks, 128, 0, st>>>(a);
            else llr_prox_kernel<T, 2, 256><<<nblocks, 256, 0, st>>>(a);
        } else if (a.R > 64) {
            if constexpr (T <= 5) llr_prox_kernel<T, 4, 64><<<nblocks, 64, 0, st>>>(a);
            else llr_prox_kernel<T, 2, 128><<<nblocks, 128, 0, st>>>(a);
        } else if (a.R > 32) {
            llr_prox_kernel<T, 2, 32><<<nblocks, 32, 0, st>>>(a);
        } else {
            llr_prox_kernel<T, 1, 32><<<nblocks, 32, 0, st>>>(a);
        }
        return cudaGetLastError();
    }
}

}  // namespace

extern thread_local int64_t g_launches;
extern thread_local Profiler* g_profiler;

pp_status launch_prox_llr(int ndim, int nx, int ny, int nz, int T, int block, const int* shift,
                          float lambda, const float2* in, float2* out, cudaStream_t st) {
    LlrArgs a;
    a.in = in; a.out = out;
    a.ndim = ndim; a.nx = nx; a.ny = ny; a.nz = ndim == 3 ? nz : 1;
    a.nimg = (int64_t)nx * ny * a.nz;
    a.block = block;
    a.lb = block == 4 ? 2 : (block == 8 ? 3 : 4);
    auto wrap = [](int s, int n) { s %= n; return s < 0 ? s + n : s; };
    a.sx = shift ? wrap(shift[0], nx) : 0;
    a.sy = shift ? wrap(shift[1], ny) : 0;
    a.sz = (shift && ndim == 3) ? wrap(shift[2], a.nz) : 0;
    a.nbx = nx / block;
    a.nby = ny / block;
    a.R = ndim == 3 ? block * block * block : block * block;
    a.lam = lambda;
    const int64_t nblocks = (int64_t)a.nbx * a.nby * (ndim == 3 ? a.nz / block : 1);
    if (nblocks <= 0) return PP_OK;
    if (nblocks > 0x7fffffff) {
        set_error("pp_prox_llr: too many blocks");
        return PP_ERR_UNSUPPORTED;
    }
    cudaError_t e = cudaErrorInvalidValue;
    switch (T) {
        case 1: e = llr_launch_t<1>(a, (int)nblocks, st); break;
        case 2: e = llr_launch_t<2>(a, (int)nblocks, st); break;
        case 3: e = llr_launch_t<3>(a, (int)nblocks, st); break;
        case 4: e = llr_launch_t<4>(a, (int)nblocks, st); break;
        case 5: e = llr_launch_t<5>(a, (int)nblocks, st); break;
        case 6: e = llr_launch_t<6>(a, (int)nblocks, st); break;
        case 7: e = llr_launch_t<7>(a, (int)nblocks, st); break;
        case 8: e = llr_launch_t<8>(a, (int)nblocks, st); break;
        default: break;
    }
    if (e != cudaSuccess) return cuda_status(e, "llr_prox_kernel");
    ++g_launches;
    if (g_profiler) g_profiler->mark("llr_prox_kernel");
    return PP_OK;
}

}  // namespace pp
