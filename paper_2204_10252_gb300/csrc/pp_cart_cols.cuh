// Column-resident form of the fused 2-D Cartesian normal operator and of chains of
// it (the gradient and the Horner recursion of Listing "pcode"), single or
// batched.
//
// A mask constant along the readout leaves the image columns independent of one
// another: N_hat, and with it p(N_hat), maps every column to itself.  A CTA owns W
// (1, 2 or 4) columns and applies the operator J times without leaving the SM:
//   in_0 = x, out_j = sc_j sum_c conj(S_c) F^H (mask_fo . F (S_c in_j)) + al_j op_j,
//   in_{j+1} = out_j,
// so a preconditioned gradient of degree d is one launch instead of d + 1, and the
// maps are read once for all of them when they fit shared memory.
//
// Layout: 8 coils x W columns lie in 8 W adjacent lanes (coil slow), thread r of a
// lane is m2 in the phases 1 and 3 and k1 in phase 2 (pp_fft4.cuh's decomposition
// n = N1 N2, N1 <= N2, inverse mirrored).  Coils are taken in groups of 8, the sum
// over groups in registers and over the 8 lanes by a shuffle reduce-scatter, so
// there is no cross-CTA reduction.  A thread reads only the map elements that it
// copied itself (cp.async, one group ahead): no barrier covers them.  Two
// barriers a group and one an application.
//
// What bounds it: latency of the chain of phases for one small slice, shared
// memory (seven 8-byte accesses per element and coil) when the chip is full.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "pp_batch.h"
#include "pp_fftgen.cuh"

namespace pp {

template <int N1, int N2> struct CartCols {
    static constexpr int n = N1 * N2, P = N2 | 1;
    static constexpr int NP = (N1 + 7) / 8 * 8, RPL = NP / 8;   // rows a lane after the reduction
    // float2 elements of shared memory for W columns and NB map buffers
    static size_t elems(int W, int NB) {
        return (size_t)n + n / 2 + 2 * (size_t)n * W + (size_t)N1 * P * 8 * W + (size_t)NB * n * 8 * W;
    }
};

// *p of the same shared variable in CTA `rank` of the cluster
__device__ __forceinline__ float2 cluster_load(const float2* p, int rank) {
    unsigned remote;
    float2 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n"
                 : "=r"(remote) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(remote) : "memory");
    return v;
}

__device__ __forceinline__ void cpa8(void* smem, const void* gmem, bool valid) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(sa), "l"(gmem),
                 "r"(valid ? 8 : 0)
                 : "memory");
}

// Four CTAs of 128 threads an SM (128 registers a thread), fewer larger ones.
__host__ __device__ constexpr int cart_min_ctas(int threads) { return threads < 512 ? 512 / threads : 1; }

template <int N1, int N2, int W>
__global__ void __launch_bounds__(8 * W * N2, cart_min_ctas(8 * W * N2))
cart_cols_kernel(const SliceDesc one, const SliceDesc* __restrict__ descs,
                 const int2* __restrict__ items, int NB, int follows,
                 const float2* __restrict__ x, const CartChain ch) {
    using K = CartCols<N1, N2>;
    constexpr int n = K::n, P = K::P, NP = K::NP;
    extern __shared__ float2 sm[];
    float2* tws = sm;
    float* pm = reinterpret_cast<float*>(sm + n);
    float2* xs = sm + n + n / 2;
    float2* vs = xs + n * W;
    float2* Y = vs + n * W;
    float2* Sb = Y + N1 * P * 8 * W;
    const int2 item = items ? items[blockIdx.x] : make_int2(0, blockIdx.x * W);
    const SliceDesc D = items ? descs[item.x] : one;
    constexpr int EL = 8 * W;
    const int el = threadIdx.x % EL, r = threadIdx.x / EL;
    const int c7 = el / W, w = el - c7 * W;
    const int nx = D.nx, col = item.y + w;
    const bool colok = col < nx;
    const int G = (D.C + 7) / 8;
    const int64_t cs = (int64_t)n * nx;
    // copy of group g's map elements of this thread into buffer b
    auto stage = [&](int g, int b) {
        const int c = 8 * g + c7;
        const bool ok = c < D.C && colok;
        const float2* s = D.sens + (ok ? c * cs + (int64_t)r * nx + col : 0);
        float2* d = Sb + ((size_t)b * n + r) * EL + el;
#pragma unroll
        for (int m1 = 0; m1 < N1; ++m1) cpa8(d + N2 * m1 * EL, s + (ok ? (int64_t)N2 * m1 * nx : 0), ok);
    };
    // plan constants first: they may be copied while the previous kernel runs
    const bool resident = NB >= G;
    for (int g = 0; g < (resident ? G : 1); ++g) stage(g, g);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        tws[i] = D.twb[i];
        pm[i] = D.mask_fo[i];
    }
    // A launch that runs beside its predecessor starts after that one's waits; it
    // waits for it at the end, so that its completion stands for both.
    if (!follows) pdl_wait();
    pdl_trigger();
    const float2* xi = x + D.img_off;
    for (int e = threadIdx.x; e < n * W; e += blockDim.x) {
        const int row = e / W, cw = item.y + e % W;
        const float2 v = cw < nx ? xi[(int64_t)row * nx + cw] : make_float2(0.f, 0.f);
        xs[e] = v;
        if (ch.v_first) vs[e] = v;
    }
    __syncthreads();
    const int warp0 = threadIdx.x & ~31;
    const unsigned lanes = blockDim.x - warp0 >= 32 ? 0xffffffffu : (1u << (blockDim.x - warp0)) - 1u;
    const int steps = ch.J * G;
    int step = 0;
    for (int j = 0; j < ch.J; ++j) {
        float2 acc[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) acc[i] = make_float2(0.f, 0.f);
        for (int g = 0; g < G; ++g, ++step) {
            const int b = resident ? g : (step & 1);
            if (!resident) {
                // the other buffer was read by this thread's previous phase 3 only
                if (step + 1 < steps) stage((g + 1) % G, b ^ 1);
                asm volatile("cp.async.commit_group;\n" ::: "memory");
                asm volatile("cp.async.wait_group 1;\n" ::: "memory");
            } else if (step == 0) {
                asm volatile("cp.async.wait_group 0;\n" ::: "memory");
            }
            const float2* St = Sb + ((size_t)b * n + r) * EL + el;
            {
                float2 v[N1];
#pragma unroll
                for (int m1 = 0; m1 < N1; ++m1) v[m1] = cmul(St[N2 * m1 * EL], xs[(N2 * m1 + r) * W + w]);
                fft4_phase1_exact<N1, N2, false>(v, r, tws);
#pragma unroll
                for (int k1 = 0; k1 < N1; ++k1) Y[(k1 * P + r) * EL + el] = v[k1];
            }
            __syncthreads();
            if (r < N1) {
                float2 u[N2];
#pragma unroll
                for (int m2 = 0; m2 < N2; ++m2) u[m2] = Y[(r * P + m2) * EL + el];
                fft4_phase2<N1, N2, false>(u, tws);
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) u[k2] = cscale(u[k2], pm[r + N1 * k2]);
                RegFft<N2, true>::run(u, tws, N1);
#pragma unroll
                for (int m2 = 0; m2 < N2; ++m2) {
                    float2 t = tws[m2 * r];
                    t.y = -t.y;
                    Y[(r * P + m2) * EL + el] = m2 ? cmul(u[m2], t) : u[m2];
                }
            }
            __syncthreads();
            {
                float2 v[N1];
#pragma unroll
                for (int k1 = 0; k1 < N1; ++k1) v[k1] = Y[(k1 * P + r) * EL + el];
                RegFft<N1, true>::run(v, tws, N2);
#pragma unroll
                for (int m1 = 0; m1 < N1; ++m1) acc[m1] = cadd(acc[m1], cmulc(St[N2 * m1 * EL], v[m1]));
            }
            // the next phase 1 writes the elements of Y that this thread just read
        }
        // sum over the 8 coil lanes: lane c7 keeps rows m1 = first .. first + RPL - 1
        int first = 0;
#pragma unroll
        for (int h = NP / 2, bit = 4; bit >= 1; h >>= 1, bit >>= 1) {
            const bool up = (c7 & bit) != 0;
            if (up) first += h;
#pragma unroll
            for (int i = 0; i < h; ++i) {
                const float2 send = up ? acc[i] : acc[i + h];
                const float2 keep = up ? acc[i + h] : acc[i];
                acc[i] = cadd(keep, make_float2(__shfl_xor_sync(lanes, send.x, bit * W),
                                                __shfl_xor_sync(lanes, send.y, bit * W)));
            }
        }
        const bool ext = j == 0 && !ch.v_first;
        const float sc = ch.sc[j] * D.invL, al = ch.al[j];
#pragma unroll
        for (int i = 0; i < K::RPL; ++i) {
            const int m1 = first + i, row = N2 * m1 + r;
            if (m1 >= N1) continue;
            const int64_t o = D.img_off + (int64_t)row * nx + col;
            float2 v = cscale(acc[i], sc);
            if (ext) {
                if (ch.ext && colok) v = cadd(v, cscale(ch.ext[o], al));
            } else if (al != 0.f) {
                v = cadd(v, cscale(vs[row * W + w], al));
            }
            xs[row * W + w] = v;
            if (ext) vs[row * W + w] = v;
            if (!colok) continue;
            if (j == 0 && ch.first_out) ch.first_out[o] = v;
            if (ch.all_out) ch.all_out[j * ch.all_stride + o] = v;
            if (j == ch.J - 1 && ch.out) ch.out[o] = v;
        }
        __syncthreads();
    }
    if (follows) pdl_wait();
}

// ---------------------------------------------------------------------------
// The same chain on 8 columns per CTA, for launches that fill the chip: lanes over
// columns, so that a map row is a 64-byte run, the coils one after another in Q
// slots (Q > 1 where the columns alone are too few warps).  A thread keeps its
// N1 rows of the current image in registers through all phases and all
// applications; the maps stream through two buffers a slot, each element copied
// by the thread that reads it.  v_j of the Horner recursion is re-read from
// memory.  Bound by shared memory: 19 wavefronts per warp and element against 28
// to 36 of the column-resident form, whose scattered map copies take 8 to 16.
// ---------------------------------------------------------------------------
template <int N1, int N2> struct CartStream {
    static constexpr int n = N1 * N2, P = N2 | 1;
    static constexpr int slot = N1 * P * 8 + 2 * n * 8;   // Y and two map buffers
    static constexpr size_t smem(int Q) { return sizeof(float2) * ((size_t)n + n / 2 + (size_t)Q * slot); }
};

__host__ __device__ constexpr int stream_min_ctas(int threads) { return threads < 512 ? 512 / threads : 1; }

// Barrier of one slot's threads (whole warps), so that the slots run out of step
// and one's transforms cover another's shared-memory phases.
template <int Q, int TS> __device__ __forceinline__ void slot_sync(int q) {
    if constexpr (Q == 1 || TS % 32 != 0) __syncthreads();
    else asm volatile("barrier.cta.sync %0, %1;\n" ::"r"(q + 1), "n"(TS) : "memory");
}

// SPLIT: a cluster of R CTAs (2 or 4) owns the columns and splits the coils.  After
// each application every CTA adds the R partial sums in rank order, each slot a share of
// the rows, so that all of them hold the same next image; after the last one each rank
// adds its own share.  (A form of its own: the
// exchange costs the unsplit one registers, 16 x 16 and longer spill.  It runs at one
// CTA an SM, so small CTAs may take more of them.)
template <int N1, int N2, int Q, bool SPLIT>
__global__ void __launch_bounds__(8 * N2 * Q, SPLIT ? 1 : stream_min_ctas(8 * N2 * Q))
cart_stream_kernel(const SliceDesc one, const SliceDesc* __restrict__ descs,
                   const int2* __restrict__ items, int follows, int R, const float2* x, const CartChain ch) {
    using K = CartStream<N1, N2>;
    constexpr int n = K::n, P = K::P, TS = 8 * N2;
    extern __shared__ float2 sm[];
    float2* tws = sm;
    float* pm = reinterpret_cast<float*>(sm + n);
    const int q = Q > 1 ? threadIdx.x / TS : 0, t = threadIdx.x - q * TS;
    const int lane = t & 7, r = t >> 3;
    float2* Y = sm + n + n / 2 + q * K::slot;
    float2* Sb = Y + N1 * P * 8 + r * 8 + lane;
    const int rank = SPLIT ? blockIdx.x % R : 0, group = SPLIT ? blockIdx.x / R : blockIdx.x;
    const int2 item = items ? items[group] : make_int2(0, group * 8);
    const SliceDesc D = items ? descs[item.x] : one;
    const int nx = D.nx, col = item.y + lane;
    const bool colok = col < nx;
    const int64_t cs = (int64_t)n * nx;
    const float2* Sg = D.sens + (int64_t)r * nx + (colok ? col : 0);
    // this CTA's coils; a CTA without any takes one step of zeros
    const int c0 = SPLIT ? D.C * rank / R : 0, c1 = SPLIT ? D.C * (rank + 1) / R : D.C;
    const int steps = SPLIT ? max(1, (c1 - c0 + Q - 1) / Q) : (D.C + Q - 1) / Q;
    auto stage = [&](int step, int b) {
        const int c = c0 + step * Q + q;
        const bool ok = c < c1 && colok;
        const float2* s = ok ? Sg + c * cs : Sg;
#pragma unroll
        for (int m1 = 0; m1 < N1; ++m1) cpa8(Sb + (b * n + N2 * m1) * 8, s + N2 * m1 * nx, ok);
    };
    stage(0, 0);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        tws[i] = D.twb[i];
        pm[i] = D.mask_fo[i];
    }
    if (!follows) pdl_wait();   // see cart_cols_kernel
    pdl_trigger();
    const int64_t o0 = D.img_off + (int64_t)r * nx + col;   // this thread's first row
    float2 xr[N1];
#pragma unroll
    for (int m1 = 0; m1 < N1; ++m1) xr[m1] = colok ? x[o0 + N2 * m1 * nx] : make_float2(0.f, 0.f);
    __syncthreads();
    const float2* v = ch.v_first ? x : ch.first_out;
    int buf = 0;
    for (int j = 0; j < ch.J; ++j) {
        float2 acc[N1];
#pragma unroll
        for (int i = 0; i < N1; ++i) acc[i] = make_float2(0.f, 0.f);
        for (int step = 0; step < steps; ++step, buf ^= 1) {
            // the other buffer was read by this thread's previous phase 3 only
            if (step + 1 < steps) stage(step + 1, buf ^ 1);
            else if (j + 1 < ch.J) stage(0, buf ^ 1);
            asm volatile("cp.async.commit_group;\n" ::: "memory");
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
            const float2* St = Sb + buf * n * 8;
            {
                float2 w[N1];
#pragma unroll
                for (int m1 = 0; m1 < N1; ++m1) w[m1] = cmul(St[N2 * m1 * 8], xr[m1]);
                fft4_phase1_exact<N1, N2, false>(w, r, tws);
#pragma unroll
                for (int k1 = 0; k1 < N1; ++k1) Y[(k1 * P + r) * 8 + lane] = w[k1];
            }
            slot_sync<Q, TS>(q);
            if (r < N1) {
                float2 u[N2];
#pragma unroll
                for (int m2 = 0; m2 < N2; ++m2) u[m2] = Y[(r * P + m2) * 8 + lane];
                RegFft<N2, false>::run(u, tws, N1);
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) u[k2] = cscale(u[k2], pm[r + N1 * k2]);
                RegFft<N2, true>::run(u, tws, N1);
#pragma unroll
                for (int m2 = 0; m2 < N2; ++m2) {
                    float2 tw = tws[m2 * r];
                    tw.y = -tw.y;
                    Y[(r * P + m2) * 8 + lane] = m2 ? cmul(u[m2], tw) : u[m2];
                }
            }
            slot_sync<Q, TS>(q);
            {
                float2 w[N1];
#pragma unroll
                for (int k1 = 0; k1 < N1; ++k1) w[k1] = Y[(k1 * P + r) * 8 + lane];
                RegFft<N1, true>::run(w, tws, N2);
#pragma unroll
                for (int m1 = 0; m1 < N1; ++m1) acc[m1] = cadd(acc[m1], cmulc(St[N2 * m1 * 8], w[m1]));
            }
            // the next phase 1 writes the elements of Y that this thread just read
        }
        if constexpr (SPLIT) {
            float2* const Y0 = sm + n + n / 2 + r * 8 + lane;
            __syncthreads();   // Y is free
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) Y[(N2 * m1 + r) * 8 + lane] = acc[m1];
            constexpr int RQ = (N1 + Q - 1) / Q;   // rows q, q + Q, .. belong to slot q here
            float2* const Yr = Y0 + N2 * q * 8;
            if constexpr (Q > 1) {
                __syncthreads();
#pragma unroll
                for (int i = 0; i < RQ; ++i) {
                    if (q + Q * i >= N1) break;
                    float2 a = Yr[N2 * Q * i * 8];
#pragma unroll
                    for (int p = 1; p < Q; ++p) a = cadd(a, Yr[p * K::slot + N2 * Q * i * 8]);
                    Yr[N2 * Q * i * 8] = a;
                }
            }
            cluster_arrive_release();
            cluster_wait_acquire();
            if (j == ch.J - 1) {
                // nothing follows: each rank adds and writes a share of the rows
                const float sc = ch.sc[j] * D.invL, al = ch.al[j];
                const float2* op = j == 0 && !ch.v_first ? ch.ext : (al != 0.f ? v : nullptr);
                float2* out0 = j == 0 ? ch.first_out : nullptr;
                float2* out1 = ch.all_out ? ch.all_out + j * ch.all_stride : nullptr;
                for (int i = rank; i < RQ && q + Q * i < N1; i += R) {
                    float2 t[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) t[k] = k < R ? cluster_load(Yr + N2 * Q * i * 8, k) : make_float2(0.f, 0.f);
                    float2 s = cadd(t[0], t[1]);
                    if (R > 2) s = cadd(cadd(s, t[2]), t[3]);
                    if (!colok) continue;
                    const int64_t o = o0 + N2 * (q + Q * i) * nx;
                    s = cscale(s, sc);
                    if (op) s = cadd(s, cscale(op[o], al));
                    if (out0) out0[o] = s;
                    if (out1) out1[o] = s;
                    if (ch.out) ch.out[o] = s;
                }
                cluster_arrive_release();
                cluster_wait_acquire();
                break;
            }
            float2 a[RQ];
            for (int k = 0; k < R; ++k) {
                float2 t[RQ];
#pragma unroll
                for (int i = 0; i < RQ; ++i)
                    t[i] = q + Q * i < N1 ? cluster_load(Yr + N2 * Q * i * 8, k) : make_float2(0.f, 0.f);
#pragma unroll
                for (int i = 0; i < RQ; ++i) a[i] = k ? cadd(a[i], t[i]) : t[i];
            }
            if constexpr (Q > 1) {
                // through slot 1, whose part is not read from outside
#pragma unroll
                for (int i = 0; i < RQ; ++i)
                    if (q + Q * i < N1) Yr[K::slot + N2 * Q * i * 8] = a[i];
                __syncthreads();
#pragma unroll
                for (int m1 = 0; m1 < N1; ++m1) acc[m1] = Y0[K::slot + N2 * m1 * 8];
            } else {
#pragma unroll
                for (int m1 = 0; m1 < N1; ++m1) acc[m1] = a[m1];
            }
            cluster_arrive_release();   // Y may be written again once all have waited for this
        } else if constexpr (Q > 1) {
            // the slots' sums meet in Y, in slot order
            __syncthreads();
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) Y[(N2 * m1 + r) * 8 + lane] = acc[m1];
            __syncthreads();
            const float2* Y0 = sm + n + n / 2 + r * 8 + lane;
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) {
                float2 a = Y0[N2 * m1 * 8];
#pragma unroll
                for (int p = 1; p < Q; ++p) a = cadd(a, Y0[p * K::slot + N2 * m1 * 8]);
                acc[m1] = a;
            }
            __syncthreads();
        }
        const bool ext = j == 0 && !ch.v_first;
        const float sc = ch.sc[j] * D.invL, al = ch.al[j];
        const float2* op = ext ? ch.ext : (al != 0.f ? v : nullptr);
#pragma unroll
        for (int m1 = 0; m1 < N1; ++m1) xr[m1] = cscale(acc[m1], sc);
        if (op && colok) {
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) xr[m1] = cadd(xr[m1], cscale(op[o0 + N2 * m1 * nx], al));
        }
        if (q == 0 && rank == 0 && colok) {
            float2* out0 = j == 0 ? ch.first_out : nullptr;
            if (out0) {
#pragma unroll
                for (int m1 = 0; m1 < N1; ++m1) out0[o0 + N2 * m1 * nx] = xr[m1];
            }
            float2* out1 = ch.all_out ? ch.all_out + j * ch.all_stride : nullptr;
            if (out1) {
#pragma unroll
                for (int m1 = 0; m1 < N1; ++m1) out1[o0 + N2 * m1 * nx] = xr[m1];
            }
            float2* out2 = j == ch.J - 1 ? ch.out : nullptr;
            if (out2) {
#pragma unroll
                for (int m1 = 0; m1 < N1; ++m1) out2[o0 + N2 * m1 * nx] = xr[m1];
            }
        }
        if constexpr (SPLIT) cluster_wait_acquire();
    }
    if (follows) pdl_wait();
}

template <int N1, int N2>
cudaError_t cart_cols_launch(const CartLaunch& L, const float2* x, const CartChain& ch, cudaStream_t st) {
    using K = CartCols<N1, N2>;
    if (L.W == 8) {
        using KS = CartStream<N1, N2>;
        const int grid = (L.items ? L.nitems : (L.one.nx + 7) / 8) * L.split;
        auto go = [&](auto kernel, int Q, cudaError_t allowed) {
            if (allowed != cudaSuccess) return allowed;
            return launch_ex(kernel, dim3(grid), dim3(8 * N2 * Q), KS::smem(Q), st, L.pdl, L.split > 1 ? L.split : 0,
                             L.one, L.descs, L.items, (int)L.follows, L.split, x, ch);
        };
#define PP_GO(Q, SPLIT)                                        \
    go(cart_stream_kernel<N1, N2, Q, SPLIT>, Q, allow_smem<cart_stream_kernel<N1, N2, Q, SPLIT>, kCartSmem>())
        if constexpr (KS::smem(4) <= (size_t)kCartSmem && 32 * N2 <= 512)
            if (L.slots == 4) return L.split > 1 ? PP_GO(4, true) : PP_GO(4, false);
        if constexpr (KS::smem(2) <= (size_t)kCartSmem)
            if (L.slots >= 2) return L.split > 1 ? PP_GO(2, true) : PP_GO(2, false);
        return L.split > 1 ? PP_GO(1, true) : PP_GO(1, false);
#undef PP_GO
    }
    const int groups = (L.max_coils + 7) / 8, NB = L.resident || groups < 2 ? groups : 2;
    const size_t smem = sizeof(float2) * K::elems(L.W, NB);
    const int grid = L.items ? L.nitems : (L.one.nx + L.W - 1) / L.W;
    if (smem > kCartSmem || !cart_width_ok(K::n, L.W)) return cudaErrorInvalidValue;
    auto go = [&](auto kernel, cudaError_t allowed) {
        if (allowed != cudaSuccess) return allowed;
        return launch_ex(kernel, dim3(grid), dim3(8 * L.W * N2), smem, st, L.pdl, 0, L.one, L.descs,
                         L.items, NB, (int)L.follows, x, ch);
    };
    if (L.W == 1) return go(cart_cols_kernel<N1, N2, 1>, allow_smem<cart_cols_kernel<N1, N2, 1>, kCartSmem>());
    if (L.W == 2) return go(cart_cols_kernel<N1, N2, 2>, allow_smem<cart_cols_kernel<N1, N2, 2>, kCartSmem>());
    if constexpr (cart_width_ok(K::n, 4))
        return go(cart_cols_kernel<N1, N2, 4>, allow_smem<cart_cols_kernel<N1, N2, 4>, kCartSmem>());
    return cudaErrorInvalidValue;
}

}  // namespace pp
