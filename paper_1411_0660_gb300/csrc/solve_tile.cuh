// solve_tile.cuh -- device pieces shared by the level-by-level (factor.cu) and the dataflow
// (solve_df.cu) triangular solves: 16-byte asynchronous copies out of the packed solve factor, the
// product of one backward tile and the final reduction of a backward panel's partial sums.
//
// Backward tile: RBK rows x RBB columns of a solve panel's G = [M; L21 M] (packed column-major,
// every column 16-byte aligned, zero padding rows), times v = [y_panel; -x_below] (RBK x PB).
#pragma once

#include "plan.h"

namespace mbl {

template <class T>
struct Vec16;
template <>
struct Vec16<float> {
    using type = float4;
    static __device__ __forceinline__ float get(const float4 &v, int e) {
        return e == 0 ? v.x : (e == 1 ? v.y : (e == 2 ? v.z : v.w));
    }
    static __device__ __forceinline__ void put(float *d, const float *a) {
        *reinterpret_cast<float4 *>(d) = make_float4(a[0], a[1], a[2], a[3]);
    }
};
template <>
struct Vec16<double> {
    using type = double2;
    static __device__ __forceinline__ double get(const double2 &v, int e) { return e == 0 ? v.x : v.y; }
    static __device__ __forceinline__ void put(double *d, const double *a) {
        *reinterpret_cast<double2 *>(d) = make_double2(a[0], a[1]);
    }
};

// Column stride of a backward tile in shared memory: RBK rows plus a pad that puts the 16-byte
// reads of eight consecutive columns on distinct bank groups (stride / (16 / sizeof(T)) odd).
template <class T>
__host__ __device__ constexpr int bwd_ldg() {
    return sizeof(T) == 4 ? RBK + 4 : RBK + 2;
}

// Right-hand sides a backward tile's product takes at a time (for more than 16 it runs twice over the
// tile), and the row stride of its partial sums: a pad that spreads the 16-byte stores of a warp's lanes
// over the banks (FP64 has no shared memory left for it).
template <class T, int PB>
__host__ __device__ constexpr int bwd_qc() {
    return sizeof(T) == 4 && PB > 8 ? 16 : 8;
}
template <class T, int PB>
__host__ __device__ constexpr int bwd_ldr() {
    return bwd_qc<T, PB>() + (sizeof(T) == 4 ? 4 : 0);
}

// Shared memory of a backward step: the G tile, v, and (where the product runs more than once) the
// cross-warp partial sums, which otherwise reuse the G tile.
template <class T, int PB>
__host__ __device__ constexpr size_t bwd_tile_smem() {
    return sizeof(T) * ((size_t)RBB * bwd_ldg<T>() + (size_t)RBK * PB +
                        (PB == bwd_qc<T, PB>() ? 0 : (size_t)8 * RBB * bwd_ldr<T, PB>()));
}

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const unsigned int sa = (unsigned int)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit_wait() {
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Issue the copies of a backward tile: columns [0, wc) x 16-byte row groups [0, nrv) of G (column
// stride ld; G and ld 16-byte aligned) into Gs (column stride bwd_ldg<T>()).
template <class T>
__device__ __forceinline__ void bwd_tile_issue(T *Gs, const T *G, int64_t ld, int wc, int nrv) {
    constexpr int E = 16 / sizeof(T), LDG = bwd_ldg<T>();
    for (int c = threadIdx.x / 32; c < wc; c += blockDim.x / 32)  // a warp per column: no division per piece
        for (int v = threadIdx.x % 32; v < nrv; v += 32)
            cp_async16(Gs + c * LDG + v * E, G + (int64_t)c * ld + (int64_t)v * E);
}

// dst (256 rows x PB, zero past row `rows` and right-hand side p) from `rows` consecutive rows of p values.
// 256 threads; all of a thread's loads are issued before its first store, in 16-byte pieces where the rows
// have no padding (src is 16-byte aligned then).
template <class T, int PB>
__device__ __forceinline__ void stage_rows(T *dst, const T *src, int rows, int p) {
    constexpr int E = 16 / sizeof(T);
    using V = typename Vec16<T>::type;
    if (p == PB) {
        V v[PB / E];
#pragma unroll
        for (int u = 0; u < PB / E; ++u) {
            const int idx = threadIdx.x + 256 * u;
            v[u] = idx < rows * (PB / E) ? reinterpret_cast<const V *>(src)[idx] : V{};
        }
#pragma unroll
        for (int u = 0; u < PB / E; ++u) reinterpret_cast<V *>(dst)[threadIdx.x + 256 * u] = v[u];
    } else {
#pragma unroll
        for (int u0 = 0; u0 < PB; u0 += 8) {
            T v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int idx = threadIdx.x + 256 * (u0 + u), r = idx / PB, q = idx % PB;
                v[u] = r < rows && q < p ? src[r * p + q] : T(0);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) dst[threadIdx.x + 256 * (u0 + u)] = v[u];
        }
    }
}

// Partial products of a backward tile for right-hand sides [q0, q0 + QC): warp j takes rows
// [32 j, 32 j + 32) below nrows (a whole number of 16-byte row groups; the rows of vs past the
// panel are zero), lane l takes columns l and l + 32.  The eight warps' sums meet in red
// (8 x RBB x bwd_ldr; it may alias Gs, so the call starts with a barrier) and thread t returns the
// outputs o = t + 256 h (column c = o / QC, q = q0 + o % QC: a row's values lie side by side) in
// out[h].  256 threads.
template <class T, int PB>
__device__ __forceinline__ void bwd_tile_product(const T *Gs, const T *vs, T *red, int nrows, int q0,
                                                 T out[RBB * bwd_qc<T, PB>() / 256]) {
    constexpr int E = 16 / sizeof(T), LDG = bwd_ldg<T>(), QC = bwd_qc<T, PB>(), LDR = bwd_ldr<T, PB>();
    using V = typename Vec16<T>::type;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int i0 = wp * 32, i1 = min(i0 + 32, nrows);
    T a0[QC], a1[QC];
#pragma unroll
    for (int q = 0; q < QC; ++q) a0[q] = a1[q] = T(0);
#pragma unroll 2
    for (int i = i0; i < i1; i += E) {
        const V g0 = *reinterpret_cast<const V *>(Gs + lane * LDG + i);
        const V g1 = *reinterpret_cast<const V *>(Gs + (lane + 32) * LDG + i);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const T ga = Vec16<T>::get(g0, e), gb = Vec16<T>::get(g1, e);
            const V *vr = reinterpret_cast<const V *>(vs + (i + e) * PB + q0);
#pragma unroll
            for (int u = 0; u < QC / E; ++u) {
                const V vv = vr[u];
#pragma unroll
                for (int k = 0; k < E; ++k) {
                    const T vk = Vec16<T>::get(vv, k);
                    a0[u * E + k] += ga * vk;
                    a1[u * E + k] += gb * vk;
                }
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < QC; u += E) {
        Vec16<T>::put(red + (wp * RBB + lane) * LDR + u, a0 + u);
        Vec16<T>::put(red + (wp * RBB + lane + 32) * LDR + u, a1 + u);
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < RBB * QC / 256; ++h) {
        const int o = threadIdx.x + 256 * h, c = o / QC, q = o % QC;
        T v = T(0);
#pragma unroll
        for (int j = 0; j < 8; ++j) v += red[(j * RBB + c) * LDR + q];
        out[h] = v;
    }
}

// Last block of a (panel, column chunk): add the nb partial tiles ([c][q], RBB x PB each, stride
// apart) in a fixed order and write the result -- columns c < wc, right-hand sides q < p -- to
// zs[c p + q] and, unless xo is null, xo[c p + q].  comb: scratch of 2 x RBB x PB in shared memory.
// 256 threads.
template <class T, int PB>
__device__ void bwd_finish(const T *src, int64_t stride, int nb, int wc, int p, T *zs, T *xo, T *comb) {
    constexpr int E = 16 / sizeof(T), NV = RBB * PB / E;
    constexpr int NG = NV >= 256 ? 1 : 256 / NV;  // groups of partial tiles summed separately
    using V = typename Vec16<T>::type;
    const int g = NG > 1 ? (int)threadIdx.x / NV : 0;
    const int v0 = NG > 1 ? (int)threadIdx.x % NV : (int)threadIdx.x, vstep = NG > 1 ? NV : 256;
    for (int vi = v0; vi < NV; vi += vstep) {
        T acc[E];
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] = T(0);
#pragma unroll 8
        for (int bb = g; bb < nb; bb += NG) {
            const V v = __ldcg(reinterpret_cast<const V *>(src + (int64_t)bb * stride) + vi);
#pragma unroll
            for (int e = 0; e < E; ++e) acc[e] += Vec16<T>::get(v, e);
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int o = vi * E + e;
            if (NG > 1) {
                comb[g * RBB * PB + o] = acc[e];
            } else {
                const int c = o / PB, q = o % PB;
                if (c < wc && q < p) {
                    zs[c * p + q] = acc[e];
                    if (xo) xo[c * p + q] = acc[e];
                }
            }
        }
    }
    if (NG > 1) {
        __syncthreads();
        for (int o = threadIdx.x; o < RBB * PB; o += blockDim.x) {
            T v = T(0);
            for (int gg = 0; gg < NG; ++gg) v += comb[gg * RBB * PB + o];
            const int c = o / PB, q = o % PB;
            if (c < wc && q < p) {
                zs[c * p + q] = v;
                if (xo) xo[c * p + q] = v;
            }
        }
    }
}

}  // namespace mbl
