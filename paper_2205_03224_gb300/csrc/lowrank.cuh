// The low-rank term of the previous level (Alg. 2 step 7), added by the kernels
// that first read each tail row: conversions of W's entries and one row of W u.
#pragma once

#include "kernels.cuh"

namespace gemslr {
namespace {

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename VT, typename WT> __device__ __forceinline__ VT wval(WT w) { return (VT)to_f(w); }
template <> __device__ __forceinline__ double wval<double, double>(double w) { return w; }
template <> __device__ __forceinline__ zc wval<zc, zc>(zc w) { return w; }
// an entry of W^H (the correction is W H W^H; for real data W^T)
template <typename VT, typename WT> __device__ __forceinline__ VT wval_h(WT w) { return wval<VT, WT>(w); }
template <> __device__ __forceinline__ zc wval_h<zc, zc>(zc w) { return conj(w); }

// Row g's share of the previous level's W u (see PendingLowRank): sixteen
// columns at a time with all their loads issued first (columns past k load
// the last column again and are not added).  u is read through L2:
// the coupling kernel that reads it also rewrites it in its finisher.
template <typename VT, typename WT>
__device__ __forceinline__ VT pending_row(const PendingLowRank<VT, WT> &pl, int64_t g) {
    const WT *w = pl.W + (g - pl.row0);
    VT a0 = 0, a1 = 0;
    for (int c0 = 0; c0 < pl.k; c0 += 16) {
        WT wv[16];
        VT uv[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const int c = min(c0 + q, pl.k - 1);
            wv[q] = w[(int64_t)c * pl.ld];
            uv[q] = c0 + q < pl.k ? ldcg(pl.u + c) : (VT)0;
        }
        const int left = std::is_same_v<VT, zc> ? 16 : pl.k - c0;   // complex: contracted as always
        if (left >= 16) {
#pragma unroll
            for (int q = 0; q < 16; q += 2) {
                a0 += wval<VT, WT>(wv[q]) * uv[q];
                a1 += wval<VT, WT>(wv[q + 1]) * uv[q + 1];
            }
        } else {
#pragma unroll
            for (int q = 0; q < 16; q += 2) {
                if (q < left) a0 += wval<VT, WT>(wv[q]) * uv[q];
                if (q + 1 < left) a1 += wval<VT, WT>(wv[q + 1]) * uv[q + 1];
            }
        }
    }
    return a0 + a1;
}

}  // namespace
}  // namespace gemslr
