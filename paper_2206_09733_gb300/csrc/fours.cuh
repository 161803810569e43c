// Groups of four values in shared memory (Gauss-Legendre and mortar kernels).
#pragma once

#include <cuda_runtime.h>

namespace hs3d {

// Four values a point in shared memory.  FP32: side by side, one 16-byte access and
// packed multiply-adds (these kernels issue more shared-memory and FP32
// instructions than anything else); FP64: four arrays of `S` values, consecutive
// threads on consecutive words.  Either way 4 S values, rounded the same.
// Runs of 4 steps, NS, against single values: 32^3 N = 3 4.20 -> 4.02 ms, 24^3 N = 4 4.01 ->
// 3.71, 20^3 N = 5 4.56 -> 4.11, 16^3 N = 7 6.60 -> 6.08; Euler 32^3 N = 3 1.95 -> 1.82.
template <typename R>
struct Four {
    R x[4];
};
template <int S, typename R>
__device__ __forceinline__ Four<R> ld_four(const R *base, int i)
{
    if constexpr (sizeof(R) == 4) {
        const float4 v = ((const float4 *)base)[i];
        return {v.x, v.y, v.z, v.w};
    } else {
        return {base[i], base[S + i], base[2 * S + i], base[3 * S + i]};
    }
}
template <int S, typename R>
__device__ __forceinline__ void st_four(R *base, int i, R a, R b, R c, R d)
{
    if constexpr (sizeof(R) == 4) {
        ((float4 *)base)[i] = make_float4(a, b, c, d);
    } else {
        base[i] = a;
        base[S + i] = b;
        base[2 * S + i] = c;
        base[3 * S + i] = d;
    }
}
// a += s f
template <typename R>
__device__ __forceinline__ void add_four(Four<R> &a, R s, const Four<R> &f)
{
    if constexpr (sizeof(R) == 4) {
        const float2 s2 = make_float2(s, s);
        const float2 lo = __ffma2_rn(s2, make_float2(f.x[0], f.x[1]), make_float2(a.x[0], a.x[1]));
        const float2 hi = __ffma2_rn(s2, make_float2(f.x[2], f.x[3]), make_float2(a.x[2], a.x[3]));
        a = {lo.x, lo.y, hi.x, hi.y};
    } else {
#pragma unroll
        for (int v = 0; v < 4; ++v) a.x[v] += s * f.x[v];
    }
}

}  // namespace hs3d
