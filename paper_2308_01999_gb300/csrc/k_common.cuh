// k_common.cuh -- device helpers shared by the gate kernels.
#pragma once

#include "sv_internal.h"

namespace svk {

template <typename R> struct CT;
template <> struct CT<float> { using T = float2; };
template <> struct CT<double> { using T = double2; };

__device__ __forceinline__ float fmac(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmac(double a, double b, double c) { return __fma_rn(a, b, c); }

// acc += m * v (complex)
template <typename C>
__device__ __forceinline__ void cmad(C &acc, const C &m, const C &v) {
    acc.x = fmac(m.x, v.x, acc.x);
    acc.x = fmac(-m.y, v.y, acc.x);
    acc.y = fmac(m.x, v.y, acc.y);
    acc.y = fmac(m.y, v.x, acc.y);
}

template <typename C>
__device__ __forceinline__ C cmul(const C &a, const C &b) {
    C r;
    r.x = fmac(a.x, b.x, -a.y * b.y);
    r.y = fmac(a.x, b.y, a.y * b.x);
    return r;
}

// Zero bits inserted at G.pos (ascending), then the control bits set.
__device__ __forceinline__ uint64_t insert_zeros(uint64_t g, const GroupGeom &G) {
#pragma unroll 1
    for (int i = 0; i < G.ns; ++i) {
        const uint64_t lo = g & ((1ull << G.pos[i]) - 1ull);
        g = ((g ^ lo) << 1) | lo;
    }
    return g | G.cset;
}

template <int K> struct Offs { uint64_t o[1 << K]; };

}  // namespace svk
