// k_common.cuh -- device helpers shared by the gate kernels.
#pragma once

#include <utility>

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

// Programmatic dependent launch: a gate kernel lets the next one start as soon as
// all its blocks are running, and touches the state only after the one before
// it has finished (and its writes are visible). On small states, where a kernel
// takes about as long as its launch, the launch then overlaps the kernel before
// (300 gates on 16 qubits: 2.8 us per gate, 5.5 launched plainly).
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch a kernel that calls both. Every block has to reach wait_for_previous(),
// or a later kernel could start before an earlier one is done.
template <typename... P, typename... A>
inline cudaError_t launch_dependent(void (*kern)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream,
                                    A &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
    if (e != cudaSuccess) cudaGetLastError();   // reported here, not by the next launch that asks
    return e;
}

template <int K> struct Offs { uint64_t o[1 << K]; };

}  // namespace svk
