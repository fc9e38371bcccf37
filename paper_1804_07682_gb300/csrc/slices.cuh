// slices.cuh -- the sum over the slices of a group, shared by the slice
// reductions of the survival and the any-channel chain.
#pragma once

#include <mutex>

#include "common.cuh"

namespace gna {

// The block's (point, group), blockIdx.x: its S slices of NV values in part,
// summed by W warps.  Warp w sums slices w, w + W, ... in order for every value
// (lane l: bin 32 g + l; the loads of a slice for all values are in flight
// together); the warps' sums are then added in warp order through shared
// memory, one value per warp.  The fixed order makes the result independent
// of timing.  NVM bounds the value count so that the per-lane arrays stay in
// registers.  Returns the sums in shared memory, [NV][32], readable by all warps.
template <int NVM, int W>
__device__ __forceinline__ const float2* sum_slices(const float2* __restrict__ part, int S, int NV, int w, int lane) {
    extern __shared__ float2 red[];  // [W][NV][32], then [NV][32]
    float2* fin = red + W * NV * 32;
    // the next evaluation's first kernel may be placed now; it waits for this
    // kernel to complete before it touches anything
    asm volatile("griddepcontrol.launch_dependents;");
    float2 acc[NVM];
#pragma unroll
    for (int v = 0; v < NVM; v++) acc[v] = make_float2(0.f, 0.f);
    // launched as a programmatic dependent of the node kernel: the blocks may
    // be resident before it ends; wait (in hardware) until it has completed
    // and its writes are visible
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const float2* base = part + (int64_t)blockIdx.x * S * NV * 32 + lane;
    const int64_t stride = (int64_t)NV * 32;
    for (int sl = w; sl < S; sl += W) {
        const float2* src = base + sl * stride;
        float2 t[NVM];
#pragma unroll
        for (int v = 0; v < NVM; v++) t[v] = (v < NV) ? __ldg(src + v * 32) : make_float2(0.f, 0.f);
#pragma unroll
        for (int v = 0; v < NVM; v++)
            if (v < NV) acc[v] = ff_add(acc[v], t[v]);
    }
#pragma unroll
    for (int v = 0; v < NVM; v++)
        if (v < NV) red[(w * NV + v) * 32 + lane] = acc[v];
    __syncthreads();
    const int used = min(W, S);  // warps that had a slice
    for (int v = w; v < NV; v += W) {
        float2 sum = red[v * 32 + lane];
        for (int k = 1; k < used; k++) sum = ff_add(sum, red[(k * NV + v) * 32 + lane]);
        fin[v * 32 + lane] = sum;
    }
    __syncthreads();
    return fin;
}

// More than the default 48 KB of dynamic shared memory: opt in once per device and kernel.
template <auto K>
cudaError_t allow_smem(size_t bytes) {
    static std::once_flag once[64];
    static cudaError_t attr[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::call_once(once[dev], [&] {
        attr[dev] = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    });
    return attr[dev];
}

// Launch as a programmatic dependent of the kernel before.
template <typename... Args>
cudaError_t launch_blocks(void (*k)(Args...), int64_t blocks, int threads, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

}  // namespace gna
