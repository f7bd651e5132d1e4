// chain.cuh -- kernels of one stream launched as a chain (programmatic
// dependent launch).
//
// A step is a short chain of dependent kernels, and between two ordinary
// launches of a stream the GPU spends about 2 us (measured: the period of a
// small kernel launched back to back is a multiple of 2.05 us: 4.1, 6.15,
// 8.2 ...).  A kernel launched with launch_chained may start while its
// predecessor still runs: its blocks take the slots the predecessor leaves,
// compute what needs no memory and then stand in wait_for_previous() until
// every earlier kernel of the stream has finished and its writes are visible.
// 32^3 steps 6.15 -> 3.2 us, 64^3 10.3 -> 7.7 us, 128^3 at kT = 0 50.6 -> 47.9
// us, 256^3 383.5 -> 381.7 us.
//
// Rules for a kernel launched this way:
//  - every block calls wait_for_previous() before it reads or writes any
//    global memory (kernel parameters are free);
//  - global loads are plain loads ordered after it: no __ldg and no const
//    __restrict__ pointers, whose loads the compiler may move up.  The ld_*
//    functions below are volatile, which keeps them behind the wait and in
//    order among themselves, but not against ordinary stores: a kernel that
//    stores to what it has read this way, with no branch on the loaded value
//    in between, puts loads_done() before the store;
//  - it lets its own successor start only after its wait, so at most two
//    kernels of a stream are in flight and the buffers a step reads are never
//    written by an earlier kernel still running.
#pragma once

#include <cuda_runtime.h>

namespace lbi {

__device__ __forceinline__ void wait_for_previous()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Every load above stands before every store below (for the compiler).
__device__ __forceinline__ void loads_done() { asm volatile("" ::: "memory"); }

__device__ __forceinline__ float ld_f32(const float *p)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float2 ld_f32x2(const float *p)  // 8-byte aligned
{
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned short ld_u16(const void *p)
{
    unsigned short v;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned int ld_u32(const void *p)  // 4-byte aligned
{
    unsigned int v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

template <typename... K, typename... A>
cudaError_t launch_chained(void (*kernel)(K...), dim3 grid, dim3 block, cudaStream_t stream, const A &...args)
{
    cudaLaunchConfig_t lc = {};
    lc.gridDim = grid;
    lc.blockDim = block;
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&lc, kernel, static_cast<K>(args)...);
    if (e != cudaSuccess) (void)cudaGetLastError();  // reported here, not again by the next call that looks
    return e;
}

}  // namespace lbi
