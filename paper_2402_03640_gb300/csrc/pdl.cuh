// Programmatic dependent launch: a kernel launched with launch_pdl may start
// while the kernel before it in the stream still runs, once every block of
// that one has called grid_dep_launch (or ended); grid_dep_wait returns when
// it has completed and its writes are visible.  Every block waits before its
// first access to anything an earlier kernel writes or reads, so the order of
// effects is that of plain launches; what overlaps is the launch itself and
// the loads of the instance's lists, which no kernel writes.  What an earlier
// kernel or the caller's may have written is read with ld_ordered, or another
// volatile load: none moves above the wait, and none goes through the
// read-only cache, which holds only for memory that nothing writes during the
// kernel's life.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace msat {

__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ float ld_ordered(const float *p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ int8_t ld_ordered(const int8_t *p) {
    int v;
    asm volatile("ld.global.s8 %0, [%1];" : "=r"(v) : "l"(p));
    return (int8_t)v;
}

template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = grid;
    lc.blockDim = block;
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, kernel, static_cast<P>(args)...);
}

}  // namespace msat
