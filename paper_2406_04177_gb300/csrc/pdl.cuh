// Programmatic dependent launch (PTX griddepcontrol, sm_90 and later).  A grid launched with
// programmatic stream serialisation may be scheduled while the kernel before it on the stream is
// still running; pdl_wait, before the grid's first global access, holds it until that kernel has
// completed and its writes are visible.  For a grid launched without the attribute it returns at
// once.  pdl_trigger lets the next grid on the stream be scheduled once every block of this one has
// issued it (its blocks then sit in their own pdl_wait).
#pragma once

#include <cuda_runtime.h>

namespace vga {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launch with programmatic stream serialisation (the kernel must call pdl_wait first).
template <typename... KArgs, typename... Args>
void launch_pdl(void (*kernel)(KArgs...), dim3 grid, unsigned threads, cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

}  // namespace vga
