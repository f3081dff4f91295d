// launch.cuh — dependent launches: the kernels of a batch follow one another without the launch latency
// in between (programmatic stream serialization). The setup kernel lets its successor start at once; a
// fused kernel then fills its tables while the setup kernel still runs and waits for it (grid_wait)
// before it touches the workspace. Kernels that do not let their successor start early are followed
// by it as soon as they end. Measured against ordinary launches: one query on 2^16 x 32 B 49.0 -> 45.0
// us (the whole synchronous call), 16 on 2^18 x 64 B 217 -> 210.
#pragma once

#include <cuda_runtime.h>

namespace impir {

template <typename P>
cudaError_t launch_after(void (*kernel)(P), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const P& p) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, p);
}

// Waits until the kernel before this one in the stream has ended and its writes are visible (at once
// where there is nothing to wait for).
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Lets the next kernel start now, up to its grid_wait.
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

}  // namespace impir
