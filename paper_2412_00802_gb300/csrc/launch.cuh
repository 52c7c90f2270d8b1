// Programmatic dependent launches: a short chain of kernels on one stream
// whose blocks may start (shared-memory and tensor-memory set-up, barrier
// initialisation) while the kernel before them still runs.  Six launches of a
// training step and three of a forward pass, each 4 to 14 us, had paid their
// launch latency in full: a step of 4,096 rows 70 -> 61 us, one of 1,000 rows
// 61 -> 47 us, a forward pass of 1,999 rows 22.5 -> 15.7 us.
#pragma once

#include <cuda_runtime.h>

namespace hedl {

// Lets the stream's next kernel start once every block of this one has got
// here (or left); it still waits in pdl_wait for this one's results.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Returns when the stream's kernel before this one has completed and its
// writes are visible.  Nothing that it reads or writes may be touched earlier.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launches a kernel that calls pdl_wait before it touches global memory.
template <class... P, class... A>
cudaError_t launch_pdl(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &attr;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, P(args)...);
}

// Lets a kernel launch with `smem` bytes of dynamic shared memory, beyond the
// 48 KB that need no leave.  The leave belongs to the kernel on the current
// device and ends with its context: it may be remembered with what lives there
// (a handle), not for the process, and a failure not at all.
template <class... P>
cudaError_t allow_smem(void (*kernel)(P...), size_t smem) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

}  // namespace hedl
