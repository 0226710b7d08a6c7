// pdl.cuh -- programmatic dependent launch.  Kernels of a chain that start with pdl_wait()
// and are launched with launch_pdl need no drained SM between them: 1 to 2 us a launch.
//
// Such a kernel is resident while the one before it still writes, so what that one writes is
// read by plain loads only: __ldg and const __restrict__ (loads for data that is read-only for
// the kernel's whole life, which the compiler may also move above pdl_wait) are for tables that
// are complete two launches earlier -- the plan's tables, the caller's inputs, K-hat and the
// preconditioner's diagonal.
#pragma once
#include <cuda_runtime.h>

namespace firm {

// Programmatic dependent launch: the next kernel of the stream may start its blocks now
// (it waits in pdl_wait until this one has finished and its writes are visible).
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launches of more blocks than this (a few waves) are ordinary ones: beside work of that
// size the gap between two kernels is nothing, and the next kernel's early blocks take
// slots from it (512^3 transforms 0.59 -> 0.52 ms, both channels at N = 128, 50,000 images
// 32.1 -> 31.5 ms as ordinary launches; the sums of 200 images at N = 32 0.24 -> 0.18 ms as
// dependent ones).
constexpr long long kPdlBlocks = 2048;

template <class... KArgs, class... Args>
static cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, int block, size_t smem, cudaStream_t s,
                              Args... args) {
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3((unsigned)block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = at;
    c.numAttrs = (long long)grid.x * grid.y * grid.z <= kPdlBlocks ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, KArgs(args)...);
}

}  // namespace firm
