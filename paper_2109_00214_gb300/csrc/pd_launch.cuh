// pd_launch.cuh -- kernels launched while the one before them on the stream ends.
//
// A chain of kernels of some ten microseconds spends a tenth of its time between
// them: the launch, the first loads and the drain of the last wave.  A kernel
// launched by launch() starts as soon as all blocks of the one before have
// started and their SMs have room, and waits on the device, in chained(), for its
// end; what it does before that call overlaps.
//
// Every kernel launched this way calls chained() in every thread, and before it
// reads or writes only what no kernel after the last but one touches: chained()
// lets the next kernel start only once the kernels before this one have ended.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <utility>

namespace pd {

// Waits until the kernel before has ended and its writes are visible, then lets
// the next one start; false never.  The caller returns on false: as the value (a
// grid has blocks) is not known to the compiler, no load, not even one it holds to
// be constant during the kernel, can move above the wait.
__device__ __forceinline__ bool chained() {
    uint32_t blocks;
    asm volatile(
        "griddepcontrol.wait;\n"
        "griddepcontrol.launch_dependents;\n"
        "mov.u32 %0, %%nctaid.x;\n"
        : "=r"(blocks)::"memory");
    return blocks != 0u;
}

template <typename... P, typename... A>
inline void launch(bool overlap, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                   A&&... args) {
    cudaLaunchConfig_t c = {};
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = overlap ? 1 : 0;
    cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);
}

}  // namespace pd
