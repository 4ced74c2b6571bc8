// Launches that follow a kernel of the same call on the same stream.
//
// A render is a chain of launches, each reading what the one before wrote, and between two ordinary
// launches the device stays empty while the first one's writes are flushed and the second one is
// set up.  launch_step() lets that set-up run ahead: the grid may start once every block of the one
// before has ended, and each of its threads waits in start_of_step(), before its first access to
// memory, until that grid is complete and its writes are visible.  Rules:
//  - every kernel given to launch_step() begins with start_of_step(), in all its threads (a grid is
//    then complete only after the one before it, so it also follows all earlier ones).  Only behind
//    that wait are an earlier grid's writes promised to be visible, so none reads anything before it;
//  - what an earlier launch of the chain writes is read through plain pointers (chained_ptr):
//    a const __restrict__ parameter may be read by loads that take memory as constant for the
//    whole life of the grid, which begins before the wait;
//  - chained is set only where the operation before on the stream is a kernel of the same call: the
//    first launch of a call, and one behind a copy, a memset, a recorded event (stage times) or a
//    wait for an event, is an ordinary one.
// Measured: 64 x 64 pixels, 6 launches, 98.4 -> 88.9 us; 500 x 333 in 64-slot groups, 20 launches,
// 808 -> 769; 1920 x 1080, 1174 -> 1158; 24 server requests 6530 -> 6460.  Letting blocks start
// while the one before is still running (an early trigger) gave nothing more: they then fill the
// SMs in the order in which these drain, and the 64-slot groups took 781 to 800 us.  Nodes of a
// captured graph follow each other closely already (16-job batch 5424 us against 5440), so a
// capture gets ordinary launches.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace cr {

__device__ __forceinline__ void start_of_step() { cudaGridDependencySynchronize(); }

template <typename... P, typename... A>
void launch_step(bool chained, void (*kernel)(P...), uint32_t grid, uint32_t block, size_t smem, cudaStream_t st,
                 A&&... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = chained ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Kernel parameters that point at what earlier launches write (kChained: launched by launch_step
// with chained set).
template <bool kChained, typename T>
struct ChainedPtr {
    using type = const T*;
};
template <typename T>
struct ChainedPtr<false, T> {
    using type = const T* __restrict__;
};
template <bool kChained, typename T>
using chained_ptr = typename ChainedPtr<kChained, T>::type;

} // namespace cr
