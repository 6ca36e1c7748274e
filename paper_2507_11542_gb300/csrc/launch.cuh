// launch.cuh -- kernels of one stream that start before the kernel in front of
// them has ended (programmatic dependent launch). Between two kernels that
// follow each other in a stream this GPU leaves 2 to 4 us (a kernel's end is
// noticed in steps of about 2 us: a kernel of 1.0 us takes 4.1 us of a stream,
// one of 6.0 us 8.2); with this attribute 0.5 us (1.6 and 6.9 us). A stage
// kernel of the smaller grids takes 2 to 20 us.
//
// Rules: a kernel that is launched with launch_dependent calls grid_wait() (or
// grid_wait_only()) before it touches global memory, in every thread. It returns
// when every earlier kernel of the stream has ended and its results are visible:
// the kernel in front ends only after its own wait. Loads of what other kernels
// write are neither read-only (.nc) nor through const __restrict__ kernel
// parameters, which the compiler may move above the wait.
//
// The next kernel may start (grid_next()) only after the wait, so that one kernel
// at most waits on the SMs beside the running one. Allowed before the wait, the
// whole rest of the stream that fits comes to wait there, blocks are dealt out
// around them, and some SMs get two of a kernel's blocks and others none: 40 x 1000
// FP64 ENO3, 30 us a step with four steps in flight and 65 with 256 (now 25 and
// 24), 21^3 30 and 53 (29 and 29), 101^2 WENO5 15.3 and 17.4 (13.8 and 12.7; a
// solve 2280 -> 1800 us). The stage kernels call it when their first planes are
// staged: right behind the wait the next kernel's blocks set themselves up while
// this one's first loads are due (51^2 FP32 5.4 us a step, now 4.9; 161x113x79 51.9
// and 50.8).
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace hj {

__device__ __forceinline__ void grid_wait_only() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_wait() {
    grid_wait_only();
    grid_next();
}

template <typename... Params, typename... Args>
inline cudaError_t launch_dependent(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                    Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace hj
