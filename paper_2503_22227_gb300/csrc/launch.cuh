// Launches with programmatic dependent launch: the kernel may be scheduled
// while the previous kernel on the stream finishes its last CTAs, and waits
// (griddepcontrol.wait) until that kernel has completed and its memory is
// visible.  Before the wait a kernel touches nothing that a launch writes: the
// tensor-core conversions allocate TMEM and load their plan, which has been on
// the device since it was made; in all others the wait is the first statement.
// This hides the launch gap between the kernels of an operation.
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "lanes.h"

namespace catfhe {

// Shared memory's part of an SM's L1, in percent of the largest (164 KB of
// 228).  An SM has one split at a time and changes it only when it is idle, so
// kernels that run side by side and ask for different ones keep each other
// off the SMs; left to itself the runtime takes the split that fits the most
// CTAs of each kernel.  72 still holds two CTAs of the conversion and three of
// the inner product at three digits, and leaves the transforms their L1.
// - Batches over several lanes (lanes.h) use it for every launch: 256 uneven
//   operations 9456 -> 9281 us, two encrypted queries 19.2 -> 18.7 ms (at 58
//   percent 9440 and 19.0, at 86 percent 9460 and 20.1).
// - Otherwise the conversions and the tensor product ask for it, which run
//   beside the other half's transforms: 5 products at N = 2^15 204 -> 196.5
//   us on the device (200 a public call), 16 BFV products 724 -> 717, 8 at N =
//   2^16 1105 -> 1101.  The inner
//   product does not (16 BGV products 315 -> 325 us), nor do the transforms'
//   row passes (one product at N = 2^16 198 -> 200).
constexpr unsigned kSharedPercent = 72;

// shared_percent: the split the launch asks for, 0 for the runtime's choice.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_split(unsigned shared_percent, void (*kernel)(KArgs...), dim3 grid,
                                    dim3 block, size_t smem, cudaStream_t s, Args &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (LaneScope::active()) shared_percent = kSharedPercent;
    if (shared_percent) {
        attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
        attr[1].val.sharedMemCarveout = shared_percent;
        cfg.numAttrs = 2;
    }
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t s, Args &&...args) {
    return launch_pdl_split(0, kernel, grid, block, smem, s, std::forward<Args>(args)...);
}

}  // namespace catfhe
