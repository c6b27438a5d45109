// mpm_launch.h -- programmatic dependent launches.  A kernel launched so starts
// when every CTA of the one before it in the stream has started (has called
// let_next_start) or ended; it does what needs nothing of that one, and every
// thread waits for its end, and for its writes, with wait_for_previous.  Since
// each kernel of such a chain waits in every thread, the end of one implies that
// of all before it.  Both calls do nothing in a kernel launched the ordinary way.
#ifndef MPM_LAUNCH_H
#define MPM_LAUNCH_H
#include <cuda_runtime.h>

namespace mpm {

__device__ __forceinline__ void let_next_start() { cudaTriggerProgrammaticLaunchCompletion(); }
__device__ __forceinline__ void wait_for_previous() { cudaGridDependencySynchronize(); }

// dependent: the operation before this one in the stream is a kernel of the same
// chain (no copy, memset, event or graph); else an ordinary launch
template <typename... Params, typename... Args>
cudaError_t launch_kernel(bool dependent, void (*kernel)(Params...), int grid, int block, size_t smem, cudaStream_t st,
                          Args... args) {
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}

}  // namespace mpm
#endif
