// mpm_scratch.h -- stream-ordered scratch memory of the entry points that have
// no context (mpm_mcis, mpm_render).
//
// The device's default memory pool gives everything back to the driver at each
// synchronisation, and these entry points synchronise: mapping their scratch
// anew took 0.4 to 0.5 ms of every call.  The library keeps a pool of its own
// per device that holds on to at most SCRATCH_KEEP bytes between calls; what
// goes beyond returns at the next synchronisation, and scratch_trim returns the
// rest: when the last context is destroyed, when the caller asks for it
// (mpm_release_scratch), and when an allocation finds no memory.  Allocation and release are
// ordered on the caller's stream, so calls on several streams and threads never
// share live memory.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

namespace mpm {

constexpr unsigned long long SCRATCH_KEEP = 256ull << 20;

// memory on the current device, ordered on st; released by cudaFreeAsync
cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t st);
// gives the kept memory of every device back
void scratch_trim();
// cudaMalloc, once more without the kept memory where there is none left
cudaError_t device_alloc(void **p, size_t bytes);

}  // namespace mpm
