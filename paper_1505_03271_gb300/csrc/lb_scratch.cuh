// lb_scratch.cuh -- device memory borrowed for the length of a call
// (lb_scratch.cu), and allocation that takes it back when memory runs out.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

namespace lbgb {

// Borrow and give back, in the order of the stream.  A borrower joins before
// its first loan and leaves, its streams synchronised, after its last.
cudaError_t scratch_take(void** p, size_t bytes, int device, cudaStream_t s);
void scratch_give(void* p, cudaStream_t s);
void scratch_join(int device);
void scratch_leave(int device);
// Return what nobody borrows to the device; false if there was nothing.
// Synchronises the device.
bool scratch_reclaim(int device);
// cudaMalloc on the current device, once more after scratch_reclaim.
cudaError_t device_malloc(void** p, size_t bytes);

}  // namespace lbgb
