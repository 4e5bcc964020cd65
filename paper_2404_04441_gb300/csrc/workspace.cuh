// The gradient's kept workspace (wave.cu) as other allocations see it.
#pragma once

#include <cuda_runtime.h>

namespace gbw {

// cudaMalloc on the current device; if that runs out of memory, frees the kept
// workspace and tries again.
cudaError_t device_malloc(void **p, size_t bytes);
// Frees the current CUDA context's kept workspace; false if there is none.
bool drop_kept_workspace();

}  // namespace gbw
