// Device workspaces of the calls without a context: a stream-ordered pool per
// device that keeps up to kWorkKeep bytes between calls (allocating and freeing a
// few hundred megabytes took 0.5 of the 2.1 ms of a 4096^3 product).  The pool is
// CUDA's, so threads and streams may share it; work_trim gives the kept memory
// back (mlcc3_release_workspace, when a context is destroyed, and when an allocation of
// the library fails).
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

namespace mlcc3 {

constexpr size_t kWorkKeep = (size_t)1 << 30;

cudaError_t work_alloc(void **p, size_t bytes, cudaStream_t st);
void work_free(void *p, cudaStream_t st);
void work_trim();

}  // namespace mlcc3
