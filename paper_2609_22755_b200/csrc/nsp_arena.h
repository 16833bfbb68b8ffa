// Device and pinned host memory of a plan (see nsp_arena.cu).
#pragma once
#include <cstddef>
#include <cuda_runtime.h>

namespace nsp {

struct Arena {
  int device = 0;
  void* dev = nullptr;
  void* host = nullptr;      // pinned, mapped
  char* host_dev = nullptr;  // device pointer to the same memory
  size_t dev_bytes = 0, host_bytes = 0;
  cudaStream_t build = nullptr;  // non-blocking, highest priority: uploads and list construction
  cudaEvent_t done = nullptr;    // recorded behind the last call that used the arena
  bool pending = false;          // `done` has been recorded
  bool captured = false;         // used in a stream capture: its kernels may run again at any time
};

// An arena of at least the given sizes on the current device that nothing uses any more; null when out of memory.
Arena* arena_acquire(int device, size_t dev_bytes, size_t host_bytes);
// Hands an arena back (null is a no-op); kernels recorded with arena_used may still run.
void arena_release(Arena* a);
// The work enqueued on st so far uses the arena.
void arena_used(Arena* a, cudaStream_t st);
// Frees every idle arena.
void arena_trim();

}  // namespace nsp
