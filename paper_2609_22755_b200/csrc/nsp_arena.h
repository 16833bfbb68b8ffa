// Device and pinned host memory of a plan (see nsp_arena.cu).
#pragma once
#include <cstddef>
#include <mutex>
#include <cuda_runtime.h>

namespace nsp {

struct Arena {
  int device = 0;
  void* dev = nullptr;
  void* host = nullptr;      // pinned, mapped
  char* host_dev = nullptr;  // device pointer to the same memory
  size_t dev_bytes = 0, host_bytes = 0;
  cudaStream_t build = nullptr;  // non-blocking, highest priority: uploads and list construction; the first use of a plan
  // What still may use the arena: one event per stream (by its id: a new stream may take a destroyed one's address), recorded
  // behind the last call on that stream. The events are kept, `n_uses` of them stand for work.
  struct Use {
    unsigned long long stream = 0;
    cudaEvent_t done = nullptr;
  };
  static constexpr int kMaxUses = 8;
  Use uses[kMaxUses];
  int n_uses = 0;
  bool unpooled = false;  // goes back to the driver: used in a stream capture (its kernels may run again at any time), or on
                          // more streams than there are events
  std::mutex mutex;       // uses and unpooled: calls on a plan may come from several threads
};

// Blocks of these sizes stay when their plan is destroyed; larger ones go back to the driver.
bool arena_keeps(size_t dev_bytes, size_t host_bytes);
// An arena of at least the given sizes on the current device that nothing uses any more; null when out of memory. May wait
// for work of the stream `st`, the caller's, but for no other (see kWaitFor).
Arena* arena_acquire(int device, size_t dev_bytes, size_t host_bytes, cudaStream_t st);
// Hands an arena back (null is a no-op); kernels recorded with arena_used may still run.
void arena_release(Arena* a);
// The work enqueued on st so far uses the arena.
void arena_used(Arena* a, cudaStream_t st);
// What the plan's construction has enqueued (its use of a->build, the first one) has completed / is waited for by the host.
bool arena_built(const Arena* a);
cudaError_t arena_wait_built(const Arena* a);
// What is enqueued on st from now on runs behind the construction. *built: it has completed, and nothing needs to be ordered
// behind it any more. A stream that is being captured cannot wait for work outside the capture: then the host does.
cudaError_t arena_order_built(Arena* a, cudaStream_t st, bool* built);
// Frees every idle arena.
void arena_trim();

}  // namespace nsp
