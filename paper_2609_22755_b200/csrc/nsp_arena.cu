// Memory of a plan: one device block, one pinned host block, a stream and events, kept for the next plan when a plan
// is destroyed. A training loop builds a plan per iteration, and raw allocations were most of its cost: ten cudaMalloc,
// a cudaHostAlloc, ten cudaFree (each waits for the device) and cudaGetDeviceProperties made 2.7 ms of a plan of four
// segments, against 0.7 ms of kernels of a batch of 8,192 tokens.
//
// The idle blocks are bounded in number and bytes (beyond that the oldest are freed), and all of them are given back by
// nsp_trim(), or when an allocation fails. An arena whose kernels may still run is never handed out: every call on a plan
// records the arena's event of the call's stream, and a plan that took part in a stream capture (its kernels may run again
// at any replay) gives its memory back to the driver, which waits for the device.
#include <new>
#include <vector>
#include "nsp_arena.h"

namespace nsp {
namespace {

constexpr size_t kMaxIdle = 8;                  // arenas
// With that many fitting arenas still in use by the caller's stream alone, wait for the oldest of them instead of
// allocating: the host is three batches ahead of the device, which has work enough. Arenas that other streams use are left
// alone: their work may depend on what the calling thread does next.
constexpr size_t kWaitFor = 3;
constexpr size_t kMaxIdleBytes = 64ull << 20;   // device + pinned bytes of all idle arenas

std::mutex g_mutex;
std::vector<Arena*>& idle() {
  static std::vector<Arena*>* v = new std::vector<Arena*>();  // never destroyed: plans may outlive static destructors
  return *v;
}

size_t round_up_pow2(size_t n) {
  size_t r = 64 << 10;
  while (r < n) r *= 2;
  return r;
}

void destroy(Arena* a) {  // cudaFree waits for whatever still uses the block
  cudaFree(a->dev);
  if (a->host) cudaFreeHost(a->host);
  for (const Arena::Use& u : a->uses)
    if (u.done) cudaEventDestroy(u.done);
  if (a->build) cudaStreamDestroy(a->build);
  delete a;
}

Arena* create(int device, size_t dev_bytes, size_t host_bytes) {
  Arena* a = new (std::nothrow) Arena;
  if (!a) return nullptr;
  a->device = device;
  // Powers of two, so that later plans of other sizes fit; what that makes too large to be kept takes no more than it needs.
  a->dev_bytes = round_up_pow2(dev_bytes);
  a->host_bytes = round_up_pow2(host_bytes);
  if (!arena_keeps(a->dev_bytes, a->host_bytes)) a->dev_bytes = dev_bytes, a->host_bytes = host_bytes;
  int least = 0, greatest = 0;
  void* hd = nullptr;
  const bool ok = cudaMalloc(&a->dev, a->dev_bytes) == cudaSuccess &&
                  cudaHostAlloc(&a->host, a->host_bytes, cudaHostAllocMapped) == cudaSuccess &&
                  cudaHostGetDevicePointer(&hd, a->host, 0) == cudaSuccess &&
                  cudaEventCreateWithFlags(&a->uses[0].done, cudaEventDisableTiming) == cudaSuccess &&
                  cudaDeviceGetStreamPriorityRange(&least, &greatest) == cudaSuccess &&
                  cudaStreamCreateWithPriority(&a->build, cudaStreamNonBlocking, greatest) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    destroy(a);
    return nullptr;
  }
  a->host_dev = static_cast<char*>(hd);
  return a;
}

bool in_use(const Arena* a) {
  for (int i = 0; i < a->n_uses; ++i)
    if (cudaEventQuery(a->uses[i].done) != cudaSuccess) {
      cudaGetLastError();
      return true;
    }
  return false;
}

bool used_only_by(const Arena* a, unsigned long long stream) {
  for (int i = 1; i < a->n_uses; ++i)  // behind the use of the construction, which no other stream's work holds up for long
    if (a->uses[i].stream != stream) return false;
  return a->n_uses > 1;
}

bool wait_unused(Arena* a) {
  for (int i = 0; i < a->n_uses; ++i)
    if (cudaEventSynchronize(a->uses[i].done) != cudaSuccess) return false;
  a->n_uses = 0;
  return true;
}

}  // namespace

bool arena_keeps(size_t dev_bytes, size_t host_bytes) { return dev_bytes + host_bytes <= kMaxIdleBytes / 2; }

Arena* arena_acquire(int device, size_t dev_bytes, size_t host_bytes, cudaStream_t st) {
  Arena* found = nullptr;
  unsigned long long own = 0;
  const bool have_own = cudaStreamGetId(st, &own) == cudaSuccess;
  if (!have_own) cudaGetLastError();
  {
    std::lock_guard<std::mutex> lock(g_mutex);
    auto& v = idle();
    size_t best = v.size(), oldest = v.size(), fitting = 0;
    for (size_t i = 0; i < v.size(); ++i) {
      const Arena* a = v[i];
      if (a->device != device || a->dev_bytes < dev_bytes || a->host_bytes < host_bytes) continue;
      if (best < v.size() && v[best]->dev_bytes <= a->dev_bytes) continue;
      if (!in_use(a))
        best = i;
      else if (have_own && used_only_by(a, own) && fitting++ == 0)
        oldest = i;
    }
    if (best == v.size() && fitting >= kWaitFor) best = oldest;
    if (best < v.size()) {
      found = v[best];
      v.erase(v.begin() + best);
    }
  }
  if (found && wait_unused(found)) return found;
  if (found) {
    cudaGetLastError();
    destroy(found);
  }
  Arena* a = create(device, dev_bytes, host_bytes);
  if (!a) {
    arena_trim();
    a = create(device, dev_bytes, host_bytes);
  }
  return a;
}

void arena_release(Arena* a) {
  if (!a) return;
  if (a->unpooled || !arena_keeps(a->dev_bytes, a->host_bytes)) {
    destroy(a);
    return;
  }
  std::vector<Arena*> out;
  {
    std::lock_guard<std::mutex> lock(g_mutex);
    auto& v = idle();
    v.push_back(a);
    size_t bytes = 0;
    for (const Arena* x : v) bytes += x->dev_bytes + x->host_bytes;
    while (v.size() > kMaxIdle || bytes > kMaxIdleBytes) {
      bytes -= v.front()->dev_bytes + v.front()->host_bytes;
      out.push_back(v.front());
      v.erase(v.begin());
    }
  }
  for (Arena* x : out) destroy(x);
}

void arena_used(Arena* a, cudaStream_t st) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  std::lock_guard<std::mutex> lock(a->mutex);
  if (cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone &&
      cudaStreamGetId(st, &id) == cudaSuccess) {
    int i = 0;
    while (i < a->n_uses && a->uses[i].stream != id) ++i;
    if (i < Arena::kMaxUses &&
        (a->uses[i].done || cudaEventCreateWithFlags(&a->uses[i].done, cudaEventDisableTiming) == cudaSuccess) &&
        cudaEventRecord(a->uses[i].done, st) == cudaSuccess) {
      a->uses[i].stream = id;
      if (i == a->n_uses) ++a->n_uses;
      return;
    }
  }
  cudaGetLastError();
  a->unpooled = true;
}

namespace {
// Another thread may be capturing, and looking at an event would end its capture unless this thread says that it is unrelated.
struct Unrelated {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  Unrelated() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~Unrelated() { cudaThreadExchangeStreamCaptureMode(&mode); }
};
}  // namespace

bool arena_built(const Arena* a) {
  const Unrelated here;
  if (cudaEventQuery(a->uses[0].done) == cudaSuccess) return true;
  cudaGetLastError();
  return false;
}

cudaError_t arena_wait_built(const Arena* a) {
  const Unrelated here;
  return cudaEventSynchronize(a->uses[0].done);
}

cudaError_t arena_order_built(Arena* a, cudaStream_t st, bool* built) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  *built = arena_built(a);
  if (*built) return cudaSuccess;
  cudaError_t e = cudaStreamIsCapturing(st, &cap);
  if (e != cudaSuccess) return e;
  if (cap != cudaStreamCaptureStatusNone) {
    e = arena_wait_built(a);
    *built = e == cudaSuccess;
    return e;
  }
  e = cudaStreamGetId(st, &id);
  if (e != cudaSuccess) return e;
  {
    std::lock_guard<std::mutex> lock(a->mutex);
    for (int i = 1; i < a->n_uses; ++i)
      if (a->uses[i].stream == id) return cudaSuccess;  // an earlier call on this stream waited
  }
  return cudaStreamWaitEvent(st, a->uses[0].done, 0);
}

void arena_trim() {
  std::vector<Arena*> out;
  {
    std::lock_guard<std::mutex> lock(g_mutex);
    out.swap(idle());
  }
  for (Arena* x : out) destroy(x);
}

}  // namespace nsp
