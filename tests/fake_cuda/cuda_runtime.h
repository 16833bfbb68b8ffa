// A stand-in for the part of the CUDA runtime that csrc/nsp_arena.cu uses, so that its rules run on a machine without a GPU.
// Work on a stream finishes when the test says so; an event completes with the work that was enqueued before it.
#pragma once
#include <cstddef>
#include <cstdio>
#include <cstdlib>
#include <set>

struct FakeStream {
  unsigned long long id;
  long enqueued = 0, finished = 0;
  bool capturing = false;
};
struct FakeEvent {
  FakeStream* on = nullptr;
  long at = 0;
  bool complete() const { return !on || on->finished >= at; }
};
typedef FakeStream* cudaStream_t;
typedef FakeEvent* cudaEvent_t;
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorNotReady = 600 };
enum cudaStreamCaptureMode { cudaStreamCaptureModeGlobal = 0, cudaStreamCaptureModeRelaxed = 2 };
enum cudaStreamCaptureStatus { cudaStreamCaptureStatusNone = 0, cudaStreamCaptureStatusActive = 1 };
constexpr unsigned cudaEventDisableTiming = 2, cudaHostAllocMapped = 2, cudaStreamNonBlocking = 1;

struct Fake {
  size_t device_bytes = 0, host_bytes = 0;
  size_t device_limit = ~size_t(0);
  std::set<void*> live;
  int waits = 0;            // host waits for an event that had not completed
  int stream_waits = 0;     // cudaStreamWaitEvent calls
  cudaStreamCaptureMode mode = cudaStreamCaptureModeGlobal;  // of the thread
  unsigned long long next_id = 1;
};
inline Fake& fake() {
  static Fake f;
  return f;
}

inline void* fake_block(size_t n) {
  size_t* p = static_cast<size_t*>(std::malloc(sizeof(size_t) * 2));  // the size is what counts, nothing touches the memory
  p[0] = n;
  fake().live.insert(p);
  return p;
}
inline cudaError_t cudaMalloc(void** p, size_t n) {
  if (fake().device_bytes + n > fake().device_limit) return cudaErrorInvalidValue;
  fake().device_bytes += n;
  *p = fake_block(n);
  return cudaSuccess;
}
inline cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  if (!fake().live.erase(p)) std::abort();
  fake().device_bytes -= *static_cast<size_t*>(p);
  std::free(p);
  return cudaSuccess;
}
inline cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
  fake().host_bytes += n;
  *p = fake_block(n);
  return cudaSuccess;
}
inline cudaError_t cudaFreeHost(void* p) {
  if (!fake().live.erase(p)) std::abort();
  fake().host_bytes -= *static_cast<size_t*>(p);
  std::free(p);
  return cudaSuccess;
}
inline cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) { return *d = h, cudaSuccess; }
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
inline cudaError_t cudaDeviceGetStreamPriorityRange(int* least, int* greatest) { return *least = 0, *greatest = -5, cudaSuccess; }
inline cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) {
  *s = new FakeStream{fake().next_id++};
  return cudaSuccess;
}
inline cudaError_t cudaStreamDestroy(cudaStream_t s) { return delete s, cudaSuccess; }
inline cudaError_t cudaStreamGetId(cudaStream_t s, unsigned long long* id) { return *id = s ? s->id : 0, cudaSuccess; }
inline cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* c) {
  *c = s->capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
inline cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = new FakeEvent, cudaSuccess; }
inline cudaError_t cudaEventDestroy(cudaEvent_t e) { return delete e, cudaSuccess; }
inline cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return e->on = s, e->at = s->enqueued, cudaSuccess; }
inline cudaError_t cudaEventQuery(cudaEvent_t e) { return e->complete() ? cudaSuccess : cudaErrorNotReady; }
inline cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode* m) {
  const cudaStreamCaptureMode was = fake().mode;
  fake().mode = *m, *m = was;
  return cudaSuccess;
}
inline cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned) {
  if (s->capturing) return cudaErrorInvalidValue;  // the event was recorded outside the capture
  ++fake().stream_waits;
  return cudaSuccess;
}
inline cudaError_t cudaEventSynchronize(cudaEvent_t e) {
  if (!e->complete()) {
    ++fake().waits;
    e->on->finished = e->at;
  }
  return cudaSuccess;
}
