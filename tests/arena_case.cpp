// Host-side rules of the plans' memory (csrc/nsp_arena.cu), against the stand-in runtime of tests/fake_cuda.
// usage: arena_case SCENARIO; prints the first violated expectation and returns 1.
#include <cstring>
#include "nsp_arena.h"

using namespace nsp;

#define EXPECT(c)                                                       \
  do {                                                                  \
    if (!(c)) return std::printf("line %d: %s\n", __LINE__, #c), 1;     \
  } while (0)

static void call(Arena* a, cudaStream_t st) {  // a library call: some work, then the mark
  ++st->enqueued;
  arena_used(a, st);
}
static void finish(cudaStream_t st) { st->finished = st->enqueued; }

static constexpr size_t kDev = 300 << 10, kHost = 100 << 10;

static Arena* acquire(int device, cudaStream_t st, bool built = true) {  // with the construction of a plan enqueued
  Arena* a = arena_acquire(device, kDev, kHost, st);
  call(a, a->build);
  if (built) finish(a->build);
  return a;
}

// A plan used on two streams: its memory is free only when both have finished.
static int two_streams() {
  FakeStream s1{101}, s2{102};
  for (int last = 0; last < 2; ++last) {
    Arena* a = acquire(0, nullptr);
    call(a, &s1), call(a, &s2);
    if (last) call(a, &s1);
    arena_release(a);
    finish(last ? &s1 : &s2);  // the stream used last is done, the other one is not
    Arena* b = acquire(0, nullptr);
    EXPECT(b != a);
    EXPECT(fake().waits == 0);
    finish(&s1), finish(&s2);
    arena_release(b);
    arena_trim();
  }
  // more streams than are kept track of: the memory goes back to the driver
  FakeStream many[8] = {{501}, {502}, {503}, {504}, {505}, {506}, {507}, {508}};  // and the construction's
  Arena* a = acquire(0, nullptr);
  for (FakeStream& s : many) call(a, &s);
  arena_release(a);
  EXPECT(fake().device_bytes == 0);
  return 0;
}

// A stream that was destroyed and whose address a new one took is another stream.
static int recycled_stream_address() {
  FakeStream s{201};
  Arena* a = acquire(0, nullptr);
  call(a, &s);
  FakeStream before = s;  // the first stream's work goes on
  a->uses[1].done->on = &before;
  s = FakeStream{202};
  call(a, &s);
  finish(&s);
  arena_release(a);
  EXPECT(acquire(0, nullptr) != a);
  return 0;
}

// Three fitting arenas in use by the caller's stream: the oldest is waited for. In use by others: never.
static int back_pressure() {
  FakeStream mine{401}, other{402};
  Arena* a[3];
  for (int own = 0; own < 3; ++own) {  // none, some, all of them on the caller's stream
    for (Arena*& x : a) x = acquire(0, &mine);
    for (int i = 0; i < 3; ++i) call(a[i], i < (own == 0 ? 0 : own == 1 ? 2 : 3) ? &mine : &other);
    for (Arena* x : a) arena_release(x);
    Arena* b = acquire(0, &mine);
    EXPECT(fake().waits == (own == 2));
    EXPECT((b == a[0]) == (own == 2));
    EXPECT(other.finished == 0);
    finish(&mine);
    other = FakeStream{402};
    arena_release(b);
    arena_trim();
  }
  // an arena that another stream uses as well is not waited for either
  for (Arena*& x : a) x = acquire(0, &mine);
  for (Arena* x : a) call(x, &mine), call(x, &other), arena_release(x);
  Arena* b = acquire(0, &mine);
  EXPECT(b != a[0] && b != a[1] && b != a[2] && fake().waits == 1);
  return 0;
}

// The first call on a stream is ordered behind a construction that still runs, later ones are not ordered again, and a stream
// under capture has the host wait. An arena whose construction still runs is not handed out, nor waited for.
static int order_behind_construction() {
  FakeStream s1{601}, s2{602}, captured{603};
  Arena* a = acquire(0, &s1, false);
  bool built = true;
  auto ordered = [&](FakeStream* st) { return arena_order_built(a, st, &built) == cudaSuccess; };
  EXPECT(!arena_built(a));
  EXPECT(ordered(&s1) && !built && fake().stream_waits == 1);
  call(a, &s1);
  EXPECT(ordered(&s1) && !built && fake().stream_waits == 1);
  EXPECT(ordered(&s2) && !built && fake().stream_waits == 2);
  EXPECT(fake().waits == 0);
  captured.capturing = true;
  EXPECT(ordered(&captured) && built && fake().stream_waits == 2 && fake().waits == 1);
  EXPECT(arena_built(a) && fake().mode == cudaStreamCaptureModeGlobal);
  EXPECT(ordered(&s2) && built && fake().stream_waits == 2);  // complete: nothing to be ordered
  for (int i = 0; i < 4; ++i) {
    Arena* b = acquire(0, &s1, false);
    arena_release(b);  // a plan that was never used
  }
  EXPECT(fake().waits == 1 && fake().live.size() == 2 * 5);
  return 0;
}

static int reuse_and_trim() {
  FakeStream s{301};
  Arena* a = acquire(0, nullptr);
  call(a, &s);
  arena_release(a);
  finish(&s);
  EXPECT(acquire(0, nullptr) == a);
  EXPECT(acquire(1, nullptr)->device == 1);
  s.capturing = true;
  call(a, &s);
  arena_release(a);  // its kernels may run again at any replay
  EXPECT(fake().live.size() == 2);
  return 0;
}

// A plan too large to be kept takes what it needs and no more; a kept one is rounded up for the plans after it.
static int sizes() {
  const size_t big = (48u << 20) + 512;
  fake().device_limit = big;
  Arena* a = arena_acquire(0, big, 1000, nullptr);
  EXPECT(a && a->dev_bytes == big && fake().device_bytes == big);
  arena_release(a);
  EXPECT(fake().device_bytes == 0 && fake().host_bytes == 0);
  fake().device_limit = ~size_t(0);
  // one that only its rounding would make too large is kept as it is
  a = arena_acquire(0, 17u << 20, 1000, nullptr);
  EXPECT(a && a->dev_bytes == 17u << 20);
  arena_release(a);
  EXPECT(fake().device_bytes == 17u << 20);
  arena_trim();
  a = arena_acquire(0, 300 << 10, 1000, nullptr);
  EXPECT(a && a->dev_bytes == 512 << 10);
  arena_release(a);
  EXPECT(arena_acquire(0, 500 << 10, 1000, nullptr) == a);
  // bounded in number and bytes
  Arena* many[12];
  for (Arena*& x : many) x = arena_acquire(0, 6u << 20, 1000, nullptr);
  for (Arena* x : many) arena_release(x);
  EXPECT(fake().live.size() == 2 * 7 + 2);  // eight of 8 MB would be 64 MB of device memory and their host blocks
  for (Arena*& x : many) x = arena_acquire(1, 100, 100, nullptr);
  for (Arena* x : many) arena_release(x);
  EXPECT(fake().live.size() == 2 * 8 + 2);
  return 0;
}

int main(int argc, char** argv) {
  const char* what = argc > 1 ? argv[1] : "";
  if (!std::strcmp(what, "two_streams")) return two_streams();
  if (!std::strcmp(what, "order_behind_construction")) return order_behind_construction();
  if (!std::strcmp(what, "sizes")) return sizes();
  if (!std::strcmp(what, "back_pressure")) return back_pressure();
  if (!std::strcmp(what, "recycled_stream_address")) return recycled_stream_address();
  if (!std::strcmp(what, "reuse_and_trim")) return reuse_and_trim();
  return std::printf("no scenario %s\n", what), 2;
}
