// Host side of libnsp: argument validation, plan object, tensor-map encoding and kernel launches.
// Plain C ABI (include/nsp.h); no torch types, no CPU fallback.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>
#include <cuda_bf16.h>
#include "nsp_arena.h"
#include "nsp_internal.cuh"
#include "sm100_ptx.cuh"

namespace nsp {
static std::atomic<int64_t> g_launches{0};
void count_launches(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
}  // namespace nsp

using namespace nsp;

struct nsp_plan {
  int32_t n_seg = 0, bm = kBM, bn = kBN, head_dim = kHeadDim;
  int device = 0, num_sms = 0;
  int64_t q_elems = 0, kv_elems = 0, lse_elems = 0, n_fwd = 0, n_bwd = 0;
  std::vector<SegInfo> seg;
  std::vector<RunInfo> runs;
  // device state, all of it inside the arena
  Arena* arena = nullptr;
  mutable std::atomic<bool> built{false};  // known to be complete on the device; until then every stream's first call waits for it
  SegInfo* d_seg = nullptr;
  int64_t* d_row_base = nullptr;  // [n_seg + 1] first packed (token, head) row of each segment
  nsp_tile_t* d_fwd = nullptr;
  nsp_tile_t* d_bwd = nullptr;
  // The backward items in the order the kernel walks them (nsp_plan_get, pass 2). The published work list (pass 1) is
  // sorted by cost alone; walked in that order, the CTAs that run at the same time hold key tiles of MANY (segment, kv
  // head) groups, a q tile's fp32 dQ accumulator rows are touched by a few CTAs now and by the others much later, and
  // they travel to DRAM and back every time (16 segments of 8,192 tokens, 32q/4kv: 193 GB of DRAM traffic for a backward
  // pass whose tensors total 5 GB, L2 hit rate 21 %, the kernel runs at HBM speed). Walked group by group -- all key
  // tiles of one (segment, kv head), first key tile (largest cost) first -- the CTAs of a group sweep the q tiles
  // together and every accumulator row, Q tile and dO tile is fetched once per group. Groups go by segment length
  // descending (ties: segment, then kv head, ascending): all CTAs then start the longest group at the same moment, which
  // is what keeps them on the same q tile (started after a tail of shorter groups they enter it scattered and stay
  // scattered: 131,072 tokens at 16q/1kv next to 131,072 tokens of shorter segments ran 4 % slower that way, a
  // long-tailed batch 8 %), and the walk ends with the cheapest items of the shortest segments. Same items, same costs:
  // a permutation of the published list.
  nsp_tile_t* d_bwd_exec = nullptr;
  nsp_tile_t* d_bwd_parts = nullptr;        // the same items divided into parts (see divide_items)
  nsp_tile_t* d_bwd_first_parts = nullptr;  // the first-tile kernel's items likewise
  int64_t n_parts = 0, n_first_parts = 0;   // 0: not divided
  nsp_tile_t* d_bwd_pairs = nullptr;          // items of the pair kernel: two key tiles of a segment of at least kPairTiles
  int64_t n_bwd_pairs = 0, n_bwd_paired = 0;  // their number, and how many of d_bwd_exec's first items they stand for
  bool pairs_bf16 = false;                    // with bf16 dK / dV too (see kPairRest)
  int32_t* d_turns = nullptr;               // turn counters of the divided items
  nsp_tile_t* d_bwd_first = nullptr;  // one item per (segment or pack, kv head): the first-tile kernels' list
  int64_t n_first = 0;
  nsp_tile_t* d_fwd_first = nullptr;  // the first-tile forward kernel's list: d_bwd_first, or with pairs of KV heads (cost 2)
  int64_t n_fwd_first = 0;
  RowInfo* d_rows = nullptr;          // row tables of the packs, 128 entries each (d_seg holds the packs' entries after
  int64_t n_packs = 0;                // the n_seg segments')
  nsp_tile_t* d_fwd_pairs = nullptr;  // the forward items that visit at least two key tiles, in the pairs the general
  int64_t n_pairs = 0;                // kernel runs (q tile 0 of every segment runs in the first-tile forward kernel)
  bool deterministic = false;         // plan option: dQ tiles added in key-tile order
  bool rounded_dq = false;            // plan option: dQ terms rounded to a fixed quantum (order-independent sums)
  // Small batches launch the preprocess and the main kernel chained as well (see launch_chained_if), so that the main
  // kernel runs beside the first-tile kernel on SMs that one leaves idle and neither pays its launch: 8,192 tokens at
  // 32q/4kv 615 -> 590 us, four short sequences at 8q/2kv 97 -> 64 us. A large batch fills every SM with either kernel,
  // and a block that starts on an SM still set up for its predecessor keeps that one's split between L1 and shared
  // memory: with L1 at 28 KB instead of 60 KB the main kernel is 3 % slower (425,984 tokens: 527 -> 550 ms a step) and
  // the preprocess kernel 25 %. The lines cross between 110 and 300 steps per SM.
  bool small_bwd = false;
  int32_t max_len = 0;                // longest segment: no preprocess / main / postprocess launch when <= 128
  int32_t* d_front = nullptr;        // [n_bwd / kFrontBlock + 1] start-alignment counters of the backward kernel
  int32_t* d_counters = nullptr;  // [0] forward cursor, [1] backward cursor
  int32_t* d_status = nullptr;    // {code, item, where, aux}
  int32_t* h_status = nullptr;    // the same record in mapped pinned host memory (written by the failing kernel)
  int32_t* h_status_dev = nullptr;  // device pointer to h_status
  int sticky = 0;
  long long wait_limit = NSP_WAIT_CYCLES_DEFAULT;  // SM clocks a device-side wait may take
  int withhold = 0;                                // checked build: failure-detection test switch
  int withhold_pair = 0;                           // likewise, the pair kernel of the backward pass
  // optional per-kernel timing (CUDA events on the launching stream)
  bool profiling = false;
  cudaEvent_t ev[2 * NSP_KERNEL_COUNT] = {};
  bool ev_valid[NSP_KERNEL_COUNT] = {};
  // host-to-host step (nsp_attn_step_host): a copy stream and ordering events, created at its first call
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t hev[6] = {};
};

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// Tensor map of one run: a dense bf16 [tokens, heads, 128] tensor; tiles are {64 dims, 1 head, `rows` tokens}
// with 128-byte swizzle, rows past the run read as zero.
bool encode_run_map(CUtensorMap* out, const void* base, int64_t elem_off, int64_t tokens, int heads, int head_dim, int rows = kBM) {
  EncodeTiledFn enc = get_encode_fn();
  if (!enc) return false;
  if (tokens <= 0) {
    std::memset(out, 0, sizeof(*out));
    return true;
  }
  const cuuint64_t dims[3] = {static_cast<cuuint64_t>(head_dim), static_cast<cuuint64_t>(heads),
                              static_cast<cuuint64_t>(tokens)};
  const cuuint64_t strides[2] = {static_cast<cuuint64_t>(head_dim) * 2, static_cast<cuuint64_t>(heads) * head_dim * 2};
  const cuuint32_t box[3] = {64, 1, static_cast<cuuint32_t>(rows)};
  const cuuint32_t estr[3] = {1, 1, 1};
  void* ptr = const_cast<char*>(static_cast<const char*>(base)) + elem_off * 2;
  return enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, ptr, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// fp32 [tokens, heads, head_dim] output of one run, boxes of 32 columns x `rows` rows (128 bytes per row), with the 128-byte
// swizzle or row after row
bool encode_run_map_f32(CUtensorMap* out, void* base, int64_t elem_off, int64_t tokens, int heads, int head_dim, int rows = 128,
                        bool swizzled = true) {
  EncodeTiledFn enc = get_encode_fn();
  if (!enc) return false;
  if (tokens <= 0) {
    std::memset(out, 0, sizeof(*out));
    return true;
  }
  const cuuint64_t dims[3] = {static_cast<cuuint64_t>(head_dim), static_cast<cuuint64_t>(heads),
                              static_cast<cuuint64_t>(tokens)};
  const cuuint64_t strides[2] = {static_cast<cuuint64_t>(head_dim) * 4, static_cast<cuuint64_t>(heads) * head_dim * 4};
  const cuuint32_t box[3] = {32, 1, static_cast<cuuint32_t>(rows)};
  const cuuint32_t estr[3] = {1, 1, 1};
  void* ptr = static_cast<char*>(base) + elem_off * 4;
  return enc(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, ptr, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             swizzled ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The plan's failure state: set once a kernel of the plan has recorded a failure. The record sits in mapped pinned
// host memory, so looking at it costs a host load, not a synchronisation; a failure is seen by the first call made
// after the failing kernel wrote it.
int plan_failed(const nsp_plan* plan) {
  if (!plan->sticky && plan->h_status) {
    const int code = *reinterpret_cast<volatile int32_t*>(plan->h_status);
    if (code != 0) const_cast<nsp_plan*>(plan)->sticky = code;
  }
  return plan->sticky;
}
StatusWord status_word(const nsp_plan* plan) { return StatusWord{plan->d_status, plan->h_status_dev}; }

// Host-side call log: with NSP_LOG=1 in the environment (read once) every plan construction and every compute call
// prints one line to stderr. Nothing on the device changes.
bool log_on() {
  static const bool on = [] {
    const char* e = std::getenv("NSP_LOG");
    return e && e[0] && e[0] != '0';
  }();
  return on;
}
#define NSP_LOGF(...)                        \
  do {                                       \
    if (log_on()) {                          \
      std::fprintf(stderr, "[nsp] " __VA_ARGS__); \
      std::fputc('\n', stderr);              \
    }                                        \
  } while (0)

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Divides backward items into parts of at most about `most` steps (see kMaxParts) and lists them: the longest first where
// the dQ accumulator is no more than kMostByLength, otherwise in the order of the items, the walked one, which keeps the
// CTAs of a group on the same q tiles but packs the parts worse. Backward pass, us, by length / walked / undivided: 17,545
// tokens at 8q/2kv (68 MiB) 1,652 / 1,850 / 1,693; at 16q/1kv four segments of 9,000 tokens (281 MiB) 3,494 / 5,074 / 4,701,
// two of 14,000 and forty of 500 (375 MiB) 4,372 / 6,151 / 5,144; 8,000 tokens and twenty times 500 at 64q/4kv (562 MiB) 3,049 /
// 4,493 / 4,173; beyond, 79,335 and 79,500 long-tailed tokens at 16q/1kv (620 MiB) 1,654 / 1,599 / 1,925 and 4,362 / 4,243 /
// 5,412, 53,428 at 32q/2kv (834 MiB) 2,186 / 2,182 / 2,397, 47,878 tokens at 64q/4kv in 173 segments (1,500 MiB) 3,187 / 3,121 a
// step. A part has its own K / V loads and its own dK / dV epilogue, ~14,000 clocks or the time of 3-4 steps.
// Returns an empty list when nothing is divided.
// Where the lines lie: an item is divided when it is longer than the SMs' share of all steps, because the longest item
// then bounds the kernel. Microseconds a step with parts of at most share / 2, share, whole: 8,192 tokens in one
// segment at 32q/4kv 2,198, 2,124, 2,462; 17,545 tokens at 8q/2kv 1,063, 1,043, 1,158; 8,192 tokens in ten segments 718,
// 694, 737. Smaller parts than kMinPart steps cost more than they give: 1,511 tokens of three head structures, parts of
// 24 / 16 / 12 / 8 / 4 steps: 101, 85, 88, 109, 125 us (whole: 114). The first-tile kernel's items have one step per q
// head of twice that length and run beside the main kernel: divided they are worth it where they, not the main kernel,
// bound the call (20 segments of about 100 tokens at 64q/4kv 233 -> 216 us; parts of eight steps 248, of two 215). The pair
// kernel does not start beside them: there they are divided where the parts fit one wave (first-tile kernel, us, whole /
// parts: 8 segments of 2,048 tokens at 64q/4kv 103 / 65, 16 of 8,192 at 32q/4kv 85 / 65; in two or more waves 32 of
// 4,096 90 / 112, 64 of 2,048 156 / 195, 64 of 2,048 at 64q/4kv 285 / 310).
constexpr int kMinPart = 16, kMinFirstPart = 4;
constexpr int64_t kMostByLength = 600ll << 20;
// Backward items that run on CTA pairs: segments of at least kPairTiles key tiles and kPairSteps steps for the first of them,
// taken from the longest down to the first that has fewer (a batch whose longest has too few steps is left alone). A
// pair computes one tile more than it needs (the second key tile has nothing of the item's last q tile) and meets its partner
// between items. Backward pass over about 131,072 tokens, ms, pairs / single CTAs: 32q/4kv in segments of 1,024 tokens (8
// tiles) 4.25 / 4.22, 1,536 5.55 / 5.71 (main kernels alone 4.74 / 4.71), 2,048 6.68 / 6.71 (5.88 / 6.07), 3,072 9.56 /
// 9.81, 4,096 12.2 / 12.6; 64q/4kv in 1,024 8.9 / 8.9, 2,048 14.0 / 14.4, 4,096 24.4 / 25.7; one head per KV head (16q/16kv)
// 2,000 4.10 / 3.84, 3,000 5.32 / 5.10, 4,000 6.50 / 6.69. Batches whose longest
// item would bound the kernel are divided instead (divide_items), and small ones (small_bwd) run their kernels side by side.
constexpr int kPairTiles = 16, kPairSteps = 32;
// The items that are left run behind the pairs, and with bf16 gradients undivided: that launch then lasts at least as long as
// its longest item. There nothing is paired unless this item is, times the SMs, at most 1 / kPairRest of the paired items'
// steps (counted per key tile). Main kernels, us, pairs / single CTAs, at 32q/4kv and bf16 gradients, by that share: 16 segments of 2,048
// tokens and one of 1,900 at 64q/4kv (23 %) 3,370 / 3,030, 14 of 2,048 and four of 1,900 (26 %) 1,672 / 1,549, 32 of 2,048 and one of
// 1,900 (11 %) 3,180 / 3,030, 16 of 4,096 and one (6 %) 5,785 / 5,984, 64 of 2,048 and one (5.7 %) 6,220 / 6,149, 24 of 4,096 and one
// (4 %) 8,492 / 8,704, 32 of 4,096 and 20 of 1,000 (1.5 %) 11,310 / 11,550, 16 of 8,192 and one (1.5 %) 20,500 / 21,800.
constexpr int kPairRest = 20;
struct WholeItem {
  int32_t seg, head, tile, steps;
};
std::vector<nsp_tile_t> divide_items(const std::vector<WholeItem>& items, int64_t most, bool by_length, int32_t* n_turns) {
  struct Part {
    nsp_tile_t t;
    int32_t steps;
  };
  std::vector<Part> out;
  const int32_t turn0 = *n_turns;
  for (const WholeItem& w : items) {
    const int64_t k = std::min<int64_t>(std::min<int64_t>(kMaxParts, w.steps), (w.steps + most - 1) / most);
    const int32_t turn = k > 1 ? (*n_turns)++ : 0;
    for (int32_t p = 0; p < k; ++p)
      out.push_back(Part{nsp_tile_t{w.seg, w.head, w.tile | p << 16 | static_cast<int32_t>(k) << 24, turn},
                         static_cast<int32_t>(w.steps / k + (p < w.steps % k))});
  }
  std::vector<nsp_tile_t> list;
  if (*n_turns == turn0) return list;
  // the parts of an item do not grow with their number, so a stable sort keeps them in order
  if (by_length)
    std::stable_sort(out.begin(), out.end(), [](const Part& a, const Part& b) { return a.steps > b.steps; });
  for (const Part& p : out) list.push_back(p.t);
  return list;
}

// Up to that many (tile, segment) terms the list kernel takes the positions as sums over the segments, beyond it the host
// counts them (plan_tile_bases). Whole construction in ms, sums / counted: 1,000 segments of 24 tiles (24 M terms) 0.42 /
// 0.50, 2,000 of 64 tiles (256 M) 7.0 / 7.4, 8,192 of one tile (67 M) 2.0 / 2.1, 65,535 of four tiles 74 / 11, of eight 142 / 16.
constexpr int64_t kMostSumTerms = 1ll << 26;

void free_plan(nsp_plan* p) {
  if (!p) return;
  for (cudaEvent_t e : p->ev)
    if (e) cudaEventDestroy(e);
  for (cudaEvent_t e : p->hev)
    if (e) cudaEventDestroy(e);
  if (p->copy_stream) cudaStreamDestroy(p->copy_stream);
  arena_release(p->arena);
  delete p;
}

// Brackets every call that enqueues work of a plan, however it returns: behind the plan's construction (see
// arena_order_built), and with the arena marked as used by the stream (see arena_used).
struct UsesArena {
  const nsp_plan* plan;
  cudaStream_t st;
  cudaError_t ready;
  UsesArena(const nsp_plan* p, cudaStream_t stream) : plan(p), st(stream), ready(cudaSuccess) {
    bool built = p->built.load(std::memory_order_acquire);
    if (!built) {
      ready = arena_order_built(p->arena, st, &built);
      if (built) p->built.store(true, std::memory_order_release);
    }
  }
  ~UsesArena() { arena_used(plan->arena, st); }
};

// Do backward calls with dK / dV of that type run the plan's long segments on CTA pairs?
bool runs_on_pairs(const nsp_plan* plan, int dkv_dtype) {
  return plan->n_bwd_pairs > 0 && (dkv_dtype == NSP_F32 || plan->pairs_bf16);
}

// Record the start / stop event of kernel `id` when profiling is on.
void prof_mark(const nsp_plan* plan, int id, int stop, cudaStream_t st) {
  if (!plan->profiling) return;
  nsp_plan* p = const_cast<nsp_plan*>(plan);
  cudaEventRecord(p->ev[2 * id + stop], st);
  if (stop) p->ev_valid[id] = true;
}

}  // namespace

extern "C" {

const char* nsp_status_string(int code) {
  switch (code) {
    case NSP_OK: return "ok";
    case NSP_ERR_INVALID_ARG: return "invalid argument";
    case NSP_ERR_UNSUPPORTED: return "unsupported configuration";
    case NSP_ERR_ALLOC: return "allocation failed";
    case NSP_ERR_CUDA: return "CUDA call failed";
    case NSP_ERR_DEVICE_TIMEOUT: return "device-side wait timed out";
    case NSP_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    case NSP_ERR_DEVICE_ASSERT: return "device-side index check failed (checked build)";
    case NSP_ERR_INFEASIBLE: return "no plan within the token budget";
    default: return "unknown status";
  }
}

int64_t nsp_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

int nsp_plan_tiles(const int32_t* cu_seqlens, const int32_t* hq, const int32_t* hkv, int32_t n_seg, int32_t head_dim,
                   const nsp_plan_opts* opts, void* stream, nsp_plan_t** out_plan) {
  if (!out_plan) return NSP_ERR_INVALID_ARG;
  *out_plan = nullptr;
  if (n_seg < 0 || (n_seg > 0 && (!cu_seqlens || !hq || !hkv))) return NSP_ERR_INVALID_ARG;
  if (n_seg > 0 && cu_seqlens[0] != 0) return NSP_ERR_INVALID_ARG;
  for (int s = 0; s < n_seg; ++s) {
    if (cu_seqlens[s + 1] < cu_seqlens[s]) return NSP_ERR_INVALID_ARG;
    if (hq[s] <= 0 || hkv[s] <= 0 || hq[s] % hkv[s] != 0) return NSP_ERR_INVALID_ARG;
  }
  int bm = kBM, bn = kBN;
  if (opts) {
    if (opts->bm <= 0 || opts->bn <= 0) return NSP_ERR_INVALID_ARG;
    bm = opts->bm;
    bn = opts->bn;
    if (opts->order_version != 1 || (opts->flags & ~(NSP_PLAN_DETERMINISTIC_DQ | NSP_PLAN_ROUNDED_DQ)) != 0) return NSP_ERR_UNSUPPORTED;
  }
  if (head_dim != 128 && head_dim != 64) return NSP_ERR_UNSUPPORTED;
  if (bm != kBM || bn != kBN) return NSP_ERR_UNSUPPORTED;
  if (n_seg >= 65536) return NSP_ERR_UNSUPPORTED;

  nsp_plan* p = new (std::nothrow) nsp_plan;
  if (!p) return NSP_ERR_ALLOC;
  p->n_seg = n_seg;
  p->head_dim = head_dim;
  p->deterministic = opts && (opts->flags & NSP_PLAN_DETERMINISTIC_DQ) != 0;
  p->rounded_dq = opts && !p->deterministic && (opts->flags & NSP_PLAN_ROUNDED_DQ) != 0;
  p->bm = bm;
  p->bn = bn;
  std::vector<int64_t> row_base;
  std::vector<int32_t> tile_base;
  std::vector<PlanKey> keys;
  try {
    p->seg.resize(n_seg);
    row_base.resize(n_seg + 1);
    tile_base.resize(n_seg + 1);
    keys.resize(n_seg);
  } catch (...) {
    delete p;
    return NSP_ERR_ALLOC;
  }
  int64_t q_off = 0, kv_off = 0, lse_off = 0, nf = 0, nb = 0, tiles = 0;
  for (int s = 0; s < n_seg; ++s) {
    const int64_t L = static_cast<int64_t>(cu_seqlens[s + 1]) - cu_seqlens[s];
    const int64_t Mt = (L + bm - 1) / bm, Nt = (L + bn - 1) / bn;
    if (hq[s] > 256 || Mt >= 65536 || Nt >= 65536 || (hq[s] / hkv[s]) * Mt >= (1 << 24)) {
      delete p;
      return NSP_ERR_UNSUPPORTED;
    }
    const bool new_run = s == 0 || hq[s] != hq[s - 1] || hkv[s] != hkv[s - 1];
    if (new_run) {
      if (p->runs.size() == NSP_MAX_RUNS) {
        delete p;
        return NSP_ERR_UNSUPPORTED;
      }
      p->runs.push_back(RunInfo{q_off, kv_off, 0, hq[s], hkv[s]});
    }
    RunInfo& run = p->runs.back();
    SegInfo& sg = p->seg[s];
    std::memset(&sg, 0, sizeof(sg));
    sg.q_off = q_off;
    sg.kv_off = kv_off;
    sg.lse_off = lse_off;
    sg.len = static_cast<int32_t>(L);
    sg.hq = hq[s];
    sg.hkv = hkv[s];
    sg.run = static_cast<int32_t>(p->runs.size() - 1);
    sg.tok_in_run = static_cast<int32_t>(run.tokens);
    sg.turn_off = static_cast<int32_t>(nf);  // one turn counter per forward item = (q head, q tile) of the segment
    run.tokens += L;
    row_base[s] = lse_off;
    tile_base[s] = static_cast<int32_t>(tiles);
    keys[s] = PlanKey{static_cast<int32_t>(Mt), hq[s], hq[s] / hkv[s], static_cast<int32_t>(L)};
    tiles += Mt;
    q_off += L * hq[s] * head_dim;
    kv_off += L * hkv[s] * head_dim;
    lse_off += L * hq[s];
    nf += Mt * hq[s];
    nb += Nt * hkv[s];
  }
  for (int s = 0; s < n_seg; ++s) p->seg[s].run_tokens = static_cast<int32_t>(p->runs[p->seg[s].run].tokens);
  row_base[n_seg] = lse_off;
  tile_base[n_seg] = static_cast<int32_t>(tiles);
  p->q_elems = q_off;
  p->kv_elems = kv_off;
  p->lse_elems = lse_off;
  p->n_fwd = nf;
  p->n_bwd = nb;
  if (nf >= (1ll << 31) || nb >= (1ll << 31)) {
    delete p;
    return NSP_ERR_UNSUPPORTED;
  }

  int64_t bwd_steps = 0;  // (key tile, q tile, q head) steps of the backward pass
  std::vector<int32_t> order;  // segments by length descending: the order of the groups the backward kernel walks
  std::vector<nsp_tile_t> bwd_first;
  std::vector<SegInfo> pack_segs;
  std::vector<RowInfo> pack_rows;
  try {
    order.resize(n_seg);
    for (int s = 0; s < n_seg; ++s) order[s] = s;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return p->seg[x].len > p->seg[y].len; });
    // the first-tile kernel's items: key tile 0 of every group, in the same group order; q heads of the group = steps
    // Segments of fewer than 128 tokens that follow one another inside a run (they are contiguous in every tensor)
    // and together hold at most 128 tokens share one first tile: such a pack becomes an entry of its own behind the
    // segments (len = its tokens, offsets of its first segment) with a row table, and takes its segments' places in
    // the first-tile list.
    std::vector<int32_t> pack_of(n_seg, -1);
    {
      // a pack and the one behind it hold more than 128 tokens together, or another run or a long segment lies between them
      int64_t short_segs = 0, short_tokens = 0;
      for (const SegInfo& sg : p->seg)
        if (sg.len > 0 && sg.len < kBM) ++short_segs, short_tokens += sg.len;
      pack_rows.reserve(kBM * std::min<int64_t>(short_segs / 2, 2 * short_tokens / kBM + 1));
    }
    for (int s0 = 0; s0 < n_seg;) {
      const SegInfo& first = p->seg[s0];
      if (first.len <= 0 || first.len >= kBM) { ++s0; continue; }
      int s1 = s0 + 1, tokens = first.len, members = 1;
      while (s1 < n_seg && p->seg[s1].run == first.run && p->seg[s1].len < kBM && tokens + p->seg[s1].len <= kBM) {
        tokens += p->seg[s1].len;
        members += p->seg[s1].len > 0;
        ++s1;
      }
      if (members >= 2) {
        SegInfo pk = first;
        pk.len = tokens;
        pk.rows = static_cast<int32_t>(pack_rows.size() / kBM) + 1;
        int row = 0;
        for (int s = s0; s < s1; ++s) {
          const SegInfo& sg = p->seg[s];
          if (sg.len <= 0) continue;
          pack_of[s] = n_seg + static_cast<int32_t>(pack_segs.size());
          RowInfo ri{};
          ri.lse_base = sg.lse_off - row;
          ri.len = sg.len;
          ri.lo = static_cast<uint8_t>(row);
          ri.hi = static_cast<uint8_t>(row + sg.len);
          for (int i = 0; i < sg.len; ++i) pack_rows.push_back(ri);
          row += sg.len;
        }
        pack_rows.resize(pack_rows.size() + (kBM - tokens), RowInfo{});
        pack_segs.push_back(pk);
      }
      s0 = s1;
    }
    p->n_packs = static_cast<int64_t>(pack_segs.size());
    {
      std::vector<char> listed(pack_segs.size(), 0);
      for (const int s : order) {
        if (p->seg[s].len == 0) break;  // empty segments come last
        if (pack_of[s] >= 0) {
          if (listed[pack_of[s] - n_seg]) continue;
          listed[pack_of[s] - n_seg] = 1;
        }
        const SegInfo& sg = p->seg[s];
        for (int g = 0; g < sg.hkv; ++g)
          bwd_first.push_back(nsp_tile_t{pack_of[s] >= 0 ? pack_of[s] : s, g, 0, sg.hq / sg.hkv});
      }
    }
    p->n_first = static_cast<int64_t>(bwd_first.size());
    for (const SegInfo& sg : p->seg) {
      const int64_t Mt = (static_cast<int64_t>(sg.len) + bm - 1) / bm;
      bwd_steps += sg.hq * (Mt * (Mt + 1) / 2);
      if (Mt > 1) p->n_pairs += (sg.hq / sg.hkv) % 2 == 0 ? sg.hq / 2 * (Mt - 1) : sg.hq * (Mt / 2);
    }
    for (const SegInfo& sg : p->seg) p->max_len = std::max(p->max_len, sg.len);
  } catch (...) {
    delete p;
    return NSP_ERR_ALLOC;
  }

  // ---- device side
  int major = 0;
  if (cudaGetDevice(&p->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&p->num_sms, cudaDevAttrMultiProcessorCount, p->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, p->device) != cudaSuccess) {
    delete p;
    return NSP_ERR_CUDA;
  }
  p->small_bwd = bwd_steps <= static_cast<int64_t>(kSmallBwdStepsPerSm) * p->num_sms;
  if (major != 10) {
    delete p;
    return NSP_ERR_UNSUPPORTED;
  }
  // Two KV heads of one q head each as one item of the first-tile forward kernel: its two halves then both work, for a
  // little more latency per item, so only where there are more items than SMs (16q/16kv, forward: 56,657 tokens in segments
  // of about 100 423 -> 363 us, at head_dim 64 319 -> 261).
  std::vector<nsp_tile_t> fwd_first;
  if (p->n_first > p->num_sms) {
    try {
      for (const nsp_tile_t& t : bwd_first) {
        const int hkv = (t.seg < n_seg ? p->seg[t.seg] : pack_segs[t.seg - n_seg]).hkv;
        if (t.cost > 1)
          fwd_first.push_back(t);
        else if (t.head % 2 == 0)
          fwd_first.push_back(nsp_tile_t{t.seg, t.head, 0, t.head + 1 < hkv ? 2 : 1});
      }
    } catch (...) {
      delete p;
      return NSP_ERR_ALLOC;
    }
    if (fwd_first.size() == bwd_first.size()) fwd_first.clear();
  }
  std::vector<nsp_tile_t> parts, first_parts, pairs;
  std::vector<TileBase> bases;
  int32_t n_turns = 0;
  try {
    if (tiles * n_seg > kMostSumTerms) bases = plan_tile_bases(keys, order);
    if (!p->deterministic && !p->rounded_dq) {
      std::vector<WholeItem> main_items, first_items;
      int64_t main_steps = 0, first_steps = 0, pair_steps = 0, longest_left = 0;
      size_t paired = 0;  // segments, in the order of their lengths, whose items run on CTA pairs
      if (head_dim == 128 && !p->small_bwd) {
        int64_t steps = 0, longest = 0;
        for (; paired < order.size(); ++paired) {
          const SegInfo& sg = p->seg[order[paired]];
          const int32_t Mt = (sg.len + bm - 1) / bm, G = sg.hq / sg.hkv;
          if (Mt < kPairTiles || G * Mt < kPairSteps) break;
          for (int g = 0; g < sg.hkv; ++g)
            for (int32_t n = 0; n < Mt; n += 2) {
              pairs.push_back(nsp_tile_t{order[paired], g, n / 2, G * (Mt - std::max(n, 1))});
              steps += pairs.back().cost;
              longest = std::max<int64_t>(longest, pairs.back().cost);
            }
          p->n_bwd_paired += static_cast<int64_t>(sg.hkv) * Mt;
        }
        // Not where the longest item would bound the kernel, nor where other segments have more than a quarter of the steps:
        // the two launches each have a tail. Backward pass, ms, pairs / single CTAs: 131,072 tokens around 432 at 32q/4kv, its
        // segments of 2,048 tokens and more on pairs, 6.15 / 6.01; 65,536 around 1,024 (nearly all steps) 12.3 / 13.05.
        if (longest * (p->num_sms / 2) > steps || 8 * steps < 3 * bwd_steps) {
          paired = 0;
          p->n_bwd_paired = 0;
          pairs.clear();
        }
        pair_steps = steps;
      }
      for (size_t at = paired; at < order.size(); ++at) {
        const int s = order[at];
        const SegInfo& sg = p->seg[s];
        const int32_t Mt = (sg.len + bm - 1) / bm, G = sg.hq / sg.hkv;
        for (int g = 0; g < sg.hkv; ++g)
          for (int32_t n = 0; n < Mt; ++n) {
            const int32_t steps = G * (Mt - std::max(n, 1));
            if (steps > 0) main_items.push_back(WholeItem{s, g, n, steps});
            main_steps += steps;
            longest_left = std::max<int64_t>(longest_left, steps);
          }
      }
      p->pairs_bf16 = !pairs.empty() && kPairRest * longest_left * p->num_sms <= 2 * pair_steps;
      for (const nsp_tile_t& t : bwd_first) {
        first_items.push_back(WholeItem{t.seg, t.head, 0, t.cost});
        first_steps += t.cost;
      }
      parts = divide_items(main_items, std::max<int64_t>(kMinPart, main_steps / p->num_sms),
                           q_off * 4 <= kMostByLength, &n_turns);
      first_parts = divide_items(first_items, std::max<int64_t>(kMinFirstPart, (first_steps + main_steps) / (2 * p->num_sms)), true,
                                 &n_turns);
      if (!pairs.empty() && static_cast<int64_t>(first_parts.size()) > p->num_sms) first_parts.clear();
    }
    p->n_bwd_pairs = static_cast<int64_t>(pairs.size());
    p->n_parts = static_cast<int64_t>(parts.size());
    p->n_first_parts = static_cast<int64_t>(first_parts.size());
  } catch (...) {
    delete p;
    return NSP_ERR_ALLOC;
  }
  // Layout of the arena's device block: what the host uploads (counters and status first, all zero), then the lists the
  // device builds and the start-alignment counters. The pinned host block holds the host's copy of the status record
  // and, behind it, the image of the upload. A block that no later plan will use is not worth pinning: cudaHostAlloc
  // of 4 MB takes 3-5 ms, of 16 MB 7-18. The image of a plan that is too large to be kept is ordinary memory (65,535 segments
  // of 16 tokens at 32q/4kv 55 -> 29 ms, of 1,024 tokens at 4q/1kv 41 -> 16 ms).
  size_t at = 0;
  auto take = [&](size_t bytes) {
    const size_t here = at;
    at += align_up(bytes, 256);
    return here;
  };
  const size_t o_counters = take(16 * sizeof(int32_t));
  const size_t o_seg = take(sizeof(SegInfo) * (n_seg + pack_segs.size()));
  const size_t o_rows = take(sizeof(RowInfo) * pack_rows.size());
  const size_t o_row_base = take(sizeof(int64_t) * (n_seg + 1));
  const size_t o_first = take(sizeof(nsp_tile_t) * p->n_first);
  const size_t o_keys = take(sizeof(PlanKey) * n_seg);
  const size_t o_tiles = take(sizeof(int32_t) * (n_seg + 1));
  const size_t o_parts = take(sizeof(nsp_tile_t) * parts.size());
  const size_t o_first_parts = take(sizeof(nsp_tile_t) * first_parts.size());
  const size_t o_bwd_pairs = take(sizeof(nsp_tile_t) * pairs.size());
  const size_t o_fwd_first = take(sizeof(nsp_tile_t) * fwd_first.size());
  const size_t o_turns = take(sizeof(int32_t) * n_turns);
  const size_t o_bases = take(sizeof(TileBase) * bases.size());
  const size_t upload = at;
  const size_t o_fwd = take(sizeof(nsp_tile_t) * nf);
  const size_t o_bwd = take(sizeof(nsp_tile_t) * nb);
  const size_t o_exec = take(sizeof(nsp_tile_t) * nb);
  const size_t o_pairs = take(sizeof(nsp_tile_t) * 2 * p->n_pairs);
  const size_t o_front = take(sizeof(int32_t) * (nb / kFrontBlock + 1 + pairs.size() / kFrontBlock + 1));
  const bool pinned = arena_keeps(at, 256 + upload);
  std::vector<char> pageable;
  try {
    if (!pinned) pageable.resize(upload);
  } catch (...) {
    delete p;
    return NSP_ERR_ALLOC;
  }
  p->arena = arena_acquire(p->device, at, pinned ? 256 + upload : 256, static_cast<cudaStream_t>(stream));
  if (!p->arena) {
    delete p;
    return NSP_ERR_ALLOC;
  }
  char* const d = static_cast<char*>(p->arena->dev);
  p->d_counters = reinterpret_cast<int32_t*>(d + o_counters);  // [0] forward, [1] backward main, [2] first-tile backward, [3] first-tile forward, [8] pairs
  p->d_status = p->d_counters + 4;
  p->d_seg = reinterpret_cast<SegInfo*>(d + o_seg);
  p->d_rows = reinterpret_cast<RowInfo*>(d + o_rows);
  p->d_row_base = reinterpret_cast<int64_t*>(d + o_row_base);
  p->d_bwd_first = reinterpret_cast<nsp_tile_t*>(d + o_first);
  p->d_fwd = reinterpret_cast<nsp_tile_t*>(d + o_fwd);
  p->d_bwd = reinterpret_cast<nsp_tile_t*>(d + o_bwd);
  p->d_bwd_exec = reinterpret_cast<nsp_tile_t*>(d + o_exec);
  p->d_fwd_pairs = reinterpret_cast<nsp_tile_t*>(d + o_pairs);
  p->d_front = reinterpret_cast<int32_t*>(d + o_front);
  p->d_bwd_parts = reinterpret_cast<nsp_tile_t*>(d + o_parts);
  p->d_bwd_first_parts = reinterpret_cast<nsp_tile_t*>(d + o_first_parts);
  p->d_bwd_pairs = reinterpret_cast<nsp_tile_t*>(d + o_bwd_pairs);
  p->d_turns = reinterpret_cast<int32_t*>(d + o_turns);
  p->d_fwd_first = fwd_first.empty() ? p->d_bwd_first : reinterpret_cast<nsp_tile_t*>(d + o_fwd_first);
  p->n_fwd_first = fwd_first.empty() ? p->n_first : static_cast<int64_t>(fwd_first.size());
  p->h_status = static_cast<int32_t*>(p->arena->host);
  p->h_status_dev = reinterpret_cast<int32_t*>(p->arena->host_dev);
  char* const image = pinned ? static_cast<char*>(p->arena->host) + 256 : pageable.data();
  auto put = [&](size_t off, const void* src, size_t bytes) {
    if (bytes) std::memcpy(image + off, src, bytes);
  };
  std::memset(p->h_status, 0, 256);
  std::memset(image, 0, 16 * sizeof(int32_t));
  put(o_seg, p->seg.data(), sizeof(SegInfo) * n_seg);
  put(o_seg + sizeof(SegInfo) * n_seg, pack_segs.data(), sizeof(SegInfo) * pack_segs.size());
  put(o_rows, pack_rows.data(), sizeof(RowInfo) * pack_rows.size());
  put(o_row_base, row_base.data(), sizeof(int64_t) * (n_seg + 1));
  put(o_first, bwd_first.data(), sizeof(nsp_tile_t) * p->n_first);
  put(o_keys, keys.data(), sizeof(PlanKey) * n_seg);
  put(o_tiles, tile_base.data(), sizeof(int32_t) * (n_seg + 1));
  put(o_parts, parts.data(), sizeof(nsp_tile_t) * parts.size());
  put(o_first_parts, first_parts.data(), sizeof(nsp_tile_t) * first_parts.size());
  put(o_bwd_pairs, pairs.data(), sizeof(nsp_tile_t) * pairs.size());
  put(o_fwd_first, fwd_first.data(), sizeof(nsp_tile_t) * fwd_first.size());
  std::memset(image + o_turns, 0, sizeof(int32_t) * n_turns);
  put(o_bases, bases.data(), sizeof(TileBase) * bases.size());
  // On the arena's own stream: nothing here depends on the caller's work. It takes ~20 us where an SM has room for a block of
  // the list kernel. A backward kernel leaves none (its shared memory, at head_dim 64 its registers), and then the lists
  // are ready when one of its CTAs ends: waited for here, the host stood still for up to the rest of a running backward
  // pass (13 ms, four segments of 16,384 tokens at 32q/4kv, head_dim 64). So the host looks for kBuildPoll and then leaves the
  // waiting to the streams that use the plan. Plans that are ready at once save those a dependency in front of their first
  // kernel.
  constexpr auto kBuildPoll = std::chrono::microseconds(40);
  cudaStream_t bs = p->arena->build;
  const bool enqueued =
      cudaMemcpyAsync(d, image, upload, cudaMemcpyHostToDevice, bs) == cudaSuccess &&
      (pinned || cudaStreamSynchronize(bs) == cudaSuccess) &&
      launch_plan_lists(reinterpret_cast<const PlanKey*>(d + o_keys), reinterpret_cast<const int32_t*>(d + o_tiles),
                        bases.empty() ? nullptr : reinterpret_cast<const TileBase*>(d + o_bases), n_seg, static_cast<int>(tiles),
                        p->d_fwd, p->d_bwd, p->d_bwd_exec, p->d_fwd_pairs, bs) == cudaSuccess;
  arena_used(p->arena, bs);
  if (!enqueued || p->arena->n_uses != 1) {
    p->arena->unpooled = true;
    free_plan(p);
    return NSP_ERR_CUDA;
  }
  const auto begun = std::chrono::steady_clock::now();
  bool built = false;
  while (!(built = arena_built(p->arena)) && std::chrono::steady_clock::now() - begun < kBuildPoll) {}
  p->built.store(built, std::memory_order_release);
  NSP_LOGF("plan %p: %d segments, %zu runs, head_dim %d, q_elems %lld, kv_elems %lld, fwd items %lld, bwd items %lld%s",
           static_cast<void*>(p), n_seg, p->runs.size(), head_dim, static_cast<long long>(p->q_elems),
           static_cast<long long>(p->kv_elems), static_cast<long long>(nf), static_cast<long long>(nb),
           p->deterministic ? ", deterministic dQ" : "");
  *out_plan = p;
  return NSP_OK;
}

int nsp_plan_sizes(const nsp_plan_t* plan, int64_t* q_elems, int64_t* kv_elems, int64_t* lse_elems,
                   size_t* fwd_ws_bytes, size_t* bwd_ws_bytes) {
  if (!plan) return NSP_ERR_INVALID_ARG;
  if (q_elems) *q_elems = plan->q_elems;
  if (kv_elems) *kv_elems = plan->kv_elems;
  if (lse_elems) *lse_elems = plan->lse_elems;
  if (fwd_ws_bytes) *fwd_ws_bytes = 0;
  if (bwd_ws_bytes)  // fp32 dQ accumulator, delta, and (deterministic dQ) one turn counter per (q head, q tile)
    *bwd_ws_bytes = align_up(static_cast<size_t>(plan->q_elems) * 4, 256) +
                    align_up(static_cast<size_t>(plan->lse_elems) * 4, 256) +
                    (plan->deterministic ? align_up(static_cast<size_t>(plan->n_fwd) * 4, 256) : 0);
  return NSP_OK;
}

int nsp_plan_get(const nsp_plan_t* plan, int pass, nsp_tile_t* host_out, int64_t cap, int64_t* n_items) {
  if (!plan || !n_items || pass < 0 || pass > 2 || cap < 0) return NSP_ERR_INVALID_ARG;
  const int64_t n = pass == 0 ? plan->n_fwd : plan->n_bwd;
  *n_items = n;
  if (!host_out || cap == 0 || n == 0) return NSP_OK;
  const int64_t m = cap < n ? cap : n;
  if (!plan->built.load(std::memory_order_acquire) && arena_wait_built(plan->arena) != cudaSuccess) return NSP_ERR_CUDA;
  const nsp_tile_t* src = pass == 0 ? plan->d_fwd : (pass == 1 ? plan->d_bwd : plan->d_bwd_exec);
  if (cudaMemcpy(host_out, src, sizeof(nsp_tile_t) * m, cudaMemcpyDeviceToHost) !=
      cudaSuccess)
    return NSP_ERR_CUDA;
  return NSP_OK;
}

int nsp_plan_pair_items(const nsp_plan_t* plan, int dkv_dtype, int64_t* n_pairs, int64_t* n_left) {
  if (!plan || (dkv_dtype != NSP_BF16 && dkv_dtype != NSP_F32)) return NSP_ERR_INVALID_ARG;
  const bool paired = runs_on_pairs(plan, dkv_dtype);
  if (n_pairs) *n_pairs = paired ? plan->n_bwd_pairs : 0;
  if (n_left) *n_left = paired ? plan->n_bwd - plan->n_bwd_paired : plan->n_bwd;
  return NSP_OK;
}

int nsp_attn_fwd(const nsp_plan_t* plan, const void* q, const void* k, const void* v, void* o, float* lse,
                 float softmax_scale, void* ws, size_t ws_bytes, void* stream) {
  (void)ws;
  (void)ws_bytes;
  if (!plan) return NSP_ERR_INVALID_ARG;
  if (const int failed = plan_failed(plan)) return failed;
  if (!(softmax_scale > 0.f) || !std::isfinite(softmax_scale)) return NSP_ERR_INVALID_ARG;
  if (plan->n_fwd == 0) return NSP_OK;
  if (!q || !k || !v || !o || !lse) return NSP_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o) || !aligned16(lse)) return NSP_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const UsesArena uses(plan, st);
  if (uses.ready != cudaSuccess) return NSP_ERR_CUDA;
  FwdMaps maps;
  std::memset(&maps, 0, sizeof(maps));
  for (size_t r = 0; r < plan->runs.size(); ++r) {
    const RunInfo& run = plan->runs[r];
    if (!encode_run_map(&maps.q[r], q, run.q_off, run.tokens, run.hq, plan->head_dim) ||
        !encode_run_map(&maps.k[r], k, run.kv_off, run.tokens, run.hkv, plan->head_dim) ||
        !encode_run_map(&maps.v[r], v, run.kv_off, run.tokens, run.hkv, plan->head_dim) ||
        !encode_run_map(&maps.o[r], o, run.q_off, run.tokens, run.hq, plan->head_dim))
      return NSP_ERR_CUDA;
  }
  FwdArgs a;
  a.seg = plan->d_seg;
  a.status = status_word(plan);
  a.o = static_cast<__nv_bfloat16*>(o);
  a.lse = lse;
  a.scale_log2 = softmax_scale * 1.4426950408889634f;
  a.wait_limit = plan->wait_limit;
  a.withhold = plan->withhold;
  a.q_elems = plan->q_elems;
  a.lse_elems = plan->lse_elems;
  a.seg_mask = nullptr;
  a.rows = plan->d_rows;
  a.d_o = nullptr;
  a.delta = nullptr;
  NSP_LOGF("fwd plan %p stream %p scale %g", static_cast<const void*>(plan), stream, softmax_scale);
  // q tile 0 of every segment (the cost-1 tail of the list): one item per (segment, kv head)
  a.pairs = plan->d_fwd_first != plan->d_bwd_first;
  a.items = plan->d_fwd_first;
  a.n_items = static_cast<int32_t>(plan->n_fwd_first);
  a.counter = plan->d_counters + 3;
  prof_mark(plan, NSP_KERNEL_FWD_FIRST, 0, st);
  if (!plan->withhold && launch_fwd_first(maps, a, plan->head_dim, plan->num_sms, st) != cudaSuccess) return NSP_ERR_CUDA;
  prof_mark(plan, NSP_KERNEL_FWD_FIRST, 1, st);
  // everything else, in pairs (with the test switch of the checked build: the whole list, general kernel)
  a.items = plan->withhold ? plan->d_fwd : plan->d_fwd_pairs;
  a.n_items = static_cast<int32_t>(plan->withhold ? plan->n_fwd : 2 * plan->n_pairs);
  a.counter = plan->d_counters;
  prof_mark(plan, NSP_KERNEL_FWD, 0, st);
  if (launch_fwd(maps, a, plan->head_dim, plan->num_sms, !plan->withhold, st) != cudaSuccess) return NSP_ERR_CUDA;
  prof_mark(plan, NSP_KERNEL_FWD, 1, st);
  return NSP_OK;
}

namespace {

size_t recompute_ws_bytes(const nsp_plan_t* plan) {
  size_t base = 0;
  nsp_plan_sizes(plan, nullptr, nullptr, nullptr, nullptr, &base);
  return base + align_up(static_cast<size_t>(plan->lse_elems) * 4, 256) + align_up(static_cast<size_t>(plan->n_seg), 256);
}

// Backward pass. recompute == nullptr: the plain pass. Otherwise host flags per segment: for a marked segment o and
// lse are not read; its LSE and delta are recomputed by a forward launch restricted to the marked segments.
int bwd_impl(const nsp_plan_t* plan, const uint8_t* recompute, const void* q, const void* k, const void* v,
             const void* o, const void* d_o, const float* lse, void* dq, void* dk, void* dv, int dq_dtype,
             int dkv_dtype, float softmax_scale, void* ws, size_t ws_bytes, void* stream) {
  if (!plan) return NSP_ERR_INVALID_ARG;
  if (const int failed = plan_failed(plan)) return failed;
  if (!(softmax_scale > 0.f) || !std::isfinite(softmax_scale)) return NSP_ERR_INVALID_ARG;
  if ((dq_dtype != NSP_BF16 && dq_dtype != NSP_F32) || (dkv_dtype != NSP_BF16 && dkv_dtype != NSP_F32))
    return NSP_ERR_INVALID_ARG;
  if (plan->n_bwd == 0) return NSP_OK;
  if (!q || !k || !v || !o || !d_o || !lse || !dq || !dk || !dv) return NSP_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o) || !aligned16(d_o) || !aligned16(lse) ||
      !aligned16(dq) || !aligned16(dk) || !aligned16(dv))
    return NSP_ERR_INVALID_ARG;
  size_t base = 0;
  nsp_plan_sizes(plan, nullptr, nullptr, nullptr, nullptr, &base);
  const size_t need = recompute ? recompute_ws_bytes(plan) : base;
  if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255) != 0 || ws_bytes < need) return NSP_ERR_WORKSPACE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const UsesArena uses(plan, st);
  if (uses.ready != cudaSuccess) return NSP_ERR_CUDA;
  char* wsb = static_cast<char*>(ws);
  float* dq_acc = static_cast<float*>(ws);
  float* delta = reinterpret_cast<float*>(wsb + align_up(static_cast<size_t>(plan->q_elems) * 4, 256));
  int32_t* dq_turn = plan->deterministic
                         ? reinterpret_cast<int32_t*>(wsb + align_up(static_cast<size_t>(plan->q_elems) * 4, 256) +
                                                      align_up(static_cast<size_t>(plan->lse_elems) * 4, 256))
                         : nullptr;
  float* lse_ws = reinterpret_cast<float*>(wsb + base);
  uint8_t* d_mask = reinterpret_cast<uint8_t*>(wsb + base + align_up(static_cast<size_t>(plan->lse_elems) * 4, 256));

  BwdMaps maps;
  std::memset(&maps, 0, sizeof(maps));
  FwdMaps fmaps;
  if (recompute) std::memset(&fmaps, 0, sizeof(fmaps));
  for (size_t r = 0; r < plan->runs.size(); ++r) {
    const RunInfo& run = plan->runs[r];
    if (!encode_run_map(&maps.q[r], q, run.q_off, run.tokens, run.hq, plan->head_dim) ||
        !encode_run_map(&maps.d_o[r], d_o, run.q_off, run.tokens, run.hq, plan->head_dim) ||
        !encode_run_map(&maps.k[r], k, run.kv_off, run.tokens, run.hkv, plan->head_dim) ||
        !encode_run_map(&maps.v[r], v, run.kv_off, run.tokens, run.hkv, plan->head_dim))
      return NSP_ERR_CUDA;
    if (dkv_dtype == NSP_F32 && (!encode_run_map_f32(&maps.dk[r], dk, run.kv_off, run.tokens, run.hkv, plan->head_dim) ||
                                 !encode_run_map_f32(&maps.dv[r], dv, run.kv_off, run.tokens, run.hkv, plan->head_dim)))
      return NSP_ERR_CUDA;
    if (recompute) fmaps.q[r] = maps.q[r], fmaps.k[r] = maps.k[r], fmaps.v[r] = maps.v[r];
  }
  if (recompute) {
    // from pageable memory the runtime stages the flags before it returns; a pinned array must stay unchanged until
    // the stream has passed this copy
    if (cudaMemcpyAsync(d_mask, recompute, static_cast<size_t>(plan->n_seg), cudaMemcpyHostToDevice, st) != cudaSuccess)
      return NSP_ERR_CUDA;
    FwdArgs fa;
    fa.seg = plan->d_seg;
    fa.items = plan->d_fwd;
    fa.n_items = static_cast<int32_t>(plan->n_fwd);
    fa.counter = plan->d_counters;
    fa.status = status_word(plan);
    fa.o = nullptr;
    fa.lse = lse_ws;
    fa.scale_log2 = softmax_scale * 1.4426950408889634f;
    fa.wait_limit = plan->wait_limit;
    fa.withhold = 0;
    fa.q_elems = plan->q_elems;
    fa.lse_elems = plan->lse_elems;
    fa.seg_mask = d_mask;
    fa.rows = plan->d_rows;
    fa.pairs = 0;
    fa.d_o = static_cast<const __nv_bfloat16*>(d_o);
    fa.delta = delta;
    prof_mark(plan, NSP_KERNEL_FWD, 0, st);
    if (launch_fwd(fmaps, fa, plan->head_dim, plan->num_sms, false, st) != cudaSuccess) return NSP_ERR_CUDA;
    prof_mark(plan, NSP_KERNEL_FWD, 1, st);
  }
  // Segments of at most 128 tokens are finished by the first-tile kernel alone; a batch made only of such segments
  // needs no accumulator, no delta and no conversion pass.
  const bool multi = plan->max_len > kBM;
  NSP_LOGF("bwd plan %p stream %p scale %g%s%s", static_cast<const void*>(plan), stream, softmax_scale,
           recompute ? ", recomputing marked segments" : "", multi ? "" : ", first-tile kernel only");
  if (dq_turn && multi &&
      cudaMemsetAsync(dq_turn, 0, static_cast<size_t>(plan->n_fwd) * 4, st) != cudaSuccess)
    return NSP_ERR_CUDA;
  prof_mark(plan, NSP_KERNEL_BWD_PRE, 0, st);
  if (multi || recompute) {
    if (launch_bwd_preprocess(plan->d_seg, plan->n_seg, plan->d_row_base, plan->lse_elems, plan->head_dim,
                              static_cast<const __nv_bfloat16*>(o), static_cast<const __nv_bfloat16*>(d_o), delta,
                              dq_acc, recompute ? d_mask : nullptr, recompute ? lse : nullptr,
                              recompute ? lse_ws : nullptr, plan->d_front,
                              static_cast<int>(plan->n_bwd / kFrontBlock + 1 + plan->n_bwd_pairs / kFrontBlock + 1),
                              plan->small_bwd, st) != cudaSuccess)
      return NSP_ERR_CUDA;
  }
  prof_mark(plan, NSP_KERNEL_BWD_PRE, 1, st);
  BwdArgs a;
  a.seg = plan->d_seg;
  a.status = status_word(plan);
  a.lse = recompute ? lse_ws : lse;
  a.delta = delta;
  a.dq_acc = dq_acc;
  a.dq = dq;
  a.dq_f32 = dq_dtype == NSP_F32;
  a.dq_turn = dq_turn;
  a.dq_rounded = plan->rounded_dq ? 1 : 0;
  a.front = plan->d_front;
  a.rows = plan->d_rows;
  a.dk = dk;
  a.dv = dv;
  a.dkv_f32 = dkv_dtype == NSP_F32;
  a.scale = softmax_scale;
  a.scale_log2 = softmax_scale * 1.4426950408889634f;
  a.wait_limit = plan->wait_limit;
  a.q_elems = plan->q_elems;
  a.kv_elems = plan->kv_elems;
  a.lse_elems = plan->lse_elems;
  a.withhold = plan->withhold_pair;
  // first-tile kernel: q tile 0 of every segment (its dQ rows; its part of, or all of, dK / dV rows 0..127)
  const bool f_parts = a.dkv_f32 && plan->n_first_parts > 0;  // bf16 gradients are not added up piece by piece
  a.items = f_parts ? plan->d_bwd_first_parts : plan->d_bwd_first;
  a.n_items = static_cast<int32_t>(f_parts ? plan->n_first_parts : plan->n_first);
  a.turn = f_parts ? plan->d_turns : nullptr;
  a.counter = plan->d_counters + 2;
  prof_mark(plan, NSP_KERNEL_BWD_FIRST, 0, st);
  if (launch_bwd_first(maps, a, plan->head_dim, plan->num_sms, st) != cudaSuccess) return NSP_ERR_CUDA;
  prof_mark(plan, NSP_KERNEL_BWD_FIRST, 1, st);
  // main kernels: everything else, the long segments on CTA pairs
  prof_mark(plan, NSP_KERNEL_BWD_MAIN, 0, st);
  a.turn = nullptr;
  const bool paired = runs_on_pairs(plan, dkv_dtype);
  if (paired) {
    BwdPairMaps pair_maps;
    std::memset(&pair_maps, 0, sizeof(pair_maps));
    static_cast<BwdMaps&>(pair_maps) = maps;
    for (size_t r = 0; r < plan->runs.size(); ++r) {
      const RunInfo& run = plan->runs[r];
      if (!encode_run_map(&pair_maps.q[r], q, run.q_off, run.tokens, run.hq, plan->head_dim, 64) ||
          !encode_run_map(&pair_maps.d_o[r], d_o, run.q_off, run.tokens, run.hq, plan->head_dim, 64) ||
          !encode_run_map_f32(&pair_maps.dq_acc[r], dq_acc, run.q_off, run.tokens, run.hq, plan->head_dim, 16, false))
        return NSP_ERR_CUDA;
    }
    a.items = plan->d_bwd_pairs;
    a.n_items = static_cast<int32_t>(plan->n_bwd_pairs);
    a.counter = plan->d_counters + 8;
    a.front = plan->d_front + plan->n_bwd / kFrontBlock + 1;
    if (launch_bwd_pair(pair_maps, a, plan->num_sms, st) != cudaSuccess) return NSP_ERR_CUDA;
    a.front = plan->d_front;
  }
  const bool m_parts = a.dkv_f32 && plan->n_parts > 0;
  const int64_t done = paired ? plan->n_bwd_paired : 0;
  a.items = m_parts ? plan->d_bwd_parts : plan->d_bwd_exec + done;
  a.n_items = static_cast<int32_t>(m_parts ? plan->n_parts : plan->n_bwd - done);
  a.turn = m_parts ? plan->d_turns : nullptr;
  a.counter = plan->d_counters + 1;
  if (multi && launch_bwd(maps, a, plan->head_dim, plan->num_sms, plan->small_bwd, st) != cudaSuccess) return NSP_ERR_CUDA;
  prof_mark(plan, NSP_KERNEL_BWD_MAIN, 1, st);
  prof_mark(plan, NSP_KERNEL_BWD_POST, 0, st);
  if (multi && launch_bwd_postprocess(plan->d_seg, plan->n_seg, plan->d_row_base, plan->lse_elems, plan->head_dim, dq_acc, dq,
                                      dq_dtype == NSP_F32, softmax_scale, st) != cudaSuccess)
    return NSP_ERR_CUDA;
  prof_mark(plan, NSP_KERNEL_BWD_POST, 1, st);
  return NSP_OK;
}

}  // namespace

int nsp_attn_bwd(const nsp_plan_t* plan, const void* q, const void* k, const void* v, const void* o, const void* d_o,
                 const float* lse, void* dq, void* dk, void* dv, int dq_dtype, int dkv_dtype, float softmax_scale,
                 void* ws, size_t ws_bytes, void* stream) {
  return bwd_impl(plan, nullptr, q, k, v, o, d_o, lse, dq, dk, dv, dq_dtype, dkv_dtype, softmax_scale, ws, ws_bytes,
                  stream);
}

namespace {

// Device layout of the host-to-host step's workspace: the nine packed tensors, then the backward workspace.
struct HostStepLayout {
  size_t q, k, v, d_o, o, lse, dq, dk, dv, bwd_ws, total;
  size_t q_bytes, kv_bytes, lse_bytes, dq_bytes, dkv_bytes, bwd_ws_bytes;
};

bool host_step_layout(const nsp_plan_t* plan, int dq_dtype, int dkv_dtype, HostStepLayout* L) {
  if ((dq_dtype != NSP_BF16 && dq_dtype != NSP_F32) || (dkv_dtype != NSP_BF16 && dkv_dtype != NSP_F32)) return false;
  size_t bwd_ws = 0;
  nsp_plan_sizes(plan, nullptr, nullptr, nullptr, nullptr, &bwd_ws);
  L->q_bytes = static_cast<size_t>(plan->q_elems) * 2;
  L->kv_bytes = static_cast<size_t>(plan->kv_elems) * 2;
  L->lse_bytes = static_cast<size_t>(plan->lse_elems) * 4;
  L->dq_bytes = static_cast<size_t>(plan->q_elems) * (dq_dtype == NSP_F32 ? 4 : 2);
  L->dkv_bytes = static_cast<size_t>(plan->kv_elems) * (dkv_dtype == NSP_F32 ? 4 : 2);
  L->bwd_ws_bytes = bwd_ws;
  size_t at = 0;
  auto take = [&](size_t bytes) {
    const size_t here = at;
    at += align_up(bytes > 0 ? bytes : 1, 256);
    return here;
  };
  L->q = take(L->q_bytes), L->k = take(L->kv_bytes), L->v = take(L->kv_bytes), L->d_o = take(L->q_bytes);
  L->o = take(L->q_bytes), L->lse = take(L->lse_bytes);
  L->dq = take(L->dq_bytes), L->dk = take(L->dkv_bytes), L->dv = take(L->dkv_bytes);
  L->bwd_ws = take(bwd_ws);
  L->total = at;
  return true;
}

}  // namespace

int nsp_plan_step_host_ws_bytes(const nsp_plan_t* plan, int dq_dtype, int dkv_dtype, size_t* bytes) {
  if (!plan || !bytes) return NSP_ERR_INVALID_ARG;
  HostStepLayout L;
  if (!host_step_layout(plan, dq_dtype, dkv_dtype, &L)) return NSP_ERR_INVALID_ARG;
  *bytes = L.total;
  return NSP_OK;
}

int nsp_attn_step_host(nsp_plan_t* plan, const void* h_q, const void* h_k, const void* h_v, const void* h_do, void* h_o,
                       float* h_lse, void* h_dq, void* h_dk, void* h_dv, int dq_dtype, int dkv_dtype,
                       float softmax_scale, void* dev_ws, size_t dev_ws_bytes, void* stream) {
  if (!plan) return NSP_ERR_INVALID_ARG;
  if (const int failed = plan_failed(plan)) return failed;
  HostStepLayout L;
  if (!host_step_layout(plan, dq_dtype, dkv_dtype, &L)) return NSP_ERR_INVALID_ARG;
  if (plan->n_fwd == 0) return NSP_OK;
  if (!h_q || !h_k || !h_v || !h_do || !h_o || !h_lse || !h_dq || !h_dk || !h_dv) return NSP_ERR_INVALID_ARG;
  if (!dev_ws || (reinterpret_cast<uintptr_t>(dev_ws) & 255) != 0 || dev_ws_bytes < L.total) return NSP_ERR_WORKSPACE;
  if (!plan->copy_stream) {
    if (cudaStreamCreateWithFlags(&plan->copy_stream, cudaStreamNonBlocking) != cudaSuccess) return NSP_ERR_CUDA;
    for (cudaEvent_t& e : plan->hev)
      if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) return NSP_ERR_CUDA;
  }
  cudaStream_t comp = static_cast<cudaStream_t>(stream), cp = plan->copy_stream;
  char* base = static_cast<char*>(dev_ws);
  enum { kFree = 0, kQkvIn, kDoIn, kFwdDone, kBwdDone, kAllOut };
  auto ok = [](cudaError_t e) { return e == cudaSuccess; };
  const cudaMemcpyKind in = cudaMemcpyHostToDevice, out = cudaMemcpyDeviceToHost;
  NSP_LOGF("host step plan %p stream %p: %zu bytes in, %zu bytes out", static_cast<const void*>(plan), stream,
           2 * L.q_bytes + 2 * L.kv_bytes, L.q_bytes + L.lse_bytes + L.dq_bytes + 2 * L.dkv_bytes);
  // the device buffers are free once everything enqueued on the caller's stream so far has run
  if (!ok(cudaEventRecord(plan->hev[kFree], comp)) || !ok(cudaStreamWaitEvent(cp, plan->hev[kFree], 0))) return NSP_ERR_CUDA;
  if (!ok(cudaMemcpyAsync(base + L.q, h_q, L.q_bytes, in, cp)) || !ok(cudaMemcpyAsync(base + L.k, h_k, L.kv_bytes, in, cp)) ||
      !ok(cudaMemcpyAsync(base + L.v, h_v, L.kv_bytes, in, cp)) || !ok(cudaEventRecord(plan->hev[kQkvIn], cp)))
    return NSP_ERR_CUDA;
  // dO travels in under the forward pass
  if (!ok(cudaMemcpyAsync(base + L.d_o, h_do, L.q_bytes, in, cp)) || !ok(cudaEventRecord(plan->hev[kDoIn], cp)))
    return NSP_ERR_CUDA;
  if (!ok(cudaStreamWaitEvent(comp, plan->hev[kQkvIn], 0))) return NSP_ERR_CUDA;
  int rc = nsp_attn_fwd(plan, base + L.q, base + L.k, base + L.v, base + L.o, reinterpret_cast<float*>(base + L.lse),
                        softmax_scale, nullptr, 0, stream);
  if (rc != NSP_OK) return rc;
  // O and LSE travel out under the backward pass
  if (!ok(cudaEventRecord(plan->hev[kFwdDone], comp)) || !ok(cudaStreamWaitEvent(cp, plan->hev[kFwdDone], 0)) ||
      !ok(cudaMemcpyAsync(h_o, base + L.o, L.q_bytes, out, cp)) || !ok(cudaMemcpyAsync(h_lse, base + L.lse, L.lse_bytes, out, cp)))
    return NSP_ERR_CUDA;
  if (!ok(cudaStreamWaitEvent(comp, plan->hev[kDoIn], 0))) return NSP_ERR_CUDA;
  rc = nsp_attn_bwd(plan, base + L.q, base + L.k, base + L.v, base + L.o, base + L.d_o,
                    reinterpret_cast<const float*>(base + L.lse), base + L.dq, base + L.dk, base + L.dv, dq_dtype, dkv_dtype,
                    softmax_scale, base + L.bwd_ws, L.bwd_ws_bytes, stream);
  if (rc != NSP_OK) return rc;
  if (!ok(cudaEventRecord(plan->hev[kBwdDone], comp)) || !ok(cudaStreamWaitEvent(cp, plan->hev[kBwdDone], 0)) ||
      !ok(cudaMemcpyAsync(h_dq, base + L.dq, L.dq_bytes, out, cp)) || !ok(cudaMemcpyAsync(h_dk, base + L.dk, L.dkv_bytes, out, cp)) ||
      !ok(cudaMemcpyAsync(h_dv, base + L.dv, L.dkv_bytes, out, cp)) || !ok(cudaEventRecord(plan->hev[kAllOut], cp)) ||
      !ok(cudaStreamWaitEvent(comp, plan->hev[kAllOut], 0)))  // the step is complete on the caller's stream
    return NSP_ERR_CUDA;
  return NSP_OK;
}

int nsp_plan_recompute_ws_bytes(const nsp_plan_t* plan, size_t* bytes) {
  if (!plan || !bytes) return NSP_ERR_INVALID_ARG;
  *bytes = recompute_ws_bytes(plan);
  return NSP_OK;
}

int nsp_attn_bwd_recompute(const nsp_plan_t* plan, const uint8_t* recompute, const void* q, const void* k,
                           const void* v, const void* o, const void* d_o, const float* lse, void* dq, void* dk,
                           void* dv, int dq_dtype, int dkv_dtype, float softmax_scale, void* ws, size_t ws_bytes,
                           void* stream) {
  if (!plan || !recompute) return NSP_ERR_INVALID_ARG;
  return bwd_impl(plan, recompute, q, k, v, o, d_o, lse, dq, dk, dv, dq_dtype, dkv_dtype, softmax_scale, ws, ws_bytes,
                  stream);
}

int nsp_recompute_mark(const int32_t* cu_seqlens, const int32_t* hq, const int32_t* level, int32_t n_seg,
                       int32_t head_dim, int64_t budget_bytes, uint8_t* recompute, int64_t* saved_bytes) {
  if (n_seg < 0 || head_dim <= 0 || budget_bytes < 0) return NSP_ERR_INVALID_ARG;
  if (n_seg > 0 && (!cu_seqlens || !hq || !level || !recompute)) return NSP_ERR_INVALID_ARG;
  for (int s = 0; s < n_seg; ++s)
    if (cu_seqlens[s + 1] < cu_seqlens[s] || hq[s] <= 0) return NSP_ERR_INVALID_ARG;
  std::vector<int> order(n_seg);
  for (int s = 0; s < n_seg; ++s) order[s] = s;
  auto len = [&](int s) { return static_cast<int64_t>(cu_seqlens[s + 1]) - cu_seqlens[s]; };
  // recomputation cost of a segment: its causal (query, key) pairs times its query heads
  auto cost = [&](int s) { return static_cast<int64_t>(hq[s]) * (len(s) * (len(s) + 1) / 2); };
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
    if (level[x] != level[y]) return level[x] > level[y];
    return cost(x) > cost(y);
  });
  int64_t used = 0;
  bool cut = false;
  for (int s : order) {
    // what saving the segment keeps alive: its slice of O (bf16) and of the LSE (fp32)
    const int64_t bytes = len(s) * hq[s] * (static_cast<int64_t>(head_dim) * 2 + 4);
    if (!cut && used + bytes <= budget_bytes) {
      used += bytes;
      recompute[s] = 0;
    } else {
      cut = true;
      recompute[s] = 1;
    }
  }
  if (saved_bytes) *saved_bytes = used;
  return NSP_OK;
}

namespace {
// One warp waits on a barrier nothing ever arrives at; the bounded wait runs out after limit_clk SM cycles and the
// warp records it in the status word exactly as the attention kernels would.
__global__ void selftest_wait_kernel(StatusWord status, long long limit_clk) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  __syncwarp();
  const bool ok = mbar_wait(&bar, 0, limit_clk);
  if (!ok && threadIdx.x == 0) report_timeout(status, -1, kWhereSelfTest, static_cast<int32_t>(limit_clk >> 10));
}
}  // namespace

int nsp_selftest_wait_timeout(const nsp_plan_t* plan, int64_t limit_clk, void* stream) {
  if (!plan || limit_clk < 1 || limit_clk > (1ll << 31)) return NSP_ERR_INVALID_ARG;
  if (const int failed = plan_failed(plan)) return failed;
  const UsesArena uses(plan, static_cast<cudaStream_t>(stream));
  if (uses.ready != cudaSuccess) return NSP_ERR_CUDA;
  selftest_wait_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(status_word(plan), limit_clk);
  count_launches(1);
  return cudaGetLastError() == cudaSuccess ? NSP_OK : NSP_ERR_CUDA;
}

int nsp_device_status(const nsp_plan_t* plan, int32_t out[4]) {
  if (!plan || !out) return NSP_ERR_INVALID_ARG;
  if (cudaDeviceSynchronize() != cudaSuccess) return NSP_ERR_CUDA;
  if (cudaMemcpy(out, plan->d_status, 4 * sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess) return NSP_ERR_CUDA;
  if (out[0] != 0 && !plan->sticky) const_cast<nsp_plan_t*>(plan)->sticky = out[0];
  return NSP_OK;
}

int nsp_plan_set_wait_limit(nsp_plan_t* plan, int64_t sm_clocks) {
  if (!plan || sm_clocks < 1000) return NSP_ERR_INVALID_ARG;
  plan->wait_limit = sm_clocks;
  return NSP_OK;
}

#ifdef NSP_CHECKED
int nsp_checked_withhold_load(nsp_plan_t* plan, int enable) {
  if (!plan) return NSP_ERR_INVALID_ARG;
  plan->withhold = enable != 0;
  return NSP_OK;
}
int nsp_checked_withhold_pair_load(nsp_plan_t* plan, int load) {
  if (!plan || load < 0 || load > NSP_WITHHOLD_Q_COLUMNS) return NSP_ERR_INVALID_ARG;
  if (load != 0 && plan->n_bwd_pairs == 0) return NSP_ERR_UNSUPPORTED;
  plan->withhold_pair = load;
  return NSP_OK;
}
#endif

int nsp_plan_set_profiling(nsp_plan_t* plan, int enable) {
  if (!plan) return NSP_ERR_INVALID_ARG;
  if (enable && !plan->ev[0]) {
    for (cudaEvent_t& e : plan->ev)
      if (cudaEventCreate(&e) != cudaSuccess) return NSP_ERR_CUDA;
  }
  plan->profiling = enable != 0;
  if (!enable)
    for (bool& v : plan->ev_valid) v = false;
  return NSP_OK;
}

int nsp_plan_kernel_ms(const nsp_plan_t* plan, int kernel_id, float* ms) {
  if (!plan || !ms || kernel_id < 0 || kernel_id >= NSP_KERNEL_COUNT) return NSP_ERR_INVALID_ARG;
  if (!plan->profiling || !plan->ev_valid[kernel_id]) return NSP_ERR_INVALID_ARG;
  if (cudaEventSynchronize(plan->ev[2 * kernel_id + 1]) != cudaSuccess) return NSP_ERR_CUDA;
  if (cudaEventElapsedTime(ms, plan->ev[2 * kernel_id], plan->ev[2 * kernel_id + 1]) != cudaSuccess) return NSP_ERR_CUDA;
  return NSP_OK;
}

int nsp_trim(void) {
  arena_trim();
  return NSP_OK;
}

int nsp_plan_destroy(nsp_plan_t* plan) {
  free_plan(plan);
  return NSP_OK;
}

}  // extern "C"
