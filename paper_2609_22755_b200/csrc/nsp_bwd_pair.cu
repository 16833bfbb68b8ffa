// Backward main kernel for long segments: CTA pairs (clusters of two, tcgen05 cta_group::2), head dimension 128.
//
// A pair works on two neighbouring key tiles of one (segment, kv head): CTA r has key tile n = n0 + r, and both walk the same
// (q tile, q head) steps. Every product is a pair product: the rows (keys) of S^T, dP^T, dV, dK are the CTAs' own key tiles,
// and the B operand (Q or dO) is split between the CTAs' shared memories. dQ^T of a step contracts over the keys of BOTH
// tiles, so its reductions into the fp32 accumulator are half of what two single CTAs issue:
//     S^T  = K Q^T   -> R0        A = K [128 own keys], B = Q rows 64 r .. (64 of the 128 queries)       K-major, M = 256
//     dP^T = V dO^T  -> R1        A = V, B = dO rows 64 r ..                                             K-major, M = 256
//     dV  += P^T dO               A = P^T (bf16 over S^T in R0 [0, 64)), B = dO columns 64 r ..          M = 256
//     dK  += dS^T Q               A = dS^T (bf16 over dP^T in R1 [0, 64)), B = Q columns 64 r ..         M = 256
//     dQ^T = K^T dS^T -> R0 [64, 128)  A = K columns 64 r .. of both key tiles, B = dS^T of both key tiles for 64 of the
//                                 queries (this CTA's query set)                                         M = 128, K = 256
// For dQ^T each CTA needs the other's dS^T of its own query set: 16 KB of bf16 per step and direction through distributed
// shared memory (one bulk copy per softmax warp, under the next step).
// A step takes 3,880 active clocks, 2,570 of them of tensor pipe (ncu, 65,536 tokens at 4q/1kv beside a tail; 4,060 on single CTAs).
// What bounds it are two loops of hand-overs. One step long: dS^T 830, fence 390, copy and relay ~1,500, dQ^T ~1,000, then the dS^T
// buffers are free for the next step's: ~3,700. Two steps long, because S^T(t + 2) goes over dQ^T(t): fence, copy and relay,
// dQ^T, its drain ~800, S^T ~900, its reading 240, exponentials 1,080, dS^T: ~6,700, half of that per step. (Parts by
// clock stamps, 16 x 8,192 tokens.) Whole steps under the 1,000 W cap, single CTAs / pairs: sixteen segments of 8,192 tokens at
// 32q/4kv 33.0 / 31.2 ms, 393,216 tokens at 4q/1kv beside a tail 538.6 / 504.4.
// Query sets: softmax warpgroup w has the queries 32 w .. 32 w + 31 and 64 + 32 w .. of a tile, so that packed P^T and dS^T of
// both warpgroups go to [0, 64) of their region over columns the same thread has read, and CTA r's query set is the one of
// warpgroup r.
#include <cstddef>
#include <type_traits>
#include <cuda_bf16.h>
#include "nsp_internal.cuh"
#include "sm100_ptx.cuh"

namespace nsp {
namespace {

constexpr int D = 128;
constexpr uint32_t kHalfTileBytes = 128 * 64 * 2;  // [128 rows x 64 columns] bf16; also [64 rows x 128 columns]
constexpr int kPairThreads = 640;
constexpr uint32_t kPairTmemCols = 512;
constexpr int kRegsSoft = 136, kRegsReduce = 80, kRegsAux = 48;  // 256 * (136 + 80) + 128 * 48 = 640 * 96
constexpr float kLog2e = 1.4426950408889634f;
constexpr int kFrontMinSteps = 2048, kFrontMinGroup = 8;
constexpr long long kFrontWaitClk = 1500000;

template <int N>
__device__ __forceinline__ void pair_setmaxnreg_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void pair_setmaxnreg_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

struct PairCtx {
  int64_t q_off, kv_off, lse_off;
  int32_t it, len, hq, hkv, run, tok0;
  int32_t g, n, n0;  // kv head, this CTA's key tile, the pair's first key tile
  int32_t G, m0, per_head, steps;
};

struct PairSmem {
  uint8_t k[2][kHalfTileBytes];   // own key tile, [64-column half]
  uint8_t kt[2][kHalfTileBytes];  // both key tiles, columns 64 r .. 64 r + 63
  uint8_t v[2][kHalfTileBytes];
  uint8_t q_row[kHalfTileBytes], do_row[kHalfTileBytes];  // rows 64 r .. of the tile: two sub-tiles [64 rows x 64 columns]
  uint8_t q_col[kHalfTileBytes], do_col[kHalfTileBytes];  // columns 64 r .. of the tile: [128 rows x 64 columns]
  uint8_t x[2][kHalfTileBytes];   // dS^T of the pair's key tiles, [key][this CTA's 64 queries]
  uint8_t stage[kHalfTileBytes];  // dS^T of the own key tile for the other CTA's queries
  float dq_out[8][16][32];        // [dQ warp][query][d]: on its way into the accumulator
  alignas(16) float lse[2][128];  // [stage] LSE * log2(e) of the q tile (+inf for rows past the segment)
  float delta[2][128];
  PairCtx ctx;
  // Arrived on in the first CTA only, which issues the products: loads (both CTAs' bytes), hand-overs of both CTAs' warps
  uint64_t bar_kv, bar_qr_full, bar_qc_full, bar_dor_full, bar_doc_full;
  uint64_t bar_s_read;    // 16 warps: S^T has been read (R0 [64, 128) is free for dQ^T)
  uint64_t bar_p_ready;   // 16 warps: P^T is in R0
  uint64_t bar_ds_ready;  // 16 warps: dS^T is in R1
  uint64_t bar_dq_empty;  // 16 warps: dQ^T has been drained
  uint64_t bar_x_peer;    // 2 warps: the second CTA's dS^T buffers are complete (its own warps' part, the received one)
  // Completed in both CTAs: products
  uint64_t bar_s_full, bar_dp_full, bar_dq_full, bar_dv_done, bar_dk_done;
  // Local
  uint64_t bar_x_own;   // 4 warps: the part of dS^T that stays in this CTA is in shared memory
  uint64_t bar_x_full;  // the other CTA's part of dS^T has arrived
  uint64_t bar_ld_full[2], bar_ld_empty[2];
  uint64_t bar_out;
  uint32_t tmem_base;
  int32_t pop;
  int32_t abort;
};
static_assert(offsetof(PairSmem, lse) % 16 == 0, "16-byte loads");
static_assert(sizeof(PairSmem) <= 232448, "shared memory budget (227 KB)");

// Steps of an item: q tiles descending, heads ascending inside a q tile (see StepWalk of the single-CTA kernel for why).
struct PairWalk {
  int hh = 0, rr = 0;
  __device__ __forceinline__ void get(const PairCtx& c, int& h, int& m) const {
    h = c.g * c.G + hh;
    m = c.m0 + c.per_head - 1 - rr;
  }
  __device__ __forceinline__ void next(const PairCtx& c) {
    if (++hh == c.G) hh = 0, ++rr;
  }
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
    bwd_pair_kernel(const __grid_constant__ BwdPairMaps maps, const BwdArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  PairSmem& s = *reinterpret_cast<PairSmem*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, wg = warp >> 2;
  const uint32_t rank = cluster_rank();
  const bool misaligned = (smem_u32(smem_raw) & 1023u) != 0;
  if (tid == 0) {
    mbar_init(&s.bar_kv, 1);
    mbar_init(&s.bar_qr_full, 1);
    mbar_init(&s.bar_dor_full, 1);
    mbar_init(&s.bar_qc_full, 1);
    mbar_init(&s.bar_doc_full, 1);
    mbar_init(&s.bar_s_read, 16);
    mbar_init(&s.bar_p_ready, 16);
    mbar_init(&s.bar_ds_ready, 16);
    mbar_init(&s.bar_x_own, 4);
    mbar_init(&s.bar_dq_empty, 16);
    mbar_init(&s.bar_x_peer, 2);
    mbar_init(&s.bar_s_full, 1);
    mbar_init(&s.bar_dp_full, 1);
    mbar_init(&s.bar_dq_full, 1);
    mbar_init(&s.bar_dv_done, 1);
    mbar_init(&s.bar_dk_done, 1);
    mbar_init(&s.bar_x_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s.bar_ld_full[i], 32);
      mbar_init(&s.bar_ld_empty[i], 8);
    }
    mbar_init(&s.bar_out, 256);
    s.abort = 0;
    fence_mbar_init();
  }
  __syncwarp();
  if (warp == 0) tmem_alloc_pair(&s.tmem_base, kPairTmemCols);
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync();  // both CTAs run and their barriers are initialised
  tc_fence_after_sync();
  constexpr uint32_t tR0 = 0, tR1 = 128, tDK = 256, tDV = 384, tDQ = 64;  // the allocation is the whole TMEM
  const uint32_t lead = cluster_addr(smem_raw, 0), peer = cluster_addr(smem_raw, rank ^ 1);
  auto off = [&](const void* p) -> uint32_t { return smem_u32(p) - smem_u32(smem_raw); };
  volatile int32_t* abort_flag = &s.abort;
  auto raise_abort = [&]() {
    *abort_flag = 1;
    cluster_store(peer + off(&s.abort), 1);
  };
  if ((misaligned || s.tmem_base != 0) && tid == 0) {
    report_timeout(a.status, -1, misaligned ? kWhereBwdSmemAlign : kWhereBwdTmemBase, static_cast<int32_t>(s.tmem_base));
    raise_abort();
  }
  uint32_t gs = 0, gi = 0;  // steps and items completed by this pair
  auto together = [&](bool here) -> bool { return __all_sync(0xffffffffu, here); };
  // One lane of a warp whose part in TMEM is done, to the first CTA's barrier
  auto arrive_lead = [&](uint64_t* bar) {
    if (rank == 0)
      mbar_arrive(bar);
    else
      cluster_arrive_relaxed(lead + off(bar));
  };

  // The first CTA's thread 0 pops for both. Every thread of both CTAs goes by the popped position alone, so both leave
  // together; all waits inside an item are bounded and no role returns before the end, so the cluster barriers are reached.
  auto next_item = [&]() -> bool {
    __syncwarp();
    tc_fence_before_sync();
    cluster_sync();
    if (rank == 0 && tid == 0) {
      int idx = a.n_items;
      if (*abort_flag == 0) {
        idx = atomicAdd(a.counter, 1);
        if (idx == a.n_items + static_cast<int>(gridDim.x / 2) - 1) *reinterpret_cast<volatile int32_t*>(a.counter) = 0;
        if (idx < a.n_items) {
          // start alignment (see fetch_item of the single-CTA kernel)
          const nsp_tile_t item = a.items[idx];
          const SegInfo sg = a.seg[item.seg];
          const int G = sg.hq / sg.hkv, steps = G * ((sg.len + kBM - 1) / kBM - max(2 * item.tile, 1));
          const int blk = idx / kFrontBlock, rest = a.n_items - blk * kFrontBlock;
          const int expect = rest < kFrontBlock ? rest : kFrontBlock;
          atomicAdd(a.front + blk, 1);
          if (steps >= kFrontMinSteps && G >= kFrontMinGroup) {
            const long long t0 = clock64(), own = static_cast<long long>(steps) * 340;
            const long long limit = own < kFrontWaitClk ? own : kFrontWaitClk;
            while (*reinterpret_cast<volatile int32_t*>(a.front + blk) < expect && clock64() - t0 < limit) __nanosleep(200);
          }
        } else {
          idx = a.n_items;
        }
      }
      s.pop = idx;
      cluster_store(peer + off(&s.pop), idx);
    }
    __syncwarp();
    cluster_sync();
    if (tid == 0) {
      PairCtx& x = s.ctx;
      x.it = s.pop;
      if (x.it < a.n_items) {
        const nsp_tile_t item = a.items[x.it];
        const SegInfo sg = a.seg[item.seg];
        x.q_off = sg.q_off, x.kv_off = sg.kv_off, x.lse_off = sg.lse_off;
        x.len = sg.len, x.hq = sg.hq, x.hkv = sg.hkv, x.run = sg.run, x.tok0 = sg.tok_in_run;
        x.g = item.head, x.n0 = 2 * item.tile, x.n = x.n0 + static_cast<int>(rank);
        x.G = sg.hq / sg.hkv;
        x.m0 = max(x.n0, 1);  // q tile 0 belongs to the first-tile kernel
        x.per_head = (sg.len + kBM - 1) / kBM - x.m0;
        x.steps = x.G * x.per_head;
      }
    }
    __syncwarp();
    __syncthreads();
    tc_fence_after_sync();
    return s.ctx.it < a.n_items;
  };
  auto item_done = [&]() {
    gs += static_cast<uint32_t>(s.ctx.steps);
    gi += 1;
  };

  if (wg == 4) {
    pair_setmaxnreg_dec<kRegsAux>();
    if (warp == 16) {
      // ================================================================ TMA producer (both CTAs, each its own operands)
      while (next_item()) {
        if (lane == 0) {
          const PairCtx c = s.ctx;
          const CUtensorMap* mq = &maps.q[c.run];
          const CUtensorMap* mdo = &maps.d_o[c.run];
          const int col = 64 * static_cast<int>(rank);
          // checked build, failure-detection test: one tile of the second CTA never arrives (K / V, or in the fourth step)
          auto withheld = [&]([[maybe_unused]] int load, [[maybe_unused]] int vt) -> bool {
#ifdef NSP_CHECKED
            return a.withhold == load && rank == 1 && c.it == 0 && vt == 2;
#else
            return false;
#endif
          };
          if (rank == 0) mbar_expect_tx(&s.bar_kv, 2 * 6 * kHalfTileBytes);
          const uint32_t kv = lead + off(&s.bar_kv);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            tma_load_3d_pair(s.k[i], &maps.k[c.run], kv, 64 * i, c.g, c.tok0 + c.n * kBN);
            if (!withheld(NSP_WITHHOLD_V, 2)) tma_load_3d_pair(s.v[i], &maps.v[c.run], kv, 64 * i, c.g, c.tok0 + c.n * kBN);
            tma_load_3d_pair(s.kt[i], &maps.k[c.run], kv, col, c.g, c.tok0 + (c.n0 + i) * kBN);
          }
          // boxes of q and dO are [64 rows x 64 columns]
          auto load_row = [&](uint8_t* dst, const CUtensorMap* map, uint64_t* bar, int h, int m) {
            if (rank == 0) mbar_expect_tx(bar, 2 * kHalfTileBytes);
            const uint32_t to = lead + off(bar);
#pragma unroll
            for (int i = 0; i < 2; ++i) tma_load_3d_pair(dst + i * (kHalfTileBytes / 2), map, to, 64 * i, h, c.tok0 + m * kBM + col);
          };
          auto load_col = [&](uint8_t* dst, const CUtensorMap* map, uint64_t* bar, int h, int m) {
            if (rank == 0) mbar_expect_tx(bar, 2 * kHalfTileBytes);
            const uint32_t to = lead + off(bar);
#pragma unroll
            for (int i = 0; i < 2; ++i) tma_load_3d_pair(dst + i * (kHalfTileBytes / 2), map, to, col, h, c.tok0 + m * kBM + 64 * i);
          };
          PairWalk w;
          int h, m;
          w.get(c, h, m);
          w.next(c);
          load_row(s.q_row, mq, &s.bar_qr_full, h, m);
          load_row(s.do_row, mdo, &s.bar_dor_full, h, m);
          load_col(s.do_col, mdo, &s.bar_doc_full, h, m);
          load_col(s.q_col, mq, &s.bar_qc_full, h, m);
          // A buffer is free when its product of the step before has completed; in the order in which they complete.
#pragma unroll 1
          for (int vt = 0; vt + 1 < c.steps; ++vt) {
            if (*abort_flag) break;
            const uint32_t ph = (gs + vt) & 1;
            w.get(c, h, m);
            w.next(c);
            int at = 0;
            bool ok = mbar_wait(&s.bar_s_full, ph, a.wait_limit);
            if (ok && !withheld(NSP_WITHHOLD_Q_ROWS, vt)) load_row(s.q_row, mq, &s.bar_qr_full, h, m);
            ok = ok && (++at, mbar_wait(&s.bar_dp_full, ph, a.wait_limit));
            if (ok && !withheld(NSP_WITHHOLD_DO_ROWS, vt)) load_row(s.do_row, mdo, &s.bar_dor_full, h, m);
            ok = ok && (++at, mbar_wait(&s.bar_dv_done, ph, a.wait_limit));
            if (ok && !withheld(NSP_WITHHOLD_DO_COLUMNS, vt)) load_col(s.do_col, mdo, &s.bar_doc_full, h, m);
            ok = ok && (++at, mbar_wait(&s.bar_dk_done, ph, a.wait_limit));
            if (ok && !withheld(NSP_WITHHOLD_Q_COLUMNS, vt)) load_col(s.q_col, mq, &s.bar_qc_full, h, m);
            if (!ok) {
              report_timeout(a.status, c.it, kWhereBwdQEmpty, 100000 * at + vt);  // of S^T, dP^T, dV, dK
              raise_abort();
              break;
            }
          }
        }
        __syncwarp();
        item_done();
      }
    } else if (warp == 18) {
      // ================================================================ LSE / delta loader
      while (next_item()) {
        const PairCtx c = s.ctx;
        PairWalk w;
#pragma unroll 1
        for (int vt = 0; vt < c.steps; ++vt) {
          const uint32_t cs = gs + vt, st = cs & 1;
          if (!together(*abort_flag == 0)) break;
          if (!together(mbar_wait(&s.bar_ld_empty[st], ((cs >> 1) & 1) ^ 1, a.wait_limit))) {
            if (lane == 0) {
              report_timeout(a.status, c.it, kWhereBwdLdEmpty, vt);
              raise_abort();
            }
            break;
          }
          int h, m;
          w.get(c, h, m);
          w.next(c);
          const int64_t base = c.lse_off + static_cast<int64_t>(h) * c.len;
          float lv[4], dv_[4];
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const int qi = m * kBM + lane + 32 * x;
            lv[x] = INFINITY, dv_[x] = 0.f;
            if (qi < c.len) {
              NSP_CHECK(base + qi >= 0 && base + qi < a.lse_elems, a.status, c.it, kWhereCheckBwdLse, qi) {
                lv[x] = a.lse[base + qi] * kLog2e;
                dv_[x] = a.delta[base + qi];
              }
            }
          }
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            s.lse[st][lane + 32 * x] = lv[x];
            s.delta[st][lane + 32 * x] = dv_[x];
          }
          mbar_arrive(&s.bar_ld_full[st]);
        }
        item_done();
      }
    } else if (rank != 0) {
      // ================================================================ second CTA: no products to issue
      // Its two warps pass on that this CTA's dS^T buffers are complete, 17 the part of its own softmax warps, 19 the received one:
      // releases at cluster scope that order what was stored here ahead of the first CTA's products. (Both parts passed on by one
      // warp: 131,072 tokens at 16q/1kv 163.5 ms a backward pass, now 162.8; 16 x 8,192 at 32q/4kv 21.74 / 21.58.)
      const bool own = warp == 17;
      uint64_t* const bar = own ? &s.bar_x_own : &s.bar_x_full;
      while (next_item()) {
        if (lane == 0) {
          const int steps = s.ctx.steps, it = s.ctx.it;
#pragma unroll 1
          for (int vt = 0; vt < steps; ++vt) {
            if (*abort_flag) break;
            if (!own) mbar_expect_tx(&s.bar_x_full, kHalfTileBytes);
            if (!mbar_wait(bar, (gs + vt) & 1, a.wait_limit)) {
              report_timeout(a.status, it, own ? kWhereBwdStaged : kWhereBwdXFull, vt);
              raise_abort();
              break;
            }
            cluster_arrive_release(lead + off(&s.bar_x_peer));
          }
        }
        __syncwarp();
        item_done();
      }
    } else {
      // ================================================================ MMA issuers, for both CTAs
      // A: dV(t), S^T(t+1); B: dK(t), dP^T(t+1), dQ^T(t)
      const bool is_a = warp == 17;
      while (next_item()) {
        {
          const bool leader = elect_one();
          constexpr uint32_t idesc_kk = make_idesc_bf16(256, 128, 0, 0);
          constexpr uint32_t idesc_kn = make_idesc_bf16(256, 128, 0, 1);
          constexpr uint32_t idesc_nn = make_idesc_bf16(128, 128, 1, 1);
          const uint32_t hi = static_cast<uint32_t>(make_smem_desc_sw128(0, 16, 1024) >> 32);
          constexpr uint32_t lbo_km = (16u >> 4) << 16, lbo_mn = (kHalfTileBytes >> 4) << 16;
          const int steps = s.ctx.steps, item_it = s.ctx.it;
          // The steps of q tile n0, the last ones, lie before every key of the second CTA (with n0 = 0 that q tile belongs to the
          // first-tile kernel). Its P^T and dS^T are zero there, but zero times a value that is not finite, of that q
          // tile or of keys that may be the next segment's, is not: they are left out of its dV and dK and of dQ^T.
          const int alone = s.ctx.n0 > 0 ? steps - s.ctx.G : steps;  // first of them
          int where = 0;
          bool okm = together(cluster_wait(&s.bar_kv, gi & 1, a.wait_limit));
          if (!okm) where = kWhereBwdLoadKV;
          int vt = 0;
          // [128 own rows] x [64 + 64 rows]: S^T or dP^T
          auto issue_kk = [&](uint32_t d, uint32_t a_km, uint32_t b_km, bool go) {
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
              const uint32_t ao = ((kk >> 2) * kHalfTileBytes + (kk & 3) * 32) >> 4;
              const uint32_t bo = ((kk >> 2) * (kHalfTileBytes / 2) + (kk & 3) * 32) >> 4;
              if (go) umma2_ss_lh(d, a_km + ao, hi, b_km + bo, hi, idesc_kk, kk > 0);
            }
          };
          // packed P^T or dS^T: 16 queries = 8 columns; queries 16 kk .. belong to warpgroup (kk >> 1) & 1
          auto issue_kn = [&](uint32_t d, uint32_t a_tmem, uint32_t b_mn, int at, bool go) {
            const uint32_t acc = at > 0;
            if (at >= alone) {
#pragma unroll 1
              for (int kk = 0; kk < 8; ++kk)
                if (go) umma2_ts_lh_first(d, a_tmem + ((kk >> 1) & 1) * 32 + (kk >> 2) * 16 + (kk & 1) * 8, b_mn + kk * 128, hi,
                                          idesc_kn, acc | (kk > 0));
              return;
            }
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
              if (go) umma2_ts_lh(d, a_tmem + ((kk >> 1) & 1) * 32 + (kk >> 2) * 16 + (kk & 1) * 8, b_mn + kk * 128, hi, idesc_kn,
                                  acc | (kk > 0));
          };
          if (is_a) {
            const uint32_t k_km = smem_desc_addr(s.k[0]) | lbo_km, q_km = smem_desc_addr(s.q_row) | lbo_km;
            const uint32_t do_mn = smem_desc_addr(s.do_col) | lbo_mn;
            auto issue_s = [&](int vt, bool here) -> bool {  // here: the Q rows have arrived
              const uint32_t cs = gs + vt;
              // R0 [64, 128) held dQ^T of the step before the last one (of this item: earlier ones are long drained)
              if (vt > 0) here = cluster_wait_tmem(&s.bar_dq_empty, cs & 1, a.wait_limit) && here;
              tc_fence_after_sync();
              issue_kk(tR0, k_km, q_km, leader && here);
              if (!together(here)) { where = vt > 0 ? kWhereBwdDqEmpty : kWhereBwdLoadQ; return false; }
              if (leader) umma2_commit(&s.bar_s_full);
              return true;
            };
            okm = okm && issue_s(0, cluster_wait(&s.bar_qr_full, gs & 1, a.wait_limit));
#pragma unroll 1
            for (; okm && vt < steps; ++vt) {
              const bool calm = *abort_flag == 0;
              const uint32_t cs = gs + vt;
              const bool more = vt + 1 < steps;
              bool here = more ? cluster_wait2(&s.bar_doc_full, cs & 1, &s.bar_qr_full, (cs + 1) & 1, a.wait_limit)
                               : cluster_wait(&s.bar_doc_full, cs & 1, a.wait_limit);
              here = cluster_wait_tmem(&s.bar_p_ready, cs & 1, a.wait_limit) && here;
              tc_fence_after_sync();
              issue_kn(tDV, tR0, do_mn, vt, leader && here);
              if (!together(here && calm)) {
                if (!together(here)) where = kWhereBwdPReady;
                okm = false;
                break;
              }
              if (leader) umma2_commit(&s.bar_dv_done);
              if (more && !issue_s(vt + 1, true)) { okm = false; break; }
            }
          } else {
            const uint32_t v_km = smem_desc_addr(s.v[0]) | lbo_km, do_km = smem_desc_addr(s.do_row) | lbo_km;
            const uint32_t q_mn = smem_desc_addr(s.q_col) | lbo_mn;
            const uint32_t kt_mn = smem_desc_addr(s.kt[0]) | lbo_mn, x_mn = smem_desc_addr(s.x[0]) | lbo_mn;
            auto issue_dp = [&](bool here) -> bool {  // here: the dO rows have arrived
              issue_kk(tR1, v_km, do_km, leader && here);
              if (!together(here)) { where = kWhereBwdLoadQ; return false; }
              if (leader) umma2_commit(&s.bar_dp_full);
              return true;
            };
            // Every phase of s_read is waited for, so that none is taken for the one before; the first one here, ahead of the dP^T
            // without which the softmax warps do not get to the next step (behind dS^T of the first step the barrier may be two
            // phases ahead, and the wait for it would not end).
            const bool s_read = cluster_wait_tmem(&s.bar_s_read, gs & 1, a.wait_limit);
            okm = okm && issue_dp(cluster_wait(&s.bar_dor_full, gs & 1, a.wait_limit) && s_read);
#pragma unroll 1
            for (; okm && vt < steps; ++vt) {
              const bool calm = *abort_flag == 0;
              const uint32_t cs = gs + vt;
              if (leader) mbar_expect_tx(&s.bar_x_full, kHalfTileBytes);
              const bool more = vt + 1 < steps;
              bool here = more ? cluster_wait2(&s.bar_qc_full, cs & 1, &s.bar_dor_full, (cs + 1) & 1, a.wait_limit)
                               : cluster_wait(&s.bar_qc_full, cs & 1, a.wait_limit);
              here = cluster_wait_tmem(&s.bar_ds_ready, cs & 1, a.wait_limit) && here;
              tc_fence_after_sync();
              issue_kn(tDK, tR1, q_mn, vt, leader && here);
              if (!together(here && calm)) {
                if (!together(here)) where = kWhereBwdDsReady;
                okm = false;
                break;
              }
              if (leader) umma2_commit(&s.bar_dk_done);
              if (more && !issue_dp(true)) { okm = false; break; }
              // dQ^T over the part of R0 that packed P^T leaves free, once S^T of the next step, which waits for the drain of the
              // dQ^T before, has been read from it; behind the last S^T that drain itself is waited for
              uint64_t* const free_bar = more ? &s.bar_s_read : &s.bar_dq_empty;
              here = wait_both([&] { return mbar_try_wait(&s.bar_x_own, cs & 1); },
                               [&] { return cluster_try_wait_relaxed(free_bar, (cs + 1) & 1); }, a.wait_limit);
              here = cluster_wait2(&s.bar_x_full, cs & 1, &s.bar_x_peer, cs & 1, a.wait_limit) && here;
              tc_fence_after_sync();
              const bool go = leader && here;
#pragma unroll
              for (int kk = 0; kk < 16; ++kk)  // sixteen keys each, the first CTA's key tile first
                if (go && (kk < 8 || vt < alone)) umma2_ss_lh(tDQ, kt_mn + kk * 128, hi, x_mn + kk * 128, hi, idesc_nn, kk > 0);
              if (!together(here)) {
                where = kWhereBwdStaged;
                okm = false;
                break;
              }
              if (leader) umma2_commit(&s.bar_dq_full);
            }
          }
          if (!okm) {
            // Which of the waits in front of the failed vote: the first whose phase is still missing, or the last of them.
            // (Told apart inside the loops it cost 0.5 % of a pass.)
            const uint32_t cs = gs + vt;
            const bool more = vt + 1 < steps;
            auto missing = [&](uint64_t* bar, uint32_t parity) -> bool { return !together(mbar_test(bar, parity & 1)); };
            if (where == kWhereBwdPReady) {
              if (missing(&s.bar_doc_full, cs) || (more && missing(&s.bar_qr_full, cs + 1))) where = kWhereBwdLoadQ;
            } else if (where == kWhereBwdDsReady) {
              if (missing(&s.bar_qc_full, cs) || (more && missing(&s.bar_dor_full, cs + 1))) where = kWhereBwdLoadQ;
            } else if (where == kWhereBwdLoadQ && !is_a) {
              if (!missing(&s.bar_dor_full, gs)) where = kWhereBwdSRead;
            } else if (where == kWhereBwdStaged && !missing(&s.bar_x_own, cs)) {
              where = missing(more ? &s.bar_s_read : &s.bar_dq_empty, cs + 1) ? (more ? kWhereBwdSRead : kWhereBwdDqEmpty)
                      : missing(&s.bar_x_full, cs)                            ? kWhereBwdXFull
                                                                              : kWhereBwdXPeer;
            }
            if (leader && where != 0) report_timeout(a.status, item_it, where, is_a ? 0 : 1);
            drain_products();
            raise_abort();
          }
        }
        item_done();
      }
    }
  } else if (wg >= 2) {
    // ================================================================ dQ^T -> global fp32 accumulator
    // CTA r has d = 64 r .. 64 r + 63. Column j of the region is query j of a query set: lanes 0..63 the first CTA's,
    // lanes 64..127 the second's. A set is 32 consecutive queries from 32 w and 32 from 64 + 32 w.
    pair_setmaxnreg_dec<kRegsReduce>();
    const int quad = warp & 3, half = wg - 2;
    const int q0 = 64 * half + 32 * (quad >> 1);  // first of this warp's 32 consecutive query rows
    const int d = 64 * static_cast<int>(rank) + 32 * (quad & 1) + lane;
    const uint32_t src = tDQ + (static_cast<uint32_t>(quad * 32) << 16) + 32 * half;
    while (next_item()) {
      const PairCtx c = s.ctx;
      PairWalk w;
#pragma unroll 1
      for (int vt = 0; vt < c.steps; ++vt) {
        const uint32_t cs = gs + vt;
        if (!together(*abort_flag == 0)) break;
        if (!together(mbar_wait(&s.bar_dq_full, cs & 1, a.wait_limit))) {
          if (lane == 0) {
            report_timeout(a.status, c.it, kWhereBwdDqFull, vt);
            raise_abort();
          }
          break;
        }
        tc_fence_after_sync();
        int h, m;
        w.get(c, h, m);
        w.next(c);
        uint32_t v[32];
        tmem_ld32(src, v);
        tmem_wait_ld();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) arrive_lead(&s.bar_dq_empty);
        // Added by TMA: as 32 reductions per thread they fill the memory queue that the softmax warps' waits and shared-memory
        // accesses go through (65,536 tokens at 4q/1kv 10.4 -> 10.1 ms a backward pass). Sixteen rows at a time through the
        // warp's 2 KB. Rows past the segment's end add zeros (their dS^T columns are zero) to the first rows of the segments
        // behind it, which nobody reads, or lie outside the tensor map.
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if (lane == 0) tma_store_wait_read();
          __syncwarp();
#pragma unroll
          for (int e = 0; e < 16; ++e) s.dq_out[warp - 8][e][lane] = __uint_as_float(v[16 * i + e]);
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_reduce_add_3d(&maps.dq_acc[c.run], s.dq_out[warp - 8], d - lane, h, c.tok0 + m * kBM + q0 + 16 * i);
            tma_store_commit();
          }
        }
      }
      if (lane == 0) tma_store_wait();
      __syncwarp();
      item_done();
    }
  } else {
    // ================================================================ softmax / dS (key row r, 2 x 32 query columns)
    pair_setmaxnreg_inc<kRegsSoft>();
    const int quad = warp & 3;
    const int r = quad * 32 + lane;
    const int qb = 32 * wg;  // query columns qb .. qb + 31 and 64 + qb ..
    const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
    const uint32_t tS = tR0 + lane_off + qb, tDP = tR1 + lane_off + qb;  // also where the packed columns go
    const bool keep = wg == static_cast<int>(rank);  // this warpgroup's queries are this CTA's query set
    uint8_t* const ds_row = (keep ? s.x[rank] : s.stage) + r * 128;
    const uint32_t x_to = peer + off(s.x[rank]) + quad * 4096, x_bar = peer + off(&s.bar_x_full);
    while (next_item()) {
      const PairCtx c = s.ctx;
      bool oks = true;
      int where = 0, vt = 0;
      PairWalk w;
#pragma unroll 1
      for (; vt < c.steps; ++vt) {
        const uint32_t cs = gs + vt, st = cs & 1;
        int h, m;
        w.get(c, h, m);
        w.next(c);
        const bool calm = *abort_flag == 0;
        oks = mbar_wait2(&s.bar_ld_full[st], (cs >> 1) & 1, &s.bar_s_full, cs & 1, a.wait_limit);
        if (!together(oks && calm)) {
          if (!together(oks)) where = kWhereBwdS;
          oks = false;
          break;
        }
        tc_fence_after_sync();
        const float* lse_s = s.lse[st] + qb;
        const float* delta_s = s.delta[st] + qb;
        auto step = [&](auto diag_tag) -> bool {
          uint32_t sv[2][32];
          float4 aux[2][4];
#pragma unroll
          for (int i = 0; i < 4; ++i) aux[0][i] = lds128(lse_s + 4 * i);
          tmem_ld32(tS, sv[0]);
          tmem_ld32(tS + 64, sv[1]);
          tmem_wait_ld();
          tc_fence_before_sync();
          if (lane == 0) arrive_lead(&s.bar_s_read);
          uint32_t pp[2][16];
#pragma unroll
          for (int ch = 0; ch < 4; ++ch) {  // 16 columns each: 64 * (ch / 2) + 16 * (ch % 2)
            if (ch < 3) {
#pragma unroll
              for (int i = 0; i < 4; ++i) aux[(ch + 1) & 1][i] = lds128(lse_s + ((ch + 1) >> 1) * 64 + ((ch + 1) & 1) * 16 + 4 * i);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float4 l4 = aux[ch & 1][i];
              const int x = (ch & 1) * 16 + 4 * i;
              float x0, x1, x2, x3;
              fma2(x0, x1, __uint_as_float(sv[ch >> 1][x + 0]), __uint_as_float(sv[ch >> 1][x + 1]), a.scale_log2,
                   a.scale_log2, -l4.x, -l4.y);
              fma2(x2, x3, __uint_as_float(sv[ch >> 1][x + 2]), __uint_as_float(sv[ch >> 1][x + 3]), a.scale_log2,
                   a.scale_log2, -l4.z, -l4.w);
              pp[ch >> 1][(x >> 1) + 0] = pack_bf16x2(ex2f(x0), ex2f(x1));
              pp[ch >> 1][(x >> 1) + 1] = pack_bf16x2(ex2f(x2), ex2f(x3));
            }
            if constexpr (decltype(diag_tag)::value) {
              // a key sees only the queries at or after it (the second CTA's last q tile lies wholly before its keys)
              const int t = r + (c.n - m) * kBN - (qb + (ch >> 1) * 64 + (ch & 1) * 16);
#pragma unroll
              for (int kk = 0; kk < 8; ++kk) {
                const uint32_t mask = t <= 2 * kk ? 0xffffffffu : (t == 2 * kk + 1 ? 0xffff0000u : 0u);
                pp[ch >> 1][(ch & 1) * 8 + kk] &= mask;
              }
            }
            if (ch & 1) tmem_st16(tS + (ch >> 1) * 16, pp[ch >> 1]);
          }
          tmem_wait_st();
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) arrive_lead(&s.bar_p_ready);
#pragma unroll
          for (int i = 0; i < 4; ++i) aux[0][i] = lds128(delta_s + 4 * i);
          // the dS^T buffers are free once dQ^T of the step before has completed
          oks = mbar_wait2(&s.bar_dp_full, cs & 1, &s.bar_dq_full, (cs - 1) & 1, a.wait_limit);
          if (!together(oks)) { where = kWhereBwdDp; return false; }
          tc_fence_after_sync();
          uint32_t dpv[2][16];
          tmem_ld16(tDP, dpv[0]);
#pragma unroll
          for (int ch = 0; ch < 4; ++ch) {
            tmem_wait_ld();
            if (ch < 3) {
              tmem_ld16(tDP + ((ch + 1) >> 1) * 64 + ((ch + 1) & 1) * 16, dpv[(ch + 1) & 1]);
#pragma unroll
              for (int i = 0; i < 4; ++i) aux[(ch + 1) & 1][i] = lds128(delta_s + ((ch + 1) >> 1) * 64 + ((ch + 1) & 1) * 16 + 4 * i);
            }
            uint32_t* const dsp = &pp[ch >> 1][(ch & 1) * 8];  // in the place of P^T
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float4 d4 = aux[ch & 1][i];
              const int x = 4 * i;
              const uint32_t pa = dsp[x >> 1], pb = dsp[(x >> 1) + 1];
              float d0, d1, d2, d3;
              sub2(d0, d1, __uint_as_float(dpv[ch & 1][x + 0]), __uint_as_float(dpv[ch & 1][x + 1]), d4.x, d4.y);
              sub2(d2, d3, __uint_as_float(dpv[ch & 1][x + 2]), __uint_as_float(dpv[ch & 1][x + 3]), d4.z, d4.w);
              mul2(d0, d1, d0, d1, __uint_as_float(pa << 16), __uint_as_float(pa & 0xffff0000u));
              mul2(d2, d3, d2, d3, __uint_as_float(pb << 16), __uint_as_float(pb & 0xffff0000u));
              dsp[(x >> 1) + 0] = pack_bf16x2(d0, d1);
              dsp[(x >> 1) + 1] = pack_bf16x2(d2, d3);
            }
            if (ch & 1) tmem_st16(tDP + (ch >> 1) * 16, pp[ch >> 1]);
            *reinterpret_cast<uint4*>(ds_row + ((2 * ch) ^ (r & 7)) * 16) = make_uint4(dsp[0], dsp[1], dsp[2], dsp[3]);
            *reinterpret_cast<uint4*>(ds_row + ((2 * ch + 1) ^ (r & 7)) * 16) = make_uint4(dsp[4], dsp[5], dsp[6], dsp[7]);
          }
          tmem_wait_st();
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) {
            arrive_lead(&s.bar_ds_ready);  // dK and dP^T of the next step need no more than this
            mbar_arrive(&s.bar_ld_empty[st]);
          }
          return true;
        };
        if (m > c.n) {
          if (!step(std::false_type{})) break;
        } else {
          if (!step(std::true_type{})) break;
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          if (keep)
            mbar_arrive(&s.bar_x_own);
          else
            copy_to_cluster(x_to, s.stage + quad * 4096, 4096, x_bar);
        }
      }
      // ---- epilogue: wait for the last products of the item, then write dK (scaled) and dV of this key tile
      if (oks) {
        const uint32_t lastp = (gs + c.steps - 1) & 1;
        oks = mbar_wait(&s.bar_dv_done, lastp, a.wait_limit) && mbar_wait(&s.bar_dk_done, lastp, a.wait_limit) &&
              mbar_wait(&s.bar_dq_full, lastp, a.wait_limit);
        oks = together(oks);
        if (!oks) where = kWhereBwdMma2;
      }
      const int rows = min(kBN, c.len - c.n * kBN);  // none for the second CTA where the segment has an odd number of key tiles
      if (oks) {
        tc_fence_after_sync();
        const bool add = c.n == 0;  // the first-tile kernel left its part (q tile 0) in the output
        constexpr uint32_t kSubBytes = 128 * 32 * 4;
        uint8_t* const stage_k = &s.k[0][0];  // over K and K^T
        uint8_t* const stage_v = &s.v[0][0];  // over V and the row tiles
        if (quad * 32 < rows) {
#pragma unroll 1
          for (int i = 0; i < 4; ++i) {  // (dK, dV) x 32-column sub-tiles
            const int piece = i * 2 + wg, which = piece / 4, cc = piece % 4;
            const float mul = which == 0 ? a.scale : 1.f;
            uint32_t v[32];
            tmem_ld32(tDK + which * (tDV - tDK) + lane_off + cc * 32, v);
            tmem_wait_ld();
            uint8_t* const sub = (which == 0 ? stage_k : stage_v) + cc * kSubBytes + r * 128;
#pragma unroll
            for (int x = 0; x < 8; ++x) {
              *reinterpret_cast<float4*>(sub + ((x ^ (r & 7)) * 16)) =
                  make_float4(__uint_as_float(v[4 * x]) * mul, __uint_as_float(v[4 * x + 1]) * mul,
                              __uint_as_float(v[4 * x + 2]) * mul, __uint_as_float(v[4 * x + 3]) * mul);
            }
          }
        }
        const bool full = a.dkv_f32 && rows == kBN;
        if (full) fence_proxy_async_smem();
        const uint64_t staged = mbar_arrive_token(&s.bar_out);
        if (full) {
          if (tid == 0) {
            if (mbar_wait_token(&s.bar_out, staged, a.wait_limit)) {
              const int tok = c.tok0 + c.n * kBN;
#pragma unroll 1
              for (int i = 0; i < 4; ++i) {
                if (add) {
                  tma_reduce_add_3d(&maps.dk[c.run], stage_k + i * kSubBytes, 32 * i, c.g, tok);
                  tma_reduce_add_3d(&maps.dv[c.run], stage_v + i * kSubBytes, 32 * i, c.g, tok);
                } else {
                  tma_store_3d(&maps.dk[c.run], stage_k + i * kSubBytes, 32 * i, c.g, tok);
                  tma_store_3d(&maps.dv[c.run], stage_v + i * kSubBytes, 32 * i, c.g, tok);
                }
              }
              tma_store_commit();
              tma_store_wait_read();
            } else {
              report_timeout(a.status, c.it, kWhereBwdDqFull, 1);
              raise_abort();
            }
          }
        } else if (rows > 0) {
          // ragged tiles and bf16 outputs: a warp writes whole rows, four row passes in flight
          bool oku = mbar_wait_token(&s.bar_out, staged, a.wait_limit);
          if (!oku) {
            report_timeout(a.status, c.it, kWhereBwdDqFull, 1);
            raise_abort();
          }
          oku = together(oku);
#pragma unroll 1
          for (int it = 0; oku && it < 2 * 16; it += 4) {
            const int which = it / 16;
            const uint8_t* const st0 = (which == 0 ? stage_k : stage_v) + (lane / 8) * kSubBytes;
            void* const outp = which == 0 ? a.dk : a.dv;
            float4 w4[4];
            int64_t at[4];
            bool on[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int row = (it + u) % 16 * 8 + warp;
              on[u] = row < rows;
              at[u] = c.kv_off + (static_cast<int64_t>(c.n * kBN + row) * c.hkv + c.g) * D + 4 * lane;
              w4[u] = *reinterpret_cast<const float4*>(st0 + row * 128 + ((lane % 8) ^ (row & 7)) * 16);
#ifdef NSP_CHECKED
              if (on[u] && (at[u] < 0 || at[u] + 4 > a.kv_elems)) {
                report_status(a.status, NSP_ERR_DEVICE_ASSERT, c.it, kWhereCheckBwdDkv, row);
                on[u] = false;
              }
#endif
            }
            if (a.dkv_f32) {
              float* const o = static_cast<float*>(outp);
              if (add) {
                float4 old[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) old[u] = on[u] ? __ldcg(reinterpret_cast<const float4*>(o + at[u])) : w4[u];
#pragma unroll
                for (int u = 0; u < 4; ++u) w4[u].x += old[u].x, w4[u].y += old[u].y, w4[u].z += old[u].z, w4[u].w += old[u].w;
              }
#pragma unroll
              for (int u = 0; u < 4; ++u)
                if (on[u]) *reinterpret_cast<float4*>(o + at[u]) = w4[u];
            } else {
              __nv_bfloat16* const o = static_cast<__nv_bfloat16*>(outp);
              if (add) {
                uint2 old[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) old[u] = on[u] ? __ldcg(reinterpret_cast<const uint2*>(o + at[u])) : make_uint2(0u, 0u);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  w4[u].x += __uint_as_float(old[u].x << 16), w4[u].y += __uint_as_float(old[u].x & 0xffff0000u);
                  w4[u].z += __uint_as_float(old[u].y << 16), w4[u].w += __uint_as_float(old[u].y & 0xffff0000u);
                }
              }
#pragma unroll
              for (int u = 0; u < 4; ++u)
                if (on[u])
                  *reinterpret_cast<uint2*>(o + at[u]) = make_uint2(pack_bf16x2(w4[u].x, w4[u].y), pack_bf16x2(w4[u].z, w4[u].w));
            }
          }
          fence_proxy_async_smem();
        }
      } else if (where != 0 && lane == 0) {
        // which of the two waits of a step, or of the three behind the last
        const uint32_t cs = gs + vt;
        if (where == kWhereBwdS && !mbar_test(&s.bar_ld_full[cs & 1], (cs >> 1) & 1)) where = kWhereBwdLdFull;
        if (where == kWhereBwdDp && mbar_test(&s.bar_dp_full, cs & 1)) where = kWhereBwdDqFull;
        if (where == kWhereBwdMma2 && !mbar_test(&s.bar_dq_full, (cs - 1) & 1)) where = kWhereBwdDqFull;
        report_timeout(a.status, c.it, where, vt);
        raise_abort();
      }
      item_done();
    }
  }

  // After a failed wait (both flags are set: the barriers of next_item lie in between) roles of either CTA have left loads,
  // products and copies of dS^T to the other CTA under way, which nobody waits for any more: they end before either leaves.
  if (*abort_flag) drain_products();
  __syncwarp();
  tc_fence_before_sync();
  cluster_sync();  // neither CTA leaves while the other may still reach its shared memory or issue products into its TMEM
  if (warp == 0) tmem_dealloc_pair(s.tmem_base, kPairTmemCols);
}

}  // namespace

cudaError_t launch_bwd_pair(const BwdPairMaps& maps, const BwdArgs& args, int num_sms, cudaStream_t st) {
  if (args.n_items == 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(bwd_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sizeof(PairSmem)));
  if (e != cudaSuccess) return e;
  const int pairs = args.n_items < num_sms / 2 ? args.n_items : num_sms / 2;
  count_launches(1);
  return launch_chained_if(false, bwd_pair_kernel, 2 * pairs, kPairThreads, sizeof(PairSmem), st, maps, args);
}

}  // namespace nsp
