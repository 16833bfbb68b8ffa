// Device-side construction of the tile work lists (forward, backward, the backward items in the order the kernel
// walks them, and the forward items in the pairs its kernel runs).
//
// Item definitions and order (unique, so any correct construction gives the same lists bit for bit):
//   forward  (s, h, m): cost = ceil(min(L, (m+1)*bm) / bn)          -- key tiles the query tile visits
//   backward (s, g, n): cost = G * (Mt - floor(n*bn / bm))          -- (q head, q tile) visits of the key tile
//   order: cost descending, then segment, tile, head ascending.
//   pairs    of forward items with at least two key tiles, by the cost of their first item descending, then segment, head:
//            an even group: (s, h, m), (s, h + 1, m) for even h; otherwise (s, h, m), (s, h, m - 1) for m = Mt-1, Mt-3, ..
//            (without a second item where m - 1 = 0, which belongs to the first-tile kernel: seg = -1).
//   walked   (s, g, n): groups (s, g) by segment length descending, then s, g ascending; n ascending inside a group.
//
// With bm == bn a segment has at most one tile of a given cost, so the position of a tile's items in each list is a sum
// over the segments of a closed form: one warp per (segment, tile) takes that sum (the lanes stride over the segments)
// and writes the tile's items, no keys and no sort. A plan of 8,192 tokens at 32q/4kv spent 60 us in two radix sorts
// with their key and decode kernels; this is one launch of about 5 us. The sums are tiles x segments terms; where that is
// more than a counting pass on the host costs, the positions come from there (nsp_plan_bases.cpp).
// 128 threads of 32 registers, no shared memory: a block fits beside the general forward kernel (61,440 of the 65,536
// registers of an SM). It does not fit beside the backward kernels, which leave no shared memory for another block (and at
// head_dim 64 no registers); then it starts when one of their blocks ends, and the host does not wait for it (nsp_api.cu).
#include <cuda_bf16.h>
#include "nsp_internal.cuh"

namespace nsp {

namespace {

constexpr int kListThreads = 128;

__global__ void __launch_bounds__(kListThreads, 16)
    plan_lists_kernel(const PlanKey* __restrict__ key, const int32_t* __restrict__ tile_base,
                      const TileBase* __restrict__ bases, int n_seg, int n_tiles, nsp_tile_t* __restrict__ fwd,
                      nsp_tile_t* __restrict__ bwd, nsp_tile_t* __restrict__ exec, nsp_tile_t* __restrict__ pairs) {
  const int lane = threadIdx.x & 31;
  const int n_warps = gridDim.x * (kListThreads / 32);
  for (int t = (blockIdx.x * kListThreads + threadIdx.x) >> 5; t < n_tiles; t += n_warps) {
    int s = 0, hi = n_seg - 1;  // the last segment that starts at or before tile t (empty segments start where the next does)
    while (s < hi) {
      const int mid = (s + hi + 1) >> 1;
      if (tile_base[mid] <= t) s = mid; else hi = mid - 1;
    }
    const PlanKey k = key[s];
    const int m = t - tile_base[s];
    const int cf = m + 1, cb = k.group * (k.tiles - m);
    int nf = 0, nb = 0, ne = 0, np = 0;  // items before this tile's (before its group's, in the walked order); pairs likewise
    for (int x = bases ? n_seg : lane; x < n_seg; x += 32) {
      const PlanKey o = key[x];
      const int hkv = o.hq / o.group;
      const bool before = x < s;
      // forward: the tiles of cost > cf, and the tile of cost == cf of an earlier segment
      nf += o.hq * (max(o.tiles - cf, 0) + (before && o.tiles >= cf));
      // backward: cost = group * k, k = 1 .. tiles
      const int q = cb / o.group;
      nb += hkv * (max(o.tiles - q, 0) + (before && q * o.group == cb && q <= o.tiles));
      // pairs: an even group has hq / 2 of every cost 2 .. tiles; another hq of the costs tiles, tiles - 2, .. >= 2
      if (o.group & 1)
        np += o.hq * ((max(o.tiles - cf, 0) + 1) / 2 + (before && o.tiles >= cf && ((o.tiles - cf) & 1) == 0));
      else
        np += o.hq / 2 * (max(o.tiles - cf, 0) + (before && o.tiles >= cf));
      ne += o.len > k.len || (o.len == k.len && before) ? hkv * o.tiles : 0;
    }
    nf = __reduce_add_sync(0xffffffffu, nf);
    nb = __reduce_add_sync(0xffffffffu, nb);
    ne = __reduce_add_sync(0xffffffffu, ne);
    np = __reduce_add_sync(0xffffffffu, np);
    if (bases) {
      const TileBase b = bases[t];
      nf = b.fwd, nb = b.bwd, ne = b.exec, np = b.pairs;
    }
    if (m > 0) {
      if (!(k.group & 1)) {
        for (int h = lane; h < k.hq; h += 32) pairs[2 * np + h] = nsp_tile_t{s, h, m, cf};
      } else if (((k.tiles - cf) & 1) == 0) {
        for (int h = lane; h < k.hq; h += 32) {
          pairs[2 * (np + h)] = nsp_tile_t{s, h, m, cf};
          pairs[2 * (np + h) + 1] = m > 1 ? nsp_tile_t{s, h, m - 1, cf - 1} : nsp_tile_t{-1, 0, 0, 0};
        }
      }
    }
    for (int h = lane; h < k.hq; h += 32) fwd[nf + h] = nsp_tile_t{s, h, m, cf};
    for (int g = lane; g < k.hq / k.group; g += 32) {
      bwd[nb + g] = nsp_tile_t{s, g, m, cb};
      exec[ne + g * k.tiles + m] = nsp_tile_t{s, g, m, cb};
    }
  }
}

}  // namespace

cudaError_t launch_plan_lists(const PlanKey* d_key, const int32_t* d_tile_base, const TileBase* d_bases, int n_seg, int n_tiles,
                              nsp_tile_t* d_fwd, nsp_tile_t* d_bwd, nsp_tile_t* d_exec, nsp_tile_t* d_pairs, cudaStream_t st) {
  if (n_tiles == 0) return cudaSuccess;
  const int blocks = (n_tiles + kListThreads / 32 - 1) / (kListThreads / 32);
  plan_lists_kernel<<<blocks < 148 * 8 ? blocks : 148 * 8, kListThreads, 0, st>>>(
      d_key, d_tile_base, d_bases, n_seg, n_tiles, d_fwd, d_bwd, d_exec, d_pairs);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace nsp
