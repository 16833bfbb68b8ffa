// Where the items of every tile start in the plan's lists (see nsp_plan.cu): plain C++, host only.
#pragma once
#include <cstdint>
#include <vector>

namespace nsp {

// What the list construction needs of a segment.
struct PlanKey {
  int32_t tiles, hq, group, len;  // 128-row tiles, q heads, q heads per kv head, tokens
};

// Positions of a (segment, tile)'s first item in the forward and backward lists, of its segment's first item in the walked
// list, and (in pairs) of its first pair.
struct TileBase {
  int32_t fwd, bwd, exec, pairs;
};

// One entry per (segment, tile), tiles ascending inside a segment. by_length: the segments by length descending, ties by
// index. May throw std::bad_alloc.
std::vector<TileBase> plan_tile_bases(const std::vector<PlanKey>& key, const std::vector<int32_t>& by_length);

}  // namespace nsp
