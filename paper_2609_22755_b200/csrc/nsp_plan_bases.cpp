// The positions the list kernel otherwise takes as sums over all segments, by counting: one cursor per cost, advanced over
// the segments in order. Linear in the tiles (times the distinct group sizes for the backward list).
#include "nsp_plan_bases.h"
#include <algorithm>

namespace nsp {

std::vector<TileBase> plan_tile_bases(const std::vector<PlanKey>& key, const std::vector<int32_t>& by_length) {
  int32_t most = 0;
  int64_t n_tiles = 0;
  for (const PlanKey& k : key) most = std::max(most, k.tiles), n_tiles += k.tiles;
  std::vector<TileBase> out(static_cast<size_t>(n_tiles));

  // forward and pairs: the cost of tile m is m + 1. Items, and pairs, of cost c = those of the segments of c tiles and more;
  // an odd group has pairs at every second cost from its tile count down.
  std::vector<int32_t> fwd(most + 2, 0), even(most + 2, 0), odd(most + 3, 0), pairs(most + 2, 0);
  for (const PlanKey& k : key) {
    if (k.tiles == 0) continue;
    fwd[k.tiles] += k.hq;
    if (k.group % 2 == 0) even[k.tiles] += k.hq / 2; else odd[k.tiles] += k.hq;
  }
  for (int32_t c = most - 1; c >= 1; --c) fwd[c] += fwd[c + 1], even[c] += even[c + 1], odd[c] += odd[c + 2];
  for (int32_t c = most, f = 0, p = 0; c >= 1; --c) {  // counts become the cursors
    const int32_t nf = fwd[c], np = even[c] + odd[c];
    fwd[c] = f, pairs[c] = p;
    f += nf, p += np;
  }

  // backward: the cost of tile m is group * (tiles - m), so tiles of different groups may share a cost, and a cursor
  struct Group {
    int32_t size, most;
    std::vector<int32_t> above;   // [q] items of this group of cost > size * q
    std::vector<int32_t> owner;   // [q] the first group that has the cost size * q; its cursor is used
    std::vector<int32_t> cursor;
  };
  std::vector<Group> groups;
  std::vector<int32_t> group_of(key.size(), -1);
  for (size_t s = 0; s < key.size(); ++s) {
    if (key[s].tiles == 0) continue;
    size_t g = 0;
    while (g < groups.size() && groups[g].size != key[s].group) ++g;
    if (g == groups.size()) groups.push_back(Group{key[s].group, 0, {}, {}, {}});
    groups[g].most = std::max(groups[g].most, key[s].tiles);
    group_of[s] = static_cast<int32_t>(g);
  }
  for (Group& g : groups) g.above.assign(g.most + 2, 0), g.owner.assign(g.most + 1, 0), g.cursor.assign(g.most + 1, 0);
  for (size_t s = 0; s < key.size(); ++s)
    if (group_of[s] >= 0) groups[group_of[s]].above[key[s].tiles] += key[s].hq / key[s].group;
  for (Group& g : groups) {
    for (int32_t q = g.most - 1; q >= 1; --q) g.above[q] += g.above[q + 1];  // items of cost size * q
    int32_t sum = 0;
    for (int32_t q = g.most; q >= 0; --q) {
      const int32_t n = g.above[q];
      g.above[q] = sum;
      sum += n;
    }
  }
  for (size_t i = 0; i < groups.size(); ++i)
    for (int32_t q = 1; q <= groups[i].most; ++q) {
      const int64_t cost = static_cast<int64_t>(groups[i].size) * q;
      int32_t owner = -1, start = 0;
      for (size_t j = 0; j < groups.size(); ++j) {
        const Group& o = groups[j];
        if (owner < 0 && cost % o.size == 0 && cost / o.size <= o.most) owner = static_cast<int32_t>(j);
        start += o.above[std::min<int64_t>(cost / o.size, o.most)];
      }
      groups[i].owner[q] = owner;
      groups[i].cursor[q] = start;
    }

  int32_t exec = 0;
  std::vector<int32_t> exec_of(key.size(), 0);
  for (const int32_t s : by_length) {
    exec_of[s] = exec;
    exec += key[s].hq / key[s].group * key[s].tiles;
  }

  size_t t = 0;
  for (size_t s = 0; s < key.size(); ++s) {
    const PlanKey& k = key[s];
    const int32_t hkv = k.hq / k.group;
    for (int32_t m = 0; m < k.tiles; ++m, ++t) {
      const int32_t c = m + 1;
      Group& g = groups[group_of[s]];
      Group& o = groups[g.owner[k.tiles - m]];
      int32_t& bwd = o.cursor[static_cast<int64_t>(g.size) * (k.tiles - m) / o.size];
      out[t] = TileBase{fwd[c], bwd, exec_of[s], pairs[c]};
      fwd[c] += k.hq;
      bwd += hkv;
      if (k.group % 2 == 0)
        pairs[c] += k.hq / 2;
      else if ((k.tiles - c) % 2 == 0)
        pairs[c] += k.hq;
    }
  }
  return out;
}

}  // namespace nsp
