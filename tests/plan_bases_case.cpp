// plan_tile_bases against the sums that the list kernel takes for small plans (csrc/nsp_plan.cu), over random batches.
#include <algorithm>
#include <cstdio>
#include <random>
#include "nsp_plan_bases.h"

using namespace nsp;

static int check(const std::vector<PlanKey>& key) {
  std::vector<int32_t> order(key.size());
  for (size_t s = 0; s < key.size(); ++s) order[s] = static_cast<int32_t>(s);
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return key[x].len > key[y].len; });
  const std::vector<TileBase> got = plan_tile_bases(key, order);
  size_t t = 0;
  for (size_t s = 0; s < key.size(); ++s)
    for (int m = 0; m < key[s].tiles; ++m, ++t) {
      const PlanKey& k = key[s];
      const int cf = m + 1, cb = k.group * (k.tiles - m);
      int64_t nf = 0, nb = 0, ne = 0, np = 0;
      for (size_t x = 0; x < key.size(); ++x) {
        const PlanKey& o = key[x];
        const bool before = x < s;
        for (int c = 1; c <= o.tiles; ++c) {
          const bool first = c > cf || (c == cf && before);
          nf += first ? o.hq : 0;
          if (c >= 2 || cf == 1) np += !first ? 0 : o.group % 2 == 0 ? o.hq / 2 : (o.tiles - c) % 2 == 0 ? o.hq : 0;
          nb += o.group * c > cb || (o.group * c == cb && before) ? o.hq / o.group : 0;
        }
        ne += o.len > k.len || (o.len == k.len && before) ? o.hq / o.group * o.tiles : 0;
      }
      const TileBase b = got[t];
      const bool starts_pair = m > 0 && (k.group % 2 == 0 || (k.tiles - cf) % 2 == 0);
      if (b.fwd != nf || b.bwd != nb || b.exec != ne || (starts_pair && b.pairs != np)) {
        std::printf("segment %zu tile %d: %d %d %d %d, not %lld %lld %lld %lld\n", s, m, b.fwd, b.bwd, b.exec, b.pairs,
                    static_cast<long long>(nf), static_cast<long long>(nb), static_cast<long long>(ne), static_cast<long long>(np));
        return 1;
      }
    }
  return t == got.size() ? 0 : 1;
}

int main() {
  std::mt19937 rng(7);
  auto below = [&](int n) { return static_cast<int>(rng() % n); };
  if (check({}) || check({{0, 4, 2, 0}}) || check({{1, 1, 1, 5}})) return 1;
  for (int round = 0; round < 300; ++round) {
    std::vector<PlanKey> key;
    const int kinds = 1 + below(4), n = 1 + below(40), most = 1 + below(round % 3 == 0 ? 3 : 1500);
    int hq[4], group[4];
    for (int i = 0; i < kinds; ++i) group[i] = 1 + below(8), hq[i] = group[i] * (1 + below(4));
    for (int s = 0; s < n; ++s) {
      const int i = below(kinds), len = below(6) == 0 ? 0 : 1 + below(most);
      key.push_back(PlanKey{(len + 127) / 128, hq[i], group[i], len});
    }
    if (check(key)) return std::printf("round %d\n", round), 1;
  }
  return 0;
}
