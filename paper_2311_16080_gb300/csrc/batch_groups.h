// Which domains of a batch run on the resident kernel, and in what groups (host
// code without CUDA calls: what the GPU can hold is asked through functions).
#pragma once
#include <algorithm>
#include <functional>
#include <map>
#include <utility>
#include <vector>

#include "resident2d.h"

namespace xlb {

// Domains that one launch of the resident kernel advances.
struct Bucket {
  ResidentShape shape;
  int first = 0, count = 0;  // its domains in DomainGroups::order
};

struct DomainGroups {
  std::vector<Bucket> buckets;  // larger clusters first
  std::vector<int> order;       // the groups' domains one after the other, then the rest
  int n_rest = 0;               // domains that take the queue
};

// Group the domains of `ord` (largest first) by the launch shape they need:
// blocks per cluster, one or two blocks per SM.  shape_of(d): domain d's shape
// (ctas = 0: it fits no cluster); fits(shape): whether the GPU, or the part of
// it this process has, can hold a cluster of that shape at all.
template <typename ShapeOf, typename Fits>
DomainGroups group_domains(const std::vector<int>& ord, ShapeOf&& shape_of, Fits&& fits) {
  using Key = std::pair<int, int>;
  std::map<Key, ResidentShape, std::greater<Key>> shape;
  std::vector<Key> key(ord.size(), Key(0, 0));
  for (size_t k = 0; k < ord.size(); ++k) {
    const ResidentShape s = shape_of(ord[k]);
    if (s.ctas == 0) continue;
    key[k] = Key(s.ctas, !s.one && s.threads > 512);
    auto it = shape.find(key[k]);
    if (it == shape.end()) {
      shape[key[k]] = s;
      continue;
    }
    ResidentShape& m = it->second;
    // one cell per thread only where that serves every domain of the group
    m.threads = m.one == s.one ? std::max(m.threads, s.threads) : (m.one ? s.threads : m.threads);
    m.one = m.one && s.one;
    m.smem = std::max(m.smem, s.smem);
  }
  DomainGroups g;
  for (auto it = shape.begin(); it != shape.end();) {
    if (!fits(it->second)) {
      it = shape.erase(it);
      continue;
    }
    Bucket b;
    b.shape = it->second;
    b.first = (int)g.order.size();
    for (size_t k = 0; k < ord.size(); ++k)
      if (key[k] == it->first) g.order.push_back(ord[k]);
    b.count = (int)g.order.size() - b.first;
    g.buckets.push_back(b);
    ++it;
  }
  for (size_t k = 0; k < ord.size(); ++k)
    if (!shape.count(key[k])) g.order.push_back(ord[k]);
  g.n_rest = (int)(g.order.size() - (g.buckets.empty() ? 0 : g.buckets.back().first + g.buckets.back().count));
  return g;
}

}  // namespace xlb
