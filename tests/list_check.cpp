// Host-side check of csrc/nasg_list.h: the forward's walk over a tile's list in batches of NT meets each
// place of the list once, in order, and no other, also where the list ends next to 2^32.
#include <cstdio>
#include <initializer_list>
#include <vector>

#include "nasg_list.h"

static bool walk(uint64_t first, uint32_t n, uint32_t nt) {
  // as the sorts note it: the complement of the first place, the last place + 1; zeros for no entry
  const nasg::TileList list = nasg::tile_list(n ? ~uint32_t(first) : 0u, n ? uint32_t(first + n) : 0u);
  if (list.count != n) return false;
  std::vector<uint64_t> seen;
  uint32_t batches = 0;
  for (nasg::ListWalk w(list); w.left > 0; w.next(nt)) {
    if (++batches > n / nt + 1) return false;  // it does not end
    for (uint32_t slot = 0; slot < nt; ++slot)
      if (slot < w.left) seen.push_back(uint64_t(w.place) + slot);
  }
  if (seen.size() != n) return false;
  for (uint32_t k = 0; k < n; ++k)
    if (seen[k] != first + k) return false;
  return true;
}

int main() {
  const uint64_t top = (uint64_t(1) << 32) - 1;  // the most pairs a forward takes
  int cases = 0;
  for (uint32_t nt : {128u, 256u})
    for (uint32_t n : {0u, 1u, 31u, 127u, 128u, 129u, 255u, 256u, 257u, 1000u, 70000u})
      for (uint64_t end : {uint64_t(n), uint64_t(n) + 5, uint64_t(1) << 31, top - 300, top - 128, top - 1, top}) {
        if (end < n) continue;
        if (!walk(end - n, n, nt)) return std::printf("nt %u n %u end %llu\n", nt, n, (unsigned long long)end), 1;
        ++cases;
      }
  std::printf("ok %d\n", cases);
  return 0;
}
