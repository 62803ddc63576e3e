// Walks over a tile's list [begin, end) of (tile, primitive) pairs in batches. The lists of a frame
// may hold close to 2^32 pairs, so places past a list's end need not fit 32 bits: none is formed
// (a list holds each primitive once: fewer than 2^31 entries). Plain arithmetic, shared by the
// rendering kernels and a host-side check.
#pragma once

#include <stdint.h>

#if defined(__CUDACC__)
#define NASG_LIST_HD __host__ __device__ __forceinline__
#else
#define NASG_LIST_HD inline
#endif

namespace nasg {

struct TileList {
  uint32_t begin, count;
};

// The range as the sorts leave it, x: complement of the first place, y: last place + 1 (both zero
// for no entry).
NASG_LIST_HD TileList tile_list(uint32_t not_first, uint32_t end) {
  return {~not_first, end ? end - ~not_first : 0u};
}

// From the beginning: the batch's first place and the entries from there on (slot t < left holds
// place + t); next by `size` entries.
struct ListWalk {
  uint32_t place, left;

  NASG_LIST_HD explicit ListWalk(TileList l) : place(l.begin), left(l.count) {}
  NASG_LIST_HD void next(uint32_t size) {
    place += size;
    left = left > size ? left - size : 0u;
  }
};

}  // namespace nasg
