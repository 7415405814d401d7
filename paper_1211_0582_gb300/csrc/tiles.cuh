// Element ranges of the tiles of a persistent launch.
#pragma once
#include <cstdint>

namespace dgmx {

// Whole rounds of full tiles (`full` elements each, `grid` tiles per round),
// then the remaining elements in tiles of `small` elements, sized so that the
// last round spreads over the whole grid instead of leaving most blocks idle
// behind a few full tiles.
struct TileMap {
  int nfull, small, ntiles, full;
  __host__ __device__ int64_t start(int t) const {
    return t < nfull ? int64_t(t) * full : int64_t(nfull) * full + int64_t(t - nfull) * small;
  }
  __host__ __device__ int size(int t, int64_t K) const {
    const int64_t k0 = start(t), n = t < nfull ? full : small;
    return int(K - k0 < n ? K - k0 : n);
  }
};

inline TileMap make_tiles(int64_t K, int grid, int full) {
  const int64_t nfull = K / full / grid * grid;
  const int64_t rest = K - nfull * full;
  int64_t small = (rest + grid - 1) / grid;
  if (small < 1) small = 1;
  if (small > full) small = full;
  const int64_t nsmall = (rest + small - 1) / small;
  return TileMap{int(nfull), int(small), int(nfull + nsmall), full};
}

} // namespace dgmx
