// Element ranges of the tiles of a persistent launch.
#pragma once
#include <cstdint>

namespace dgmx {

// Whole rounds of full tiles (FULL elements each, `grid` tiles per round), then
// the remaining elements in tiles of `small` elements, sized so that the last
// round spreads over the whole grid instead of leaving most blocks idle behind
// a few full tiles. A mesh of less than a round is spread over all blocks: a
// smaller tile is through its phases sooner. (The N = 6, 7 stage and the reverse
// stage, us per launch against full tiles and one ragged last one: N=6 6,000
// tets 42.2 -> 27.4, N=7 162 tets 16.7 -> 13.6 and 24,576 tets 153 -> 136;
// traces and their gradient, N=5, 3,024 tets, 9.48 -> 8.64 ms.)
template <int FULL>
struct TileMap {
  int nfull, small, ntiles;
  __host__ __device__ int64_t start(int t) const {
    return t < nfull ? int64_t(t) * FULL : int64_t(nfull) * FULL + int64_t(t - nfull) * small;
  }
  __host__ __device__ int size(int t, int64_t K) const {
    const int64_t k0 = start(t), n = t < nfull ? FULL : small;
    return int(K - k0 < n ? K - k0 : n);
  }
};

template <int FULL>
TileMap<FULL> make_tiles(int64_t K, int grid) {
  const int64_t nfull = K / FULL / grid * grid;
  const int64_t rest = K - nfull * FULL;
  int64_t small = (rest + grid - 1) / grid;
  if (small < 1) small = 1;
  if (small > FULL) small = FULL;
  const int64_t nsmall = (rest + small - 1) / small;
  return TileMap<FULL>{int(nfull), int(small), int(nfull + nsmall)};
}

// Blocks of a launch that may have `cap` resident at once: half of them where
// their tiles then have at most `most` elements. The other half of the SMs' room
// takes the next stage's blocks, whose setup (operators, tables, tensor memory)
// overlaps this stage (programmatic dependent launch) instead of following it;
// in the FP32 stage a block that has its SM to itself is also through its tile
// sooner. `most` is where each launch stops gaining, from sweeps over every tile
// size (us per stage, all blocks and half): FP16x3 N=4 1,520 tets 7.37 -> 6.79,
// N=5 1,520 tets 9.73 -> 8.01; N=7 912 tets 15.3 -> 15.1, but 1,520 tets 16.3 ->
// 17.3: 12 elements at N = 6, 7. A right-hand side has no stage after it: on its
// own it takes the same time either way up to 12 elements and longer from there
// (FP16x3 N=4 760 tets 11.0 and 11.1, 1,216 tets 11.1 -> 12.6; only a chain of
// nothing but right-hand sides gains there, 6.71 -> 5.89).
template <int FULL>
int small_mesh_blocks(int64_t K, int cap, int most = FULL) {
  return cap >= 2 && K <= int64_t(most) * (cap / 2) ? cap / 2 : cap;
}

} // namespace dgmx
