// Persistent multi-step form of the FP32 fused stage, for ensembles of meshes.
//
// An ensemble of independent meshes is stored as one disjoint union (elements
// of mesh i contiguous, neighbours always inside the same mesh, each element
// carrying its mesh's time step in geo[k][G_DT]). One cooperative launch then
// advances every mesh by `nsteps` LSERK4 steps: each block loops over
// element tiles of Cfg::EB elements (picked by the autotuner), and a
// grid-wide barrier separates the five stages of every step, because a stage
// reads the neighbours' states written by the previous stage. Field loads go
// through L2 (the L1 of another SM may hold a stale copy from two stages ago).
#pragma once
#include "grid_sync.cuh"
#include "simt_stage.cuh"

namespace dgmx {

// u_a holds the state at entry; stages alternate u_a -> u_b -> u_a ...
template <int N, class Cfg>
__global__ void __launch_bounds__(Cfg::NT, Cfg::MINB)
    k_ensemble_persistent(StageArgs a, StageCoeffs rk, float *u_a, float *u_b, int nsteps, GridBarrier *gb,
                          TileMap<Cfg::EB> tm, int *err_flag) {
  extern __shared__ float4 smem4[];
  uint8_t *smem = reinterpret_cast<uint8_t *>(smem4);
  bool flip = false;
  simt_setup<Cfg>(a, smem4);
  for (int step = 0; step < nsteps; ++step)
    for (int st = 0; st < 5; ++st) {
      a.u = flip ? u_b : u_a;
      a.u_out = flip ? u_a : u_b;
      a.rk_a = rk.a[st];
      a.rk_b = rk.b[st];
      for (int t = blockIdx.x; t < tm.ntiles; t += gridDim.x) {
        __syncthreads(); // shared memory of the previous tile is no longer read
        simt_stage_tile<N, MODE_LSERK, Cfg, true>(a, tm.start(t), tm.size(t, a.K), smem);
      }
      if (!grid_barrier(gb, a.wait_limit > 0 ? a.wait_limit : (1ll << 31))) {
        if (threadIdx.x == 0) atomicExch(err_flag, 1);
        return;
      }
      flip = !flip;
    }
}

} // namespace dgmx

namespace dgmx {

// Tile candidates of the autotuner for order N, in elements: where the
// one-element shape serves alone its tile and three, two and one quarter of it;
// elsewhere the two-element shape's tile, the wide one-element shape's, and the
// narrow one's and half of it. (Half of the two-element tile, in the wide one's
// place before, was never the fastest; us per stage, without and with the wide
// tile: N=4 8,484 tets 31.5 -> 27.4, 44,982 tets 140 -> 132; N=5 2,976 tets 28.2 ->
// 23.1; N=7 1,458 tets 45.5 -> 36.1; N=8 1,458 tets 66.5 -> 61.8; N=9 1,458 tets
// 128 -> 121.)
template <int N>
struct EnsembleCandidates {
  static constexpr int shape(int i) { return simt_one_only<N>() || i >= 2 ? SHAPE_ONE : i == 1 ? SHAPE_ONE_WIDE : SHAPE_TWO; }
  static constexpr int c(int i) {
    if (simt_one_only<N>()) return SimtShape<N, SHAPE_ONE>::EB * (4 - i) / 8 * 2;
    if (i < 2) return i ? SimtShape<N, SHAPE_ONE_WIDE>::EB : SimtShape<N, SHAPE_TWO>::EB;
    return SimtShape<N, SHAPE_ONE>::EB / (i == 3 ? 4 : 2) * 2;
  }
  template <int I>
  using Cfg = SimtCfg<N, shape(I), c(I)>;
};

// occ = 0: as many blocks per SM as fit; occ = 1: half as many (rounded up),
// a second tuning axis (fewer blocks take part in each grid barrier, more
// tiles per block); the blocks per SM launched go to *used (may be null)
template <int N, class Cfg>
cudaError_t launch_ensemble_cfg(const StageArgs &a, const StageCoeffs &rk, float *ua, float *ub, int nsteps,
                               GridBarrier *gb, int *flag, cudaStream_t s, int sms, int occ, int *used) {
  auto kern = k_ensemble_persistent<N, Cfg>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(Cfg::SMEM));
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, Cfg::NT, Cfg::SMEM);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  if (occ == 1) per_sm = (per_sm + 1) / 2;
  if (used) *used = per_sm;
  const TileMap<Cfg::EB> tm = make_tiles<Cfg::EB>(a.K, per_sm * sms);
  const unsigned grid = unsigned(tm.ntiles < per_sm * sms ? tm.ntiles : per_sm * sms);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(Cfg::NT);
  cfg.dynamicSmemBytes = Cfg::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a, rk, ua, ub, nsteps, gb, tm, flag);
}

// Candidate cand: tile C::c(cand % 4), occupancy level cand / 4.
template <int N>
cudaError_t launch_ensemble_order(int cand, const StageArgs &a, const StageCoeffs &rk, float *ua, float *ub,
                                  int nsteps, GridBarrier *gb, int *flag, cudaStream_t s, int sms, int *used) {
  using C = EnsembleCandidates<N>;
  const int occ = cand / 4;
  switch (cand % 4) {
  case 0: return launch_ensemble_cfg<N, typename C::template Cfg<0>>(a, rk, ua, ub, nsteps, gb, flag, s, sms, occ, used);
  case 1: return launch_ensemble_cfg<N, typename C::template Cfg<1>>(a, rk, ua, ub, nsteps, gb, flag, s, sms, occ, used);
  case 2: return launch_ensemble_cfg<N, typename C::template Cfg<2>>(a, rk, ua, ub, nsteps, gb, flag, s, sms, occ, used);
  default: return launch_ensemble_cfg<N, typename C::template Cfg<3>>(a, rk, ua, ub, nsteps, gb, flag, s, sms, occ, used);
  }
}

} // namespace dgmx
