// Single-bin Hermite kernels (body per lane) through a list of observation times, n = 2..8.
#include "hermite_impl.cuh"

namespace swarm {

cudaError_t launch_hermite_obs_bpl_a(int n, const BinView &B, int nunits, const StepParams &P, int grid, cudaStream_t st, int *blocks) {
  switch (n) {
    case 2:
      if (blocks) *blocks = hermite_uniform_blocks_n<SWARM_MAP_BODY_PER_LANE, 2, false, true>();
      return grid > 0 ? launch_hermite_uniform_n<SWARM_MAP_BODY_PER_LANE, 2, false, true>(B, nunits, P, grid, st) : cudaSuccess;
    case 3:
      if (blocks) *blocks = hermite_uniform_blocks_n<SWARM_MAP_BODY_PER_LANE, 3, false, true>();
      return grid > 0 ? launch_hermite_uniform_n<SWARM_MAP_BODY_PER_LANE, 3, false, true>(B, nunits, P, grid, st) : cudaSuccess;
    case 4:
      if (blocks) *blocks = hermite_uniform_blocks_n<SWARM_MAP_BODY_PER_LANE, 4, false, true>();
      return grid > 0 ? launch_hermite_uniform_n<SWARM_MAP_BODY_PER_LANE, 4, false, true>(B, nunits, P, grid, st) : cudaSuccess;
    case 5:
      if (blocks) *blocks = hermite_uniform_blocks_n<SWARM_MAP_BODY_PER_LANE, 5, false, true>();
      return grid > 0 ? launch_hermite_uniform_n<SWARM_MAP_BODY_PER_LANE, 5, false, true>(B, nunits, P, grid, st) : cudaSuccess;
    case 6:
      if (blocks) *blocks = hermite_uniform_blocks_n<SWARM_MAP_BODY_PER_LANE, 6, false, true>();
      return grid > 0 ? launch_hermite_uniform_n<SWARM_MAP_BODY_PER_LANE, 6, false, true>(B, nunits, P, grid, st) : cudaSuccess;
    case 7:
      if (blocks) *blocks = hermite_uniform_blocks_n<SWARM_MAP_BODY_PER_LANE, 7, false, true>();
      return grid > 0 ? launch_hermite_uniform_n<SWARM_MAP_BODY_PER_LANE, 7, false, true>(B, nunits, P, grid, st) : cudaSuccess;
    case 8:
      if (blocks) *blocks = hermite_uniform_blocks_n<SWARM_MAP_BODY_PER_LANE, 8, false, true>();
      return grid > 0 ? launch_hermite_uniform_n<SWARM_MAP_BODY_PER_LANE, 8, false, true>(B, nunits, P, grid, st) : cudaSuccess;
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace swarm
