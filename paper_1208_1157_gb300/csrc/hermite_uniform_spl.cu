// Single-bin persistent Hermite kernels (system per lane), n = 2..4.
#include "hermite_impl.cuh"

namespace swarm {

cudaError_t launch_hermite_uniform_spl(int n, const BinView &B, int nunits, const StepParams &P, int grid, cudaStream_t st, int *blocks) {
  constexpr int M = SWARM_MAP_SYSTEM_PER_LANE;
  const bool ad = P.integrator == SWARM_HERMITE4_ADAPTIVE;
  switch (n) {
    case 2: return launch_hermite_uniform_pick<M, 2>(B, nunits, P, grid, st, blocks, ad);
    case 3: return launch_hermite_uniform_pick<M, 3>(B, nunits, P, grid, st, blocks, ad);
    case 4: return launch_hermite_uniform_pick<M, 4>(B, nunits, P, grid, st, blocks, ad);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace swarm
