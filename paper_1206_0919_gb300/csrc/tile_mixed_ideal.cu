// tile_mixed_ideal.cu -- tiled sweeps: precision mixed, ideal equation of state.
#include "sweep_tile_launch.cuh"

namespace shasta {

cudaError_t prepare_tile_mixed_ideal(int axis, int shape, int* blocks_per_sm) {
  return tile::prepare<EOS_IDEAL, fast::REC_DF>(axis, shape, blocks_per_sm);
}

cudaError_t launch_tile_mixed_ideal(const SweepParams& P, const TilePlan& t, int axis, int sm_count, bool chain,
                                    cudaStream_t s) {
  return tile::launch<EOS_IDEAL, fast::REC_DF>(P, t, axis, sm_count, chain, s);
}

}  // namespace shasta
