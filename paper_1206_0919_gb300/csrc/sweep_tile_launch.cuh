// sweep_tile_launch.cuh -- kernel tables and launchers of the tiled FP32 /
// MIXED sweeps (sweep_tile.cuh), one equation of state and recovery per
// including unit.
#pragma once

#include "chain.cuh"
#include "kernels.h"
#include "sweep_tile.cuh"

namespace shasta {
namespace tile {

template <int EOS, int REC, int AXIS, int I>
struct Entry {
  static constexpr int C = kTileShapes[I].c, XL = kTileShapes[I].xl;
  using L = Lay<AXIS, C, XL>;
  // C <= 7 fits 128 registers (16 warps per SM); 8 and 9 need 168 (12 warps)
  static constexpr int MINB = C <= 7 ? 4 : 3;
  static void* fun() { return (void*)sweep_tile_kernel<EOS, AXIS, REC, C, XL, MINB>; }
};

struct Kern {
  void* fun;
  int smem, warps, units;  // bytes and warps per block; lines per work unit
};

template <int EOS, int REC, int AXIS, int I>
Kern kern() {
  if constexpr (AXIS != 0 && kTileShapes[I].xl != 2) {
    return Kern{nullptr, 0, 0, 0};
  } else {
    using E = Entry<EOS, REC, AXIS, I>;
    return Kern{E::fun(), E::L::SMEM, E::L::WARPS, AXIS == 0 ? E::XL : YL};
  }
}

template <int EOS, int REC, int AXIS>
Kern kern_of(int i) {
  switch (i) {
    case 0: return kern<EOS, REC, AXIS, 0>();
    case 1: return kern<EOS, REC, AXIS, 1>();
    case 2: return kern<EOS, REC, AXIS, 2>();
    case 3: return kern<EOS, REC, AXIS, 3>();
    case 4: return kern<EOS, REC, AXIS, 4>();
    case 5: return kern<EOS, REC, AXIS, 5>();
    case 6: return kern<EOS, REC, AXIS, 6>();
    case 7: return kern<EOS, REC, AXIS, 7>();
    case 8: return kern<EOS, REC, AXIS, 8>();
    case 9: return kern<EOS, REC, AXIS, 9>();
    case 10: return kern<EOS, REC, AXIS, 10>();
  }
  return Kern{nullptr, 0, 0, 0};
}

template <int EOS, int REC>
Kern lookup(int axis, int shape) {
  return axis == 0 ? kern_of<EOS, REC, 0>(shape)
                   : (axis == 1 ? kern_of<EOS, REC, 1>(shape) : kern_of<EOS, REC, 2>(shape));
}

template <int EOS, int REC>
cudaError_t prepare(int axis, int shape, int* blocks_per_sm) {
  const Kern k = lookup<EOS, REC>(axis, shape);
  *blocks_per_sm = 0;
  if (!k.fun) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k.fun, cudaFuncAttributeMaxDynamicSharedMemorySize, k.smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k.fun, k.warps * 32, k.smem);
}

template <int EOS, int REC>
cudaError_t launch(const SweepParams& P, const TilePlan& t, int axis, int sm_count, bool chain, cudaStream_t s) {
  if (P.plane <= 0) return cudaSuccess;
  const Kern k = lookup<EOS, REC>(axis, t.shape);
  if (!k.fun || t.blocks_per_sm < 1 || t.ntile < 1) return cudaErrorInvalidValue;
  TileArgs A;
  A.ntile = t.ntile;
  A.len = t.len;
  set_divisor(A, (unsigned)P.nb);
  const long long tiles = (P.plane + k.units - 1) / k.units * t.ntile;
  const long long need = axis == 0 ? (tiles + k.warps - 1) / k.warps : tiles;  // x: one tile per warp
  const long long wave = (long long)sm_count * t.blocks_per_sm;
  void* args[] = {const_cast<SweepParams*>(&P), &A};
  return launch_sweep_kernel(k.fun, dim3((unsigned)(need < wave ? need : wave)), dim3(k.warps * 32), args, k.smem,
                             chain, s);
}

}  // namespace tile
}  // namespace shasta
