// tile_plan.h -- which tile shape a line takes (host code, no CUDA).
#pragma once

namespace shasta {

// Tile shapes of the tiled sweeps: c cells per lane, xl lines per warp, so
// 32 c / xl positions per tile, 12 of them halo.  Shapes of one line per warp
// serve x sweeps only (along y and z a warp would touch half of each sector).
struct TileShape {
  int c, xl;
};
constexpr TileShape kTileShapes[] = {{4, 2}, {5, 2}, {6, 2}, {7, 2}, {8, 2}, {9, 2}, {5, 1}, {6, 1}, {7, 1}};
constexpr int kTileShapeCount = 9;
constexpr int kTileHalo = 12;  // halo positions of a tile, both sides
// the kernels' int positions hold lines this long with room for the halo
constexpr long long kTileMaxLine = 1LL << 30;

inline int tile_positions(int shape) { return 32 * kTileShapes[shape].c / kTileShapes[shape].xl; }
inline int tile_own(int shape) { return tile_positions(shape) - kTileHalo; }

// One axis: shape (-1: the streaming sweep), tiles per line and their length.
struct TilePlan {
  int shape;
  int ntile, len;
  int blocks_per_sm;
};

inline void tile_cut(TilePlan& t, int n) {
  t.ntile = (n + tile_own(t.shape) - 1) / tile_own(t.shape);
  t.len = (n + t.ntile - 1) / t.ntile;
}

// The shape that computes the fewest positions for a line of n cells: every
// computed cell costs about the same in all of them (11-12 ps at 200^3, C = 4
// .. 9, one or two lines per warp).  On a tie the fewer cells per lane, which
// is the shorter chain.
inline int tile_shape_for(int n, int axis) {
  int best = 0;
  long long cost = -1;
  for (int i = 0; i < kTileShapeCount; ++i) {
    if (axis != 0 && kTileShapes[i].xl != 2) continue;
    const long long k = ((long long)n + tile_own(i) - 1) / tile_own(i) * tile_positions(i);
    if (cost < 0 || k < cost) {
      cost = k;
      best = i;
    }
  }
  return best;
}

}  // namespace shasta
