// tile_plan.h -- which tile shape a line takes (host code, no CUDA).
#pragma once

namespace shasta {

// Tile shapes of the tiled sweeps: c cells per lane, xl lines per warp, so
// 32 c / xl positions per tile, 12 of them halo.  Shapes of one line per warp
// serve x sweeps only (along y and z a warp would touch half of each sector).
struct TileShape {
  int c, xl;
};
constexpr TileShape kTileShapes[] = {{4, 2}, {5, 2}, {6, 2}, {7, 2}, {8, 2}, {9, 2},
                                     {5, 1}, {6, 1}, {7, 1}, {8, 1}, {9, 1}};
constexpr int kTileShapeCount = 11;
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

// The shape that computes the fewest positions for a line of n cells: a
// computed cell costs about the same in all of them (11-12 ps at 200^3, C = 4
// .. 9), 3% more with 8 or 9 cells per lane (12 warps per SM instead of 16;
// 256^3 along x, C = 9 against 5) and 4% less with one line per warp (200^3
// along x: 90.3 us against 94.4).  On a tie the fewer cells per lane, which is
// the shorter chain.
inline int tile_shape_for(int n, int axis) {
  int best = 0;
  double cost = -1.0;
  for (int i = 0; i < kTileShapeCount; ++i) {
    if (axis != 0 && kTileShapes[i].xl != 2) continue;
    const double k = (double)(((long long)n + tile_own(i) - 1) / tile_own(i) * tile_positions(i)) *
                     (kTileShapes[i].c >= 8 ? 1.03 : 1.0) * (kTileShapes[i].xl == 1 ? 0.96 : 1.0);
    if (cost < 0 || k < cost) {
      cost = k;
      best = i;
    }
  }
  return best;
}

}  // namespace shasta
