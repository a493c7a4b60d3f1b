// tile_plan.h -- which tile shape a line takes, and where tiles are worth it
// (host code, no CUDA).
#pragma once

#include <algorithm>

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

// Estimated times (us, 152 SMs) of one sweep over `lines` lines of n cells: on
// tiles, streamed with a timed choice of ranges, and streamed untimed (ranges
// of at least 24 positions, so lines shorter than that are taken one after the
// other by a warp).  A tile computes all its positions, own or not, so short
// lines waste most of it (a line of 16 cells: 64 positions), where streaming
// pays a lead-in of 14 to 26 positions; the double recovery (rec64) makes each
// position ten times dearer in both.  g: line groups per warp of one wave of 16
// per SM; below one the streamed chain is bound by its latency.
// Measured against (x, FP32, us, tiles / timed / untimed): 200 x 200 lines of 8
// cells 33.7 / 25.5 / 47.9, of 24 33.5 / 37.7 / 37.8; 400 x 400 of 5 143 / 66 /
// 89, of 16 116 / 87 / 87, of 32 114 / 121 / 120; 1024 x 1024 of 1 908 / 295 /
// 390, of 16 780 / 509 / 511, of 48 771 / 871 / 877; z is 12% faster streamed.
// MIXED_FP64: 128 x 96 of 16 94 / 99 / 172; 200 x 200 of 16 291 / 182 / 220, of
// 128 627 / 677 / 699; 256 x 256 of 256 2023 / 1906 / 1919; 1024 x 1024 of 16
// 7588 / 3044 / 3141.
struct SweepCost {
  double tile, stream, untimed;
};
inline SweepCost sweep_cost(long long lines, int n, int axis, int shape, bool rec64, int sm_count) {
  const double g = (double)lines / (512.0 * sm_count);
  const long long cut = ((long long)n + tile_own(shape) - 1) / tile_own(shape);
  const double computed = (double)(cut * tile_positions(shape));
  const double below = std::min(g, 1.0);
  const double queue = n < 24 ? (double)((23 + n) / n) : 1.0;  // lines one after the other
  SweepCost c;
  if (rec64) {
    const double per = 8.5 * g + (2.2 - 1.5 * below) * std::min(1.0, 48.0 / n);
    c.tile = 10.0 + 8.5 * g * computed;
    c.stream = (n + 14) * per;
    c.untimed = (n + 14) * std::max(per, queue > 1.0 ? 3.3 * queue : 0.0);
  } else {
    const double dir = axis == 0 ? 1.0 : 0.88;
    const double per = dir * std::max(0.6 + 0.6 * below * below, g);
    // lines shorter than the halo take the tile's general ghost mapping
    c.tile = 4.0 + 0.85 * g * computed * (n < 6 ? 1.2 : 1.0);
    c.stream = (n + 26) * per;
    c.untimed = (n + 26) * std::max(per, queue > 1.0 ? 0.48 * dir * queue : 0.0);
  }
  return c;
}
// Where the choice between tiles and streaming goes by these estimates too:
// lines that leave most of a tile unused, and the double recovery at any size.
inline bool by_cost(int n, bool rec64) { return rec64 || n < 50; }

}  // namespace shasta
