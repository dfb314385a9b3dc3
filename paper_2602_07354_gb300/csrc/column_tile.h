// Tiling of the kernels whose threads own voxel columns and march z (smoothing, hotspots, stress).
#pragma once

#include "elas_internal.h"

namespace elas {

struct ColumnTile {
  int tx = 0, ty = 0, zc = 0;  // columns of a tile, layers of an item
  int items = 0;               // one block per item
  int threads = 0;             // of a block, where the kernel has a choice
};

// Tile of at most `threads` columns with the fewest idle threads over the grid (an idle lane costs
// its warp's FP64 instructions as much as a busy one), then the fewest staged columns (a halo of hx
// and hy in all); layers per item so that the busiest SM (its blocks share its pipes) has the least
// work, an item's neighbour planes counted as `extra` layers.  One block per item: the hardware
// hands them out as SMs free up.  max_pos: staged columns a block has room for; max_items: a limit on
// the blocks (0: none).
inline ColumnTile column_tile(const Geo& g, int threads, int hx, int hy, double extra, int sm_count, int max_pos,
                              int max_items = 0) {
  ColumnTile best{};
  double cost0 = 1e300;
  for (int tx = 4; tx <= 64; ++tx) {
    const int ty = threads / tx;
    const int pos = (tx + hx) * (ty + hy);
    if (ty < 1 || pos > max_pos) continue;
    const double cost = (double)((g.nx - 1) / tx + 1) * ((g.ny - 1) / ty + 1) * (threads + 0.3 * pos);
    if (cost < cost0) {
      cost0 = cost;
      best.tx = tx;
      best.ty = ty;
    }
  }
  const long long tiles = (long long)((g.nx - 1) / best.tx + 1) * ((g.ny - 1) / best.ty + 1);
  double c0 = 1e300;
  for (int zc = 1; zc <= g.nz && (zc <= 256 || best.zc == 0); zc = next_chunk(g.nz, zc)) {
    const long long items = tiles * ((g.nz - 1) / zc + 1);
    if (items > (1 << 30) || (max_items && items > max_items && zc < g.nz)) continue;
    const double c = (double)((items + sm_count - 1) / sm_count) * (zc + extra);
    if (c < c0) {
      c0 = c;
      best.zc = zc;
      best.items = (int)items;
    }
  }
  return best;
}

}  // namespace elas
