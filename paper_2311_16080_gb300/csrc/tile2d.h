// Host interface of the tiled D2Q9 kernel (tile2d.cu): several updates per
// launch on lattices too large for one cluster.
#pragma once
#include <stdint.h>

#include "xlb_types.h"

namespace xlb {

// Tiles of bx x by cells (the last ones may be smaller), tx of them per row of
// tiles, each with a ring of `halo` cells; halo updates per launch.
// halo = 0: no plan.
struct Tile2dPlan {
  int bx, by, tx, ty, halo;
  float us;   // the time per update by which plans are compared
  int waves;  // of blocks, one per SM
};

Tile2dPlan tile2d_plan(int storage, int coll, int nx, int ny);

// Cells of one region with rules of their own (INLET, beside an OUTLET,
// Bouzidi links) that a block has room for.
constexpr int TILE_LIST = 1536;

struct Tile2dArgs {
  StepParams p;          // flags null: every cell FLUID
  int storage, coll;
  const void* src;       // post-collision populations
  void* dst;             // the same `steps` updates later (another buffer)
  // per cell 0 or 1 + its row in bz_q (rows < 65535), or null; 0 for OUTLET
  // cells, which the kernel updates without a row
  const int* bz;
  // 9 pairs per row.  Pair i of a link in direction i with wall distance q:
  // {2q, 1 - 2q} or {1/(2q), 1 - 1/(2q)} (q >= 1/2); {1, 0}, the halfway rule as
  // q = 1/2, for a distance below 1/2 where the cell behind is not FLUID.  Pair
  // 0: the bit sets of the links with q < 1/2 and of those with q >= 1/2.
  const float* bz_q;
  Tile2dPlan plan;
  int steps;             // 1 .. halo
  void* stream;
};

int launch_tile2d(const Tile2dArgs& a);

}  // namespace xlb
