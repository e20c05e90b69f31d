// stage_8x2.cu -- the plain stage kernels for small grids: tiles of 8 x 2 cells on 128 threads,
// x and r directions side by side.
#include "stage.cuh"

namespace ct {
const StageSet* stage_set_8x2() {
  static const StageSet s = make_stage_set_small<Tile<8, 2, 4, 2, 128, true>>();
  return &s;
}
}  // namespace ct
