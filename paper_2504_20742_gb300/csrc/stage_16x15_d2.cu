// stage_16x15_d2.cu -- the plain FP64 stage kernels for tiles of 16 x 15 cells with registers
// and shared memory budgeted for two CTAs per SM.
#include "stage.cuh"

namespace ct {
const StageSet* stage_set_16x15_d2() {
  // 240 cells, 255 x faces and 256 r faces on 256 threads: two warps per scheduler in every phase
  static const StageSet s = make_stage_set_fp64<Tile<16, 15, 2, 2, 256>>();
  return &s;
}
}  // namespace ct
