// kern_2d.cu -- 2D stage-kernel instantiations.  FP32 runs on independent warps
// (stage_strip.cuh; the tile index chooses the strips per CTA: 2, 4 or 8.  Two
// end a stage soonest: 28.2 and 26.6 us at 1024^2 against 33.0 and 30.7 with
// four, whose CTAs wait for their last warp's partial sums), FP64 on row tiles of TX cells that march along y.
#include "instantiate.cuh"

namespace gh {

int tile_count_2d() { return 3; }

bool stage_variant_2d(bool fp64, int solver, int stage, int tile, StageVariant* out) {
  if (solver == SOLVER_HLLC_SW)
    return tile == 0 && (fp64 ? pick_switch<2, double, 128, 1>(stage, out) : pick_strip_switch<float, 2>(stage, out));
  switch (tile) {
    case 0: return fp64 ? pick_variant<2, double, 128, 1>(solver, stage, out) : pick_strip<float, 2>(solver, stage, out);
    case 1: return fp64 ? pick_variant<2, double, 64, 1>(solver, stage, out) : pick_strip<float, 4>(solver, stage, out);
    case 2: return fp64 ? pick_variant<2, double, 256, 1>(solver, stage, out) : pick_strip<float, 8>(solver, stage, out);
  }
  return false;
}

}  // namespace gh
