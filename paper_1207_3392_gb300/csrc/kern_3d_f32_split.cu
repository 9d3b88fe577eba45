// kern_3d_f32_split.cu -- 3D FP32 stages on independent warps (stage_strip.cuh).
#include "instantiate.cuh"

namespace gh {

bool stage_variant_3d_f32_split(int solver, int stage, StageVariant* out) {
  if (solver == SOLVER_HLLC_SW) return pick_split_switch<float>(stage, out);
  return pick_split<float>(solver, stage, out);
}

}  // namespace gh
