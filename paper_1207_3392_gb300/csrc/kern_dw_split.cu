// kern_dw_split.cu -- 3D double-word stages on independent warps (stage_strip.cuh).
#include "instantiate.cuh"

namespace gh {

bool stage_variant_dw_split(int solver, int stage, StageVariant* out) { return pick_split<dw>(solver, stage, out); }

}  // namespace gh
