// batch_f32.cu -- persistent batch-kernel instantiations (float state): warps on
// their own strips (batch_strip.cuh), 4 or 8 of them per CTA.
#include "batch_strip.cuh"

namespace gh {

bool batch_variant_f32(int solver, int stage, int tile, BatchVariant* out) {
  switch (tile) {
    case 0: return pick_batch_strip<float, 4>(solver, stage, out);
    case 1: return pick_batch_strip<float, 8>(solver, stage, out);
  }
  return false;
}

}  // namespace gh
