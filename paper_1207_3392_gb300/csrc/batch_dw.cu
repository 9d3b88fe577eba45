// batch_dw.cu -- persistent batch-kernel instantiations (double-word state, dword.cuh): warps on
// their own strips (batch_strip.cuh), 4 or 8 of them per CTA.
#include "batch_strip.cuh"

namespace gh {

bool batch_variant_dw(int solver, int stage, int tile, BatchVariant* out) {
  switch (tile) {
    case 0: return pick_batch_strip<dw, 4>(solver, stage, out);
    case 1: return pick_batch_strip<dw, 8>(solver, stage, out);
  }
  return false;
}

}  // namespace gh
