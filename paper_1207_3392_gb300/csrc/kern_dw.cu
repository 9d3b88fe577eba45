// kern_dw.cu -- 1D and 2D stage kernels with the double-word (FP32 pair)
// arithmetic of dword.cuh.
#include "instantiate.cuh"

namespace gh {

int tile_count_dw(int ndim) { return ndim == 3 ? 5 : ndim == 2 ? 2 : 1; }

bool stage_variant_dw(int ndim, int solver, int stage, int tile, StageVariant* out) {
  if (ndim == 3) return stage_variant_dw_3d(solver, stage, tile, out);
  if (ndim == 2 && tile == 1) return pick_strip<dw, 2>(solver, stage, out);
  if (tile != 0) return false;
  // 1D: seven CTAs an SM (at 86 registers five fit: 2 million cells 383 us a step,
  // with seven 313).  2D: three (at 174 two fit: 401 x 307 in chunks of 4 rows 103 us
  // a step, with three 88).
  return ndim == 1 ? pick_variant<1, dw, 128, 1, 7>(solver, stage, out)
                   : pick_variant<2, dw, 128, 1, 3>(solver, stage, out);
}

}  // namespace gh
