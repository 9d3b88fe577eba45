// batch_f32.cu -- persistent batch-kernel instantiations (float state): warps on
// their own strips (batch_strip.cuh), 4 or 8 of them per CTA.
#include "batch_registry.h"
#include "batch_strip.cuh"

namespace gh {

template <int SOLVER, int STAGE, int NW>
static void fill(BatchVariant* out) {
  out->fn = reinterpret_cast<const void*>(&hydro_batch_strip_kernel<SOLVER, STAGE, NW, false>);
  out->fn_wide = reinterpret_cast<const void*>(&hydro_batch_strip_kernel<SOLVER, STAGE, NW, true>);
  out->smem = 0;
  out->tx = 32 * NW;
  out->cols = STRIP_OWN;
  out->warps = NW;
  out->group_1d = STRIP_GROUP_1D;
}

template <int NW>
static bool pick(int solver, int stage, BatchVariant* out) {
  if (solver == SOLVER_HLL && stage == 1) fill<SOLVER_HLL, 1, NW>(out);
  else if (solver == SOLVER_HLL && stage == 2) fill<SOLVER_HLL, 2, NW>(out);
  else if (solver == SOLVER_HLLC && stage == 1) fill<SOLVER_HLLC, 1, NW>(out);
  else if (solver == SOLVER_HLLC && stage == 2) fill<SOLVER_HLLC, 2, NW>(out);
  else return false;
  return true;
}

bool batch_variant_f32(int solver, int stage, int tile, BatchVariant* out) {
  switch (tile) {
    case 0: return pick<4>(solver, stage, out);
    case 1: return pick<8>(solver, stage, out);
  }
  return false;
}

}  // namespace gh
