// batch_registry.h -- compiled variants of the persistent batch kernel.
#pragma once

#include <stddef.h>

namespace gh {

struct BatchVariant {
  const void* fn;
  size_t smem;
  int tx;    // threads per CTA (one tile row)
  int cols;  // columns of cells a tile owns
  int warps = 1;      // work items a CTA runs at once (one per warp), 1: the whole CTA runs one
  int most_1d = 1;    // most x tiles of a 1D item
  const void* fn_wide = nullptr;  // the kernel when a problem has more than 2^30 cells, where it is another
};

int batch_tile_count();
bool batch_variant_f32(int solver, int stage, int tile, BatchVariant* out);
bool batch_variant_f64(int solver, int stage, int tile, BatchVariant* out);
bool batch_variant_dw(int solver, int stage, int tile, BatchVariant* out);

}  // namespace gh
