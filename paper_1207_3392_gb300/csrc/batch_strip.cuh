// batch_strip.cuh -- persistent stage kernel (FP32, double word) over many 1D and
// 2D problems whose warps work alone: each takes the next item (a strip of 28 columns by a
// chunk of rows, or a group of 1D strips) from the global counter and runs the
// strip of stage_strip.cuh on it.  Items are sorted largest first.
//
// Bound by issue and, at the ends, by the last items: per-warp items need no
// barrier and no shared memory, and an item's last rows hide another warp's
// loads.  Stages 1 and 2 against
// the row tiles: 256 problems (13 million cells) 370 and 395 -> 222 and 252 us,
// 2048 problems 2383 and 2552 -> 1425 and 1647 us.  Double word, 48 problems, 6
// steps with their copies in and out: HLLC 7.62 -> 5.38 ms, HLL 7.37 -> 5.91; 4096
// problems, a step 65.8 -> 40.8 ms.
#pragma once

#include "batch_kernel.cuh"
#include "batch_registry.h"
#include "stage_strip.cuh"

namespace gh {

constexpr int STRIP_GROUP_1D = 8;  // most strips of a 1D item: one has a single row, less work than taking it

template <class T, int SOLVER, int STAGE, int NW, bool WIDE>
__global__ void __launch_bounds__(32 * NW, (strip_warps<T, 2>() / NW))
    hydro_batch_strip_kernel(const BatchArgs<T> B) {
  using K1 = StripKernel<1, T, SOLVER, STAGE, WIDE>;
  using K2 = StripKernel<2, T, SOLVER, STAGE, WIDE>;
  using Args = BatchKernel<T, SOLVER, STAGE, 128>;
  const int lane = threadIdx.x & 31;
  for (;;) {
    int it = 0;
    if (lane == 0) it = (int)atomicAdd(B.counter, 1u);
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it >= B.nitems) break;
    const BatchItem w = B.items[it];
    const BatchProblem<T>& P = B.probs[w.prob];
    T speed = T(0.0f);
    bool bad = false;
    if (P.ndim == 1) {
      Shares<3> tot;
      const StageArgs<T> A = Args::template args_for<1>(B, P, w.prob);
      for (int k = 0; k < B.group_1d; ++k) {
        const int x0 = (w.tx * B.group_1d + k) * STRIP_OWN;
        if (x0 >= A.n[0]) break;
        K1::strip(A, x0, 0, 1, 0, speed, tot, bad);
      }
    } else {
      Shares<4> tot;
      const StageArgs<T> A = Args::template args_for<2>(B, P, w.prob);
      const int m0 = w.chunk * B.kchunk;
      K2::strip(A, w.tx * STRIP_OWN, m0, min(A.n[1], m0 + B.kchunk), 0, speed, tot, bad);
    }
    if (bad) atomicOr(B.status + w.prob, STATUS_NONPHYS);
    if (STAGE == 1) {
      double m;
      if constexpr (std::is_same<T, float>::value) m = (double)warp_max(speed);
      else m = warp_max((double)speed);
      // positive doubles order like their bit patterns
      if (lane == 0) atomicMax(B.speed + w.prob, (unsigned long long)__double_as_longlong(m));
    }
  }
}

template <class T, int SOLVER, int STAGE, int NW>
void fill_batch_strip(BatchVariant* out) {
  out->fn = reinterpret_cast<const void*>(&hydro_batch_strip_kernel<T, SOLVER, STAGE, NW, false>);
  out->fn_wide = reinterpret_cast<const void*>(&hydro_batch_strip_kernel<T, SOLVER, STAGE, NW, true>);
  out->smem = 0;
  out->tx = 32 * NW;
  out->cols = STRIP_OWN;
  out->warps = NW;
  out->most_1d = STRIP_GROUP_1D;
}

template <class T, int NW>
bool pick_batch_strip(int solver, int stage, BatchVariant* out) {
  if (solver == SOLVER_HLL && stage == 1) fill_batch_strip<T, SOLVER_HLL, 1, NW>(out);
  else if (solver == SOLVER_HLL && stage == 2) fill_batch_strip<T, SOLVER_HLL, 2, NW>(out);
  else if (solver == SOLVER_HLLC && stage == 1) fill_batch_strip<T, SOLVER_HLLC, 1, NW>(out);
  else if (solver == SOLVER_HLLC && stage == 2) fill_batch_strip<T, SOLVER_HLLC, 2, NW>(out);
  else return false;
  return true;
}

}  // namespace gh
