// batch_strip.cuh -- persistent FP32 stage kernel over many 1D and 2D problems
// whose warps work alone: each takes the next item (a strip of 28 columns by a
// chunk of rows, or a group of 1D strips) from the global counter and runs the
// strip of stage_strip.cuh on it.  Items are sorted largest first.
//
// Bound by issue and, at the ends, by the last items: per-warp items need no
// barrier and no shared memory, and an item's last rows hide another warp's
// loads.  Stages 1 and 2 against
// the row tiles: 256 problems (13 million cells) 370 and 395 -> 222 and 252 us,
// 2048 problems 2383 and 2552 -> 1425 and 1647 us.
#pragma once

#include "batch_kernel.cuh"
#include "stage_strip.cuh"

namespace gh {

constexpr int STRIP_GROUP_1D = 8;  // strips of a 1D item: one has a single row, less work than taking it

template <int SOLVER, int STAGE, int NW, bool WIDE>
__global__ void __launch_bounds__(32 * NW, 32 / NW) hydro_batch_strip_kernel(const BatchArgs<float> B) {
  using K1 = StripKernel<1, float, SOLVER, STAGE, WIDE>;
  using K2 = StripKernel<2, float, SOLVER, STAGE, WIDE>;
  using Args = BatchKernel<float, SOLVER, STAGE, 128>;
  const int lane = threadIdx.x & 31;
  for (;;) {
    int it = 0;
    if (lane == 0) it = (int)atomicAdd(B.counter, 1u);
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it >= B.nitems) break;
    const BatchItem w = B.items[it];
    const BatchProblem<float>& P = B.probs[w.prob];
    float speed = 0.0f;
    bool bad = false;
    if (P.ndim == 1) {
      dw tot[3];
      const StageArgs<float> A = Args::template args_for<1>(B, P, w.prob);
      for (int k = 0; k < STRIP_GROUP_1D; ++k) {
        const int x0 = (w.tx * STRIP_GROUP_1D + k) * STRIP_OWN;
        if (x0 >= A.n[0]) break;
        K1::strip(A, x0, 0, 1, 0, speed, tot, bad);
      }
    } else {
      dw tot[4];
      const StageArgs<float> A = Args::template args_for<2>(B, P, w.prob);
      const int m0 = w.chunk * B.kchunk;
      K2::strip(A, w.tx * STRIP_OWN, m0, min(A.n[1], m0 + B.kchunk), 0, speed, tot, bad);
    }
    if (bad) atomicOr(B.status + w.prob, STATUS_NONPHYS);
    if (STAGE == 1) {
      const float m = warp_max(speed);
      // positive doubles order like their bit patterns
      if (lane == 0) atomicMax(B.speed + w.prob, (unsigned long long)__double_as_longlong((double)m));
    }
  }
}

}  // namespace gh
