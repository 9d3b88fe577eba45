// stage_strip.cuh -- one RK stage of a 1D or 2D FP32 mesh on independent warps.
//
// A warp takes a strip of 28 columns (lane l holds column x0 + l - 2: two
// neighbours on each side) and marches along y.  The march axis lives in a
// register ring, as in stage_kernel.cuh; along x the warp's own shuffles move
// what neighbouring columns need: W of the two neighbours for the slope, the
// upper face value of the lower neighbour, and the flux of the upper face.
// Each slope and each face flux is computed once per lane, nothing goes
// through shared memory, and no warp waits for another.
//
// What bounds it, and why this split: the 2D row tiles it replaced (one row of
// a CTA per plane, two barriers a row, every x slope formed twice) ran about
// 640 instructions a cell at 47-67% of the issue slots, their warps waiting at
// the barriers.
// Stages 1 and 2 of the row tiles and of the strips, HLLC with totals: 40.0 and
// 36.9 -> 28.2 and 26.6 us at 1024^2, 22.7 and 18.4 -> 13.2 and 12.3 us at
// 256 x 768.  565 and 523 instructions a cell at 1024^2 (of them 54 and 0 for
// the compensated totals), 78% of the issue slots at 4096^2.
#pragma once

#include <type_traits>

#include "stage_kernel.cuh"

namespace gh {

constexpr int STRIP_OWN = 28;  // columns a warp owns

// Sum of four double-word values per lane over the warp: lanes 8 v .. 8 v + 7
// of the result hold variable v.  Halving the variables with the lanes takes six
// additions instead of twenty, and on FP32 pairs: as FP64 additions this tail
// took 2-5 us of a stage on a mesh of 0.2 to 1 million cells.
__device__ __forceinline__ dw shfl_xor_dw(dw x, int o) {
  return dw(__shfl_xor_sync(0xffffffffu, x.hi, o), __shfl_xor_sync(0xffffffffu, x.lo, o));
}
__device__ __forceinline__ dw warp_sum4(const dw (&s)[4]) {
  const int lane = threadIdx.x & 31;
  const bool h = lane & 16, q = lane & 8;
  // lanes 0..15 keep variables 0, 1; lanes 16..31 keep 2, 3
  const dw a = (h ? s[2] : s[0]) + shfl_xor_dw(h ? s[0] : s[2], 16);
  const dw b = (h ? s[3] : s[1]) + shfl_xor_dw(h ? s[1] : s[3], 16);
  dw r = (q ? b : a) + shfl_xor_dw(q ? a : b, 8);
  for (int o = 4; o > 0; o >>= 1) r += shfl_xor_dw(r, o);
  return r;
}

// WIDE: 64-bit cell offsets, for meshes of more than 2^30 cells.
template <int NDIM, int SOLVER, int STAGE, bool WIDE>
struct StripKernel {
  static_assert(NDIM == 1 || NDIM == 2, "strips are 1D rows or 2D columns of rows");
  using Base = StageKernel<NDIM, float, SOLVER, STAGE, 32, 1, false>;
  using Off = typename std::conditional<WIDE, size_t, unsigned>::type;
  static constexpr int NV = NDIM + 2;
  static_assert(!Base::SW, "the switch runs on the row tiles");

  static __device__ __forceinline__ float left_of(float x) { return __shfl_up_sync(0xffffffffu, x, 1); }
  static __device__ __forceinline__ float right_of(float x) { return __shfl_down_sync(0xffffffffu, x, 1); }
  // element c of a plane: the 32-bit byte offset is added to a base that is the
  // same for the whole warp
  static __device__ __forceinline__ float at(const float* p, Off c) {
    return __ldg(reinterpret_cast<const float*>(reinterpret_cast<const char*>(p) + (Off)(c * 4)));
  }
  static __device__ __forceinline__ void set(float* p, Off c, float x) {
    *reinterpret_cast<float*>(reinterpret_cast<char*>(p) + (Off)(c * 4)) = x;
  }

  // minus the x part of the flux divergence of the lanes' cells of one row
  // (valid on the owned lanes), from W of the row
  static __device__ __forceinline__ void x_part(const StageArgs<float>& A, const float (&w)[NV], const Geo<float>& g,
                                                float iwx, float (&d)[NV]) {
    float wl[NV], wr[NV], f[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      float hi;
      face_pair(limited_slope(left_of(w[v]), w[v], right_of(w[v]), g), g.h, w[v], wr[v], hi);
      wl[v] = left_of(hi);
    }
    face_flux<float, NDIM, 0, SOLVER>(wl, wr, A.gamma, A.gm1, f);  // the face below each column
#pragma unroll
    for (int v = 0; v < NV; ++v) d[v] = mul_rn(sub_rn(f[v], right_of(f[v])), iwx);
  }

  // Strip of columns x0 .. x0 + 27, rows m0 .. m1 - 1 (2D; 1D: the one row).
  // Accumulates the lane's CFL speed and, with totals, its column's sum of
  // U dy dx (stage 1), and the non-physical flag.  The whole warp calls it.
  static __device__ __forceinline__ void strip(const StageArgs<float>& A, int x0, int m0, int m1, float& speed_out,
                                               dw (&tot)[NV], bool& bad) {
    const int lane = threadIdx.x & 31;
    const int nx = A.n[0], ny = NDIM == 2 ? A.n[1] : 1;
    const size_t vs = (size_t)nx * ny;
    const float dt = STAGE == 2 ? (float)(*A.dt) : 0.0f;
    const int col = x0 + lane - 2;
    const bool own = lane >= 2 && lane < 2 + STRIP_OWN && col < nx;
    bool fa;
    const Off off = (Off)bc_map(col, nx, A.bc_lo[0], A.bc_hi[0], fa);
    const Geo<float> gx = Base::geo(A, 0, col);
    const float iwx = A.iw[0][min(col, nx + 1) + 2];
    const float *un[NV], *k1[NV];
    float* out[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      un[v] = A.un + v * vs;
      k1[v] = A.k1 + v * vs;
      out[v] = A.out + v * vs;
    }
    ColumnSum<float> tcol[NV];
    float speed_max = 0.0f;

    // state of the cell at offset c (stage 2: U^n + dt K), x mirrored
    auto load = [&](Off c, float (&u)[NV]) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        u[v] = at(un[v], c);
        if (STAGE == 2) u[v] = fma_rn(dt, at(k1[v], c), u[v]);
      }
    };
    // Epilogue of the own cell at offset c: L = minus the divergence, source,
    // output, and in stage 1 the CFL speed.
    auto finish = [&](Off c, float (&L)[NV], const float (&w)[NV], float iwm) {
      if (A.has_source) Base::add_source(A, w, L);
      const float p = mul_rn(A.gm1, w[NV - 1]);
      float vsum = fabsf(w[1]);
      if constexpr (NDIM == 2) vsum = add_rn(vsum, fabsf(w[2]));
      const bool ok = fminf(w[0], p) > 0.0f && w[0] == w[0] && p == p && vsum < INFINITY;
      bad |= own && !ok;
      if (STAGE == 1) {
        const float cs = sound_speed(A.gamma, p, w[0]);
        float s = mul_rn(add_rn(fabsf(w[1]), cs), iwx);
        if constexpr (NDIM == 2) s = fmaxf(s, mul_rn(add_rn(fabsf(w[NDIM]), cs), iwm));
        speed_max = fmaxf(speed_max, s);
        if (own) {
#pragma unroll
          for (int v = 0; v < NV; ++v) set(out[v], c, L[v]);
        }
      } else {
        const float hdt = 0.5f * dt;
        float r[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) r[v] = fma_rn(hdt, add_rn(at(k1[v], c), L[v]), at(un[v], c));
        if (own) {
#pragma unroll
          for (int v = 0; v < NV; ++v) set(out[v], c, r[v]);
        }
      }
    };

    if constexpr (NDIM == 1) {
      float u[NV], w[NV], L[NV];
      load(off, u);
      if (STAGE == 1 && A.want_totals) {
#pragma unroll
        for (int v = 0; v < NV; ++v) tcol[v].add_product(u[v], 1.0f, 0.0f);
      }
      if (fa) u[1] = -u[1];
      recover<NDIM>(u, w);
      x_part(A, w, gx, iwx, L);
      finish(off, L, w, 0.0f);
    } else {
      // W of row m (boundary-mapped); with totals also the row's share of the
      // column sums when it is one of the strip's own
      auto row = [&](int m, float (&u)[NV]) {
        bool fm;
        const int sm = bc_map(m, ny, A.bc_lo[1], A.bc_hi[1], fm);
        load(off + (Off)sm * (Off)nx, u);
        if (STAGE == 1 && A.want_totals && m >= m0 && m < m1) {
          const float hi = A.wdh[1][m], lo = A.wdl[1][m];
#pragma unroll
          for (int v = 0; v < NV; ++v) tcol[v].add_product(u[v], hi, lo);
        }
        if (fa) u[1] = -u[1];
        if (fm) u[2] = -u[2];
      };
      // Limited slope and lower face value of row m + 1 from W(m), W(m + 1),
      // W(m + 2) and the scaled difference dlo across face m + 1/2, which moves
      // on to face m + 3/2 (a cell's upper scaled difference and its upper
      // neighbour's lower one are the same number).
      auto slope = [&](const float (&wk)[NV], const float (&wk1)[NV], const float (&w2)[NV], const Geo<float>& g,
                       float (&dlo)[NV], float (&s)[NV], float (&wr)[NV]) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const float dhi = mul_rn(sub_rn(w2[v], wk1[v]), g.tipc);
          s[v] = minmod3(dlo[v], mul_rn(sub_rn(w2[v], wk[v]), g.ipm), dhi);
          wr[v] = fma_rn(-s[v], g.h, wk1[v]);
          dlo[v] = dhi;
        }
      };
      // At the top of iteration m: wk = W(m), wk1 = W(m + 1), dlo = the scaled
      // difference across face m + 1/2, hi = the upper face value of cell m,
      // flo = the flux through face m - 1/2.
      float wk[NV], wk1[NV], w2[NV], dlo[NV], hi[NV], flo[NV], u[NV], s[NV], wr[NV];
      row(m0 - 2, u);
      recover<NDIM>(u, wk);
      row(m0 - 1, u);
      recover<NDIM>(u, wk1);
      row(m0, u);
      recover<NDIM>(u, w2);
      {
        const float t = Base::geo(A, 1, m0 - 2).tipc;
#pragma unroll
        for (int v = 0; v < NV; ++v) dlo[v] = mul_rn(sub_rn(wk1[v], wk[v]), t);
        const Geo<float> g = Base::geo(A, 1, m0 - 1);
        slope(wk, wk1, w2, g, dlo, s, wr);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          hi[v] = fma_rn(s[v], g.h, wk1[v]);
          wk[v] = wk1[v];
          wk1[v] = w2[v];
        }
      }
      row(m0 + 1, u);
      recover<NDIM>(u, w2);
      {
        const Geo<float> g = Base::geo(A, 1, m0);
        slope(wk, wk1, w2, g, dlo, s, wr);
        face_flux<float, NDIM, NDIM - 1, SOLVER>(hi, wr, A.gamma, A.gm1, flo);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          hi[v] = fma_rn(s[v], g.h, wk1[v]);
          wk[v] = wk1[v];
          wk1[v] = w2[v];
        }
      }
#pragma unroll 1
      for (int m = m0; m < m1; ++m) {
        float L[NV], fhi[NV];
        row(m + 2, u);  // lands during the x part
        x_part(A, wk, gx, iwx, L);
        recover<NDIM>(u, w2);
        const Geo<float> g = Base::geo(A, 1, m + 1);
        const float iwm = A.iw[1][m + 2];
        slope(wk, wk1, w2, g, dlo, s, wr);
        // face m + 1/2 between the upper value of m and the lower of m + 1
        face_flux<float, NDIM, NDIM - 1, SOLVER>(hi, wr, A.gamma, A.gm1, fhi);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          L[v] = fma_rn(sub_rn(flo[v], fhi[v]), iwm, L[v]);
          flo[v] = fhi[v];
        }
        finish(off + (Off)m * (Off)nx, L, wk, iwm);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          hi[v] = fma_rn(s[v], g.h, wk1[v]);
          wk[v] = wk1[v];
          wk1[v] = w2[v];
        }
      }
    }
    if (STAGE == 1 && own) {
      if (A.want_totals) {
        // the width as three floats: the pair alone would leave 2^-49 of it out
        const dw dx = dw(A.wdh[0][col], A.wdl[0][col]);
        const float dx3 = (float)((A.wd[0][col] - (double)dx.hi) - (double)dx.lo);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          dw c;
          fast_two_sum(tcol[v].hi, tcol[v].lo, c.hi, c.lo);
          const dw r = c * dx;
          fast_two_sum(r.hi, fma_rn(c.hi, dx3, r.lo), tot[v].hi, tot[v].lo);
        }
      }
      speed_out = fmaxf(speed_out, speed_max);
    }
  }
};

// 2D single mesh: CTA (x, chunk) of NW warps, each its own strip.  64
// registers, so that 32 warps stay resident on an SM.
template <int SOLVER, int STAGE, int NW, bool WIDE>
__global__ void __launch_bounds__(32 * NW, 32 / NW) hydro_strip_kernel(const StageArgs<float> A) {
  using K = StripKernel<2, SOLVER, STAGE, WIDE>;
  constexpr int NV = 4;
  __shared__ double red[NW][NV + 1];
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int x0 = (blockIdx.x * NW + warp) * STRIP_OWN;
  const int m0 = blockIdx.z * A.kchunk, m1 = min(A.n[1], m0 + A.kchunk);
  float speed = 0.0f;
  dw tot[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) tot[v] = dw(0.0f, 0.0f);
  bool bad = false;
  if (x0 < A.n[0]) K::strip(A, x0, m0, m1, speed, tot, bad);
  if (bad) atomicOr(A.status, STATUS_NONPHYS);
  if (STAGE == 1) {
    // fixed-order reduction into this CTA's partials
    const int lane = threadIdx.x & 31;
    const float s = warp_max(speed);
    if (lane == 0) red[warp][0] = (double)s;
    if (A.want_totals) {
      const dw t = warp_sum4(tot);
      if ((lane & 7) == 0) red[warp][1 + (lane >> 3)] = (double)t;
    } else if ((lane & 7) == 0) {
      red[warp][1 + (lane >> 3)] = 0.0;
    }
    __syncthreads();
    const int t = threadIdx.x;
    const size_t blk = (size_t)blockIdx.z * gridDim.x + blockIdx.x;
    if (t <= NV) {
      double acc = red[0][t];
      for (int w = 1; w < NW; ++w) acc = t == 0 ? fmax(acc, red[w][0]) : acc + red[w][t];
      if (t == 0) A.part_speed[blk] = acc;
      else A.part_tot[blk * NV + (t - 1)] = acc;
    }
  }
}

}  // namespace gh
